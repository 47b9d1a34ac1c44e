// The search kernels of BF16 storage (see kb_search.cu).
#define KB_SEARCH_STORAGE KB_BF16
#include "kb_search.cu"
