// The search kernels of F16 storage (see kb_search.cu).
#define KB_SEARCH_STORAGE KB_F16
#include "kb_search.cu"
