// Stage (b): exhaustive trajectory search of Sec. 2.2 on sm_103a.
//
// For every start pixel (x0, y0) and every velocity v, the coadd of Sec. 2.1.5
//   Psi = sum_t psi_t(x0 + dx_vt, y0 + dy_vt),  Phi = sum_t phi_t(...)
// over the epochs whose pixel lies in the image, nu = Psi / sqrt(Phi), and the
// k best (nu desc, vidx asc) valid trajectories per start pixel.
//
// Work decomposition (GB300-first, not the paper's 32x16 thread blocks):
//   - a CTA owns 8 rows x SPAN columns of start pixels, one warp per row; a lane
//     owns P loads' worth of pixels (FP32: pixel lane + 32 p; 16-bit: the pixel
//     pair 2 lane + 64 p, + 1) and runs the whole velocity loop for them;
//   - for one (velocity, epoch) a warp's loads cover SPAN consecutive pixels of
//     one plane row: fully coalesced 8-byte loads.  16-bit pairs are 8-byte
//     aligned because the planes also exist shifted by one pixel (the "phase 1"
//     copy) and odd shifts read that copy;
//   - the (velocity, epoch) table is staged per CTA in shared memory, a row per velocity:
//     one entry for each epoch whose shifted band (8 rows x SPAN columns) overlaps the
//     image, in time order, holding the offset of the shifted row start (epoch plane and
//     phase included) and for 16-bit storage the epoch's two power-of-two scales as bf16
//     bit patterns (the FMA's scale operand).  Epochs that miss the image are left out:
//     they add nothing.  Entries are read four to a group of 16-byte broadcast loads; per
//     entry and load there is an address, the gather and one packed f32x2 add per pixel
//     (16-bit: one mixed-precision FMA per value);
//   - bands that overlap the image only partly read the zero columns the planes carry left
//     and right of every row (kSpan wide) and the zero rows above and below every plane
//     (kPadRows), so "outside contributes nothing" holds exactly without a bounds check;
//   - epochs at t = t_min have offset 0 for every velocity: their contribution is
//     loaded once per pixel before the velocity loop;
//   - velocities are processed in the order the host planner gives (sorted by
//     their latest-epoch offset, for L2 locality of the resident CTAs); ties in
//     nu are broken by the caller's velocity index, so the order changes no
//     result;
//   - CTAs take their tiles in super-columns a few tiles wide, row by row within
//     each, so the CTAs resident at one time cover a compact block of start
//     pixels and the late epochs' rows they read stay in L2;
//   - top-k: each pixel's list of (nu, 16-bit velocity index), best first, and a short
//     buffer of new entries are in shared memory (slot-major: slot i of list column c at
//     c + i * LS, so the lanes of a warp touch distinct banks); the k-th entry is mirrored
//     in registers as the admission threshold.  A trajectory that beats its pixel's
//     threshold is appended to the buffer by its own lane, and when one of a warp's
//     buffers is full, all its lanes merge theirs in lock step.
// The Psi/Phi of each kept trajectory are recomputed at the end by the same
// sequence of operations (bit-identical) together with nobs.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stddef.h>
#include <string.h>

#include <algorithm>

#include "kb_device.cuh"

// This file compiles one storage's kernels: FP32's and the common entry points by itself,
// the 16-bit ones when kb_search_bf16.cu and kb_search_f16.cu include it (three translation
// units that build side by side).
#ifndef KB_SEARCH_STORAGE
#define KB_SEARCH_STORAGE KB_F32
#define KB_SEARCH_COMMON
#endif

namespace kb {

namespace {

#ifdef KB_DEBUG
// KB_DEBUG: the first out-of-bounds access of this storage's kernels, (site << 56) | offset
__device__ unsigned long long g_debug_word;
__device__ __noinline__ void debug_record(int site, long long at) {
    atomicCAS(&g_debug_word, 0ull, ((unsigned long long)site << 56) | ((unsigned long long)at & 0x00ffffffffffffffull));
}
#endif

// One load of a gather from the planes.  KB_DEBUG builds check that it lies inside
// the planes' allocation (elems pixels of type T from `planes`); one outside is
// recorded with its site and read as zero.
template <typename LT, typename T>
__device__ __forceinline__ LT gather(const LT *src, const T *planes, long long elems, int site) {
#ifdef KB_DEBUG
    const long long at = (long long)((const char *)src - (const char *)planes);
    if (at < 0 || at + (long long)sizeof(LT) > elems * (long long)sizeof(T)) {
        debug_record(site, at);
        return LT{};
    }
#else
    (void)planes;
    (void)elems;
    (void)site;
#endif
    return __ldg(src);
}

// KB_DEBUG builds: index i must lie in [0, n) (site 5: offset-table entry, 6: list column)
__device__ __forceinline__ bool debug_in(long long i, long long n, int site) {
#ifdef KB_DEBUG
    if (i < 0 || i >= n) {
        debug_record(site, i);
        return false;
    }
#else
    (void)i;
    (void)n;
    (void)site;
#endif
    return true;
}

using namespace dev;

constexpr int WARPS = 8;
constexpr int THREADS = WARPS * 32;
constexpr uint16_t kNoV = 0xFFFF;   // empty list slot (velocity indices are < 65535)
// lists up to kShortMax long merge in a network of 8,
constexpr int kKeyMax = 16;         // up to this (and key lists) in one of 16,
constexpr int kListMax = 32;        // and all others by walking

__device__ __forceinline__ float2 exp_scale(int e) {
    return make_float2(__int_as_float((e & 0xff) << 23), __int_as_float(((e >> 8) & 0xff) << 23));
}
__device__ __forceinline__ int scale_exp(float2 s) {
    return (int)((__float_as_uint(s.x) >> 23) & 0xff) | (int)(((__float_as_uint(s.y) >> 23) & 0xff) << 8);
}
// Scale operand of a 16-bit load: the bf16 bit patterns of the epoch's two
// power-of-two scales, psi in the low half and phi in the high half (a power of
// two is exactly a bf16).  Unused for FP32.
__device__ __forceinline__ uint32_t sc_of(float2 s) {
    return (__float_as_uint(s.x) >> 16) | (__float_as_uint(s.y) & 0xffff0000u);
}

// per-load traits: FP32 loads one pixel's (psi, phi), 16-bit loads two adjacent pixels' codes
template <int STORAGE>
struct Gather;
template <>
struct Gather<KB_F32> {
    typedef float2 LT;
    static constexpr int PIX = 1;
    __device__ __forceinline__ static void acc(float2 *a, LT v, uint32_t) { a[0] = add2(a[0], v); }
};
// BF16: mixed-precision fma.rn.f32.bf16 takes each code and each scale straight from
// its register half; the scale is a power of two, so code * scale is exact and the
// sum is rounded once -- the same FP32 result as unpacking and fma.rn.f32x2.
__device__ __forceinline__ void bf16_acc(float2 &a, uint32_t code, uint32_t sc) {
    asm("{\n\t.reg .b16 lo, hi, sp, sf;\n\t"
        "mov.b32 {lo, hi}, %2;\n\t"
        "mov.b32 {sp, sf}, %3;\n\t"
        "fma.rn.f32.bf16 %0, lo, sp, %0;\n\t"
        "fma.rn.f32.bf16 %1, hi, sf, %1;\n\t}"
        : "+f"(a.x), "+f"(a.y)
        : "r"(code), "r"(sc));
}
template <>
struct Gather<KB_BF16> {
    typedef uint2 LT;
    static constexpr int PIX = 2;
    __device__ __forceinline__ static void acc(float2 *a, LT v, uint32_t sc) {
        bf16_acc(a[0], v.x, sc);
        bf16_acc(a[1], v.y, sc);
    }
};
// FP16: the codes converted to FP32 and fused with the scales (fma.rn.f32x2)
template <>
struct Gather<KB_F16> {
    typedef uint2 LT;
    static constexpr int PIX = 2;
    __device__ __forceinline__ static void acc(float2 *a, LT v, uint32_t sc) {
        const float2 s = make_float2(__uint_as_float(sc << 16), __uint_as_float(sc & 0xffff0000u));
        a[0] = Store<KB_F16>::acc(a[0], v.x, s);
        a[1] = Store<KB_F16>::acc(a[1], v.y, s);
    }
};

// Staged table entry: the shifted row start of one (velocity, epoch), relative to the
// lane's place in plane 0 (LaneBase), and for 16-bit storage (SC) the epoch's scale operand.
template <typename I, bool SC>
struct Entry;
template <typename I>
struct Entry<I, false> {
    I idx;
};
template <typename I>
struct Entry<I, true> {
    I idx;
    uint32_t sc;
};
// Bytes of entries per chunk of the table.  A velocity's row is a whole number of groups of
// four entries, so a chunk holds at most a quarter as many velocities as entries.  FP32: 2 KB
// (42 velocities of 11 epochs), which with buffers of 4 leaves 4 CTAs per SM within the
// 164 KB shared-memory split and 92 KB to L1 (12 x 4096^2, k = 8: 75.8 ms; 4 KB: 78.1); the
// pruned search, which takes bounds for 32 velocities of a chunk at once, 4 KB (12 x 2048^2,
// nu_min 10: 3.68 ms; 2 KB: 3.95).  16-bit: 4 KB.
template <int STORAGE, typename I>
__host__ __device__ constexpr size_t table_entry_bytes() { return sizeof(Entry<I, STORAGE != KB_F32>); }
template <int STORAGE, typename I, bool PRUNE>
__host__ __device__ constexpr int table_entries() {
    return (int)((STORAGE == KB_F32 && !PRUNE ? 2048 : 4096) / table_entry_bytes<STORAGE, I>());
}
// The pruned FP32 search with short lists has a form for more than kPruneMany epochs past the
// reference time, where a bound is a long sum and most of a chunk's lanes have none:
//   - buffers of 2 (k = 8), so that 4 CTAs stay within the 164 KB split (92 KB of L1, not 60);
//   - the lanes of a warp share the chunk's velocities, and a sum ends once it reaches nu_min^2;
//   - the bound offsets' rows have an odd stride (at 64 epochs, 16 lanes otherwise meet in a bank);
//   - element offsets from a pointer, so that 32-bit ones reach 2^31 elements.
// 64 x 1024^2, 256 velocities, k = 8, nu_min 5 / 12 / 20: 8.42 / 8.25 / 6.82 ms without it, 6.97 /
// 7.06 / 5.94 with it; 40 x 4096^2, 96 velocities, nu_min 12: 26.9 and 23.5; 32 x 1024^2, nu_min 20:
// 0.43 and 0.42; 24 x 1024^2, nu_min 12 / 20: 1.71 / 0.37 and 1.62 / 0.43.
constexpr int kPruneMany = 28;
template <int STORAGE, int KM, bool PRUNE, bool CUT>
__host__ __device__ constexpr bool many_epochs() { return STORAGE == KB_F32 && PRUNE && CUT && KM <= kShortMax; }
template <typename I>
__device__ __forceinline__ uint32_t entry_sc(const Entry<I, false> &) { return 0u; }
template <typename I>
__device__ __forceinline__ uint32_t entry_sc(const Entry<I, true> &e) { return e.sc; }

// four consecutive table entries, the first at a multiple of four, in 16-byte loads
template <typename E>
__device__ __forceinline__ void load_four(const E *t, E (&e)[4]) {
    static_assert(sizeof(E) % 4 == 0 && sizeof(E) <= 16, "a group of four entries is a whole number of 16-byte words");
    int4 w[sizeof(E) / 4];
#pragma unroll
    for (int i = 0; i < (int)(sizeof(E) / 4); ++i) w[i] = reinterpret_cast<const int4 *>(t)[i];
    memcpy(e, w, sizeof e);
}

// A lane's place in the planes, and where its loads of an entry start.  BYTES: a 32-bit byte
// offset from the planes' base, to which the entry's is added modulo 2^32 -- one register
// instead of a pointer's two; else a pointer.
template <typename T, bool BYTES>
struct LaneBase {
    const T *p;
    __device__ __forceinline__ LaneBase(const T *planes, long long elem) : p(planes + elem) {}
    template <typename I>
    __device__ __forceinline__ const T *at(const T *, I idx) const { return p + idx; }
    __device__ __forceinline__ static long long offset(long long elem) { return elem; }
};
template <typename T>
struct LaneBase<T, true> {
    uint32_t b;
    __device__ __forceinline__ LaneBase(const T *, long long elem) : b(offset(elem)) {}
    __device__ __forceinline__ const T *at(const T *planes, int idx) const {
        return reinterpret_cast<const T *>(reinterpret_cast<const char *>(planes) + ((uint32_t)idx + b));
    }
    __device__ __forceinline__ static uint32_t offset(long long elem) { return (uint32_t)(elem * (long long)sizeof(T)); }
};
// Byte offsets where registers are short: value lists up to 8 long, held to 64 (FP32, 12 x
// 4096^2, k = 8: 75.8 ms; pointers 80.5, one value of the loop in local memory; BF16, 12 x
// 2048^2, 1024 velocities, (1, 4): 18.6 ms; pointers 21.6).  Elsewhere the extra add costs
// more: BF16 key lists 25.8 ms against 25.5 with pointers (4096 x 2048).
template <int STORAGE, int KM, bool KEYS, typename I>
__host__ __device__ constexpr bool byte_offsets() { return sizeof(I) == 4 && KM <= kShortMax && !KEYS; }

// Candidate lists of a search that only feeds the FP64 rescoring (KEYS): one
// 32-bit key per slot.  With b = a.key_bits bits for a velocity index, the high
// 32 - b bits hold nu's order-preserving FP32 encoding (sign bit flipped for
// nu >= 0, every bit flipped below) rounded upwards to a multiple of 2^b, and the
// low b bits hold 2^b - 1 - vidx, so that a larger key is a better (nu desc,
// vidx asc) candidate and one unsigned compare orders two of them.  The lists
// take 4 bytes a slot instead of 6, and the rescoring gets an upper bound on the
// reduced-precision nu of every trajectory left out: the last kept key's value (a
// trajectory outside has a smaller key, so its rounded-up nu is at most that
// value).  A key's value hi and the value lo one step of 2^b below it in the
// encoding bracket the unrounded nu: lo < nu <= hi.  Empty slots are key 0, below
// the key of every finite nu (whose encoding is at least 2^23).
__device__ __forceinline__ uint32_t nu_key(float nu, int v, int b) {
    const uint32_t u = __float_as_uint(nu), m = (1u << b) - 1u;
    const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    const uint32_t q = (ord >> b) + ((ord & m) ? 1u : 0u);   // finite nu: q << b <= encoding of +inf
    return (q << b) | (m - (uint32_t)v);
}

// ---- per-pixel top-k lists ------------------------------------------------------
// A list column (one pixel, owned by one lane) holds its k best entries, sorted, then a
// buffer of CAP entries.  A trajectory that beats the pixel's threshold (its k-th entry
// at the last merge) is appended to the buffer by its own lane, without a vote or a
// conflict; when one of the warp's buffers is full, every lane merges its own buffers
// into its lists in registers, in lock step, with a sorting network.  A pixel admits about
// k (1 + log(V / k)) entries, 47 of 1024 velocities at k = 8, and a merge costs the same
// for one new entry as for CAP.  A queue common to the warp, emptied 32 entries at a time
// with a rank insertion each (match, ranks, bank conflicts between the pixels of a round),
// executed 17.9 G warp instructions and 1.43 G shared wavefronts at 12 x 2048^2, k = 8,
// against 15.2 G and 0.95 G (and 16.6 G with the queue and the same table).  The result
// does not depend on the order of arrival: a list ends as the k best of everything offered
// to it under (nu desc, vidx asc).

// an entry as one ordered word: nu's order-preserving encoding above 0xffff - vidx
__device__ __forceinline__ unsigned long long slot_key(float nu, int v) {
    const uint32_t u = __float_as_uint(nu + 0.0f);   // -0 and +0 are one score
    const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)ord << 32) | (0xffffu - (uint32_t)v);
}
__device__ __forceinline__ float slot_nu(unsigned long long key) {
    const uint32_t ord = (uint32_t)(key >> 32);
    return __uint_as_float((ord & 0x80000000u) ? (ord & 0x7FFFFFFFu) : ~ord);
}
__device__ __forceinline__ int slot_vidx(unsigned long long key) { return (int)(0xffffu - (uint32_t)(key & 0xffffu)); }

template <typename K>
__device__ __forceinline__ void order_desc(K &a, K &b) {
    const K hi = a > b ? a : b, lo = a > b ? b : a;
    a = hi;
    b = lo;
}

// the list l (KM entries, sorted, best first) becomes the KM best of itself and b (CAP <= KM
// entries in any order): b is sorted by Batcher's odd-even merge network, its reverse
// compared with the tail of l, and the bitonic sequence this leaves is merged
template <int KM, int CAP, typename K>
__device__ __forceinline__ void merge_best(K (&l)[KM], K (&b)[CAP]) {
#pragma unroll
    for (int p = 1; p < CAP; p *= 2) {
#pragma unroll
        for (int q = p; q >= 1; q /= 2) {
#pragma unroll
            for (int j = q % p; j + q < CAP; j += 2 * q) {
#pragma unroll
                for (int i = 0; i < q; ++i)
                    if (i + j + q < CAP && (i + j) / (2 * p) == (i + j + q) / (2 * p)) order_desc(b[i + j], b[i + j + q]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < CAP; ++i) l[KM - 1 - i] = l[KM - 1 - i] > b[i] ? l[KM - 1 - i] : b[i];
#pragma unroll
    for (int h = KM / 2; h >= 1; h /= 2) {
#pragma unroll
        for (int i = 0; i < KM; ++i)
            if ((i & h) == 0) order_desc(l[i], l[i + h]);
    }
}

// Merges the n buffered entries of a column into its list of k and sets its threshold, the
// list's k-th entry; slot i lies at i * LS of ln and lv (value lists) or lk (key lists).
// Inlined: as calls they cost the longer lists 8 % and more (2111 x 2045, 14 epochs, k = 12:
// 18.4 ms against 16.6; BF16 key lists, 4096 x 2048: 27.6 against 25.5).
template <int KM, int CAP, int LS>
__device__ __forceinline__ void merge_values(float *ln, uint16_t *lv, int k, int n, float &thn, int &thv) {
    unsigned long long l[KM], b[CAP];
#pragma unroll
    for (int i = 0; i < KM; ++i) l[i] = i < k ? slot_key(ln[i * LS], lv[i * LS]) : 0ull;
#pragma unroll
    for (int i = 0; i < CAP; ++i) b[i] = i < n ? slot_key(ln[(k + i) * LS], lv[(k + i) * LS]) : 0ull;
    merge_best<KM, CAP>(l, b);
#pragma unroll
    for (int i = 0; i < KM; ++i) {
        if (i < k) {
            ln[i * LS] = slot_nu(l[i]);
            lv[i * LS] = (uint16_t)slot_vidx(l[i]);
        }
    }
    thn = ln[(k - 1) * LS];
    thv = lv[(k - 1) * LS];
}
template <int KM, int CAP, int LS>
__device__ __forceinline__ void merge_keys(uint32_t *lk, int k, int n, uint32_t &thk) {
    uint32_t l[KM], b[CAP];
#pragma unroll
    for (int i = 0; i < KM; ++i) l[i] = i < k ? lk[i * LS] : 0u;
#pragma unroll
    for (int i = 0; i < CAP; ++i) b[i] = i < n ? lk[(k + i) * LS] : 0u;
    merge_best<KM, CAP>(l, b);
#pragma unroll
    for (int i = 0; i < KM; ++i)
        if (i < k) lk[i * LS] = l[i];
    thk = lk[(k - 1) * LS];
}

// Lists of 17 to 24 (only wide rescoring searches keep them): each buffered entry walks up from
// the last slot.  A network of 32 inlined would crowd out the search's loop.
template <int LS>
__device__ __forceinline__ void insert_values(float *ln, uint16_t *lv, int k, int n, float &thn, int &thv) {
    for (int e = 0; e < n; ++e) {
        const float cn = ln[(k + e) * LS];
        const int cv = lv[(k + e) * LS];
        int i = k - 1;
        if (!better(cn, cv, ln[i * LS], lv[i * LS])) continue;
        while (i > 0) {
            const float pn = ln[(i - 1) * LS];
            const int pv = lv[(i - 1) * LS];
            if (!better(cn, cv, pn, pv)) break;
            ln[i * LS] = pn;
            lv[i * LS] = (uint16_t)pv;
            --i;
        }
        ln[i * LS] = cn;
        lv[i * LS] = (uint16_t)cv;
    }
    thn = ln[(k - 1) * LS];
    thv = lv[(k - 1) * LS];
}

// Buffer entries of a column.  More of them mean fewer merges but a larger shared-memory
// footprint, and what the lists take the L1 loses: 12 x 4096^2, k = 8, FP32: 3 entries
// 80.0 ms, 4 75.8, 6 83.4; 2111 x 2045, 14 epochs, k = 12: 3 18.0 ms, 4 16.9, 5 16.6, 6 17.1;
// key lists (4096 x 2048 BF16, k_c = 12, with the rescoring): 3 26.1 ms, 4 25.5, 5 25.8.
// Value lists of four pixels per lane: 3, so that at k = 8 the 1024-pixel CTAs' lists leave room
// for 3 CTAs per SM (FP16, 1500 x 1700, 10 epochs, 500 velocities: (2, 4) 7.52 ms; 4 entries 7.98).
template <int KM, bool KEYS, int PX>
__host__ __device__ constexpr int list_cap() { return KEYS ? 4 : KM > kShortMax ? 5 : PX == 4 ? 3 : 4; }
// Adds B epochs (a multiple of four) of one velocity to a lane's sums: every load issued
// before the first sum, the sums in epoch order.
template <int STORAGE, int P, int B, typename E, typename T, typename L>
__device__ __forceinline__ void add_epochs(const E *tab, const L &lane0, const T *planes, long long elems, float2 *acc) {
    typedef Gather<STORAGE> G;
    typedef typename G::LT LT;
    LT val[B][P];
    uint32_t sc[B];
#pragma unroll
    for (int q = 0; q < B; q += 4) {
        E e[4];
        load_four(tab + q, e);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            sc[q + h] = entry_sc(e[h]);
            const LT *src = reinterpret_cast<const LT *>(lane0.at(planes, e[h].idx));
#pragma unroll
            for (int p = 0; p < P; ++p) val[q + h][p] = gather(src + 32 * p, planes, elems, 2);
        }
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
#pragma unroll
        for (int p = 0; p < P; ++p) G::acc(acc + p * G::PIX, val[q][p], sc[q]);
    }
}

// The last 1 to 3 epochs of a velocity (n is the same for the whole warp)
template <int STORAGE, int P, typename E, typename T, typename L>
__device__ __forceinline__ void add_tail(const E *tab, int n, const L &lane0, const T *planes, long long elems, float2 *acc) {
    typedef Gather<STORAGE> G;
    typedef typename G::LT LT;
    E e[4];
    load_four(tab, e);   // the row's padding included, unused
    LT val[3][P];
#pragma unroll
    for (int h = 0; h < 3; ++h) {
        if (h < n) {
            const LT *src = reinterpret_cast<const LT *>(lane0.at(planes, e[h].idx));
#pragma unroll
            for (int p = 0; p < P; ++p) val[h][p] = gather(src + 32 * p, planes, elems, 3);
        }
    }
#pragma unroll
    for (int h = 0; h < 3; ++h) {
        if (h < n) {
#pragma unroll
            for (int p = 0; p < P; ++p) G::acc(acc + p * G::PIX, val[h][p], entry_sc(e[h]));
        }
    }
}

// One CTA tile (rows by * 8 .. +7, columns bx * SPAN .. +SPAN-1) of one search:
// the body of both the one-search kernel and the persistent batch kernel.
// KM: the lists' longest length, which says how they merge.
// PRUNE: each warp adds its shifted span's bound (one value per epoch from the span
// bound planes, kb_prune.cu: L2-resident, one per 32 columns) for 32 velocities at
// once, a lane for each, and skips the velocities whose bound cannot reach nu_min^2
// (the results do not change).  A velocity at a time (a lane for each epoch, then the
// warp's sum) is a chain of a load and six shuffles for every velocity: 12 x 2048^2,
// 1024 velocities, nu_min 10, psi/phi and bounds included: 8.72 ms that way, 4.10 this way.
// KEYS: candidate lists in key form for the FP64 rescoring (a.cand_only, k <= kKeyMax).
// SPLIT: the velocities are dealt to the CTAs of a cluster (rank `part` of `parts`, which divides
// WARPS); each keeps its own lists, then warp w's are brought together by rank w % parts, which
// reads the others' through distributed shared memory and writes the records.
// CUT: the launch shortened the columns' buffers (buffer_cap): a column has a.slots slots.  With
// PRUNE, FP32 and short lists also the form for many epochs (MANY, many_epochs()).
template <int STORAGE, int P, int C, int KM, typename I, bool PRUNE, bool KEYS, bool SPLIT, bool CUT>
__device__ __forceinline__ void search_tile(const SearchArgs &a, int bx, int by, float2 *s_scale, int4 *s_dyn4,
                                            int part = 0, int parts = 1) {
    typedef Store<STORAGE> St;
    typedef typename St::T T;         // one pixel's (psi, phi)
    typedef Gather<STORAGE> G;
    typedef typename G::LT LT;        // one load
    typedef Entry<I, STORAGE != KB_F32> E;
    static_assert(C % 4 == 0, "entries are read four at a time");
    static_assert(WARPS <= kPadRows, "a band of warps' rows must fit the planes' zero rows");
    constexpr bool MANY = many_epochs<STORAGE, KM, PRUNE, CUT>();
    constexpr int TAB = table_entries<STORAGE, I, PRUNE>(), ROWS = TAB / 4;
    constexpr int RID = PRUNE ? TAB + (MANY ? ROWS : 0) : 0;   // bound offsets
    constexpr size_t EB = table_entry_bytes<STORAGE, I>();
    constexpr int PX = P * G::PIX;    // pixels per lane
    constexpr int SPAN = 32 * PX;     // pixels per warp row segment
    constexpr int LS = THREADS * PX;  // list columns (pixels) of the CTA
    constexpr int CAP = list_cap<KM, KEYS, PX>();             // most buffer entries of a column

    // s_scale: per time-ordered epoch.  s_dyn4: table E [TAB] | (PRUNE) bound offsets I [RID] |
    // velocity ids and entry counts [ROWS] | lists with their buffers: nu float [slots * LS],
    // vidx u16 [slots * LS] (KEYS: keys u32 [slots * LS]); slots: k and the buffer's.
    E *s_tab = reinterpret_cast<E *>(s_dyn4);
    I *s_rid = reinterpret_cast<I *>(reinterpret_cast<char *>(s_dyn4) + TAB * EB);
    int *s_vid = reinterpret_cast<int *>(s_rid + RID);
    const int N = a.N, n0 = a.n0, NJ = N - n0, k = a.k;
    const int NJP = (NJ + 3) & ~3;   // table row stride: whole groups of four entries
    const int NJR = MANY ? NJ | 1 : NJP;   // bound offsets' row stride
    float *s_ln = reinterpret_cast<float *>(s_vid + ROWS);
    const int slot_end = CUT ? a.slots * LS : (k + CAP) * LS;   // slots of a column, times LS
    uint16_t *s_lv = reinterpret_cast<uint16_t *>(s_ln + slot_end);
    uint32_t *s_lk = reinterpret_cast<uint32_t *>(s_vid + ROWS);   // KEYS: the lists instead
    for (int j = threadIdx.x; j < N; j += THREADS)
        s_scale[j] = (STORAGE == KB_F32) ? make_float2(1.0f, 1.0f) : exp_scale(scale_exp(a.scales[a.epoch_of[j]]));
    for (int i = threadIdx.x; i < k * LS; i += THREADS) {
        if constexpr (KEYS) {
            s_lk[i] = 0u;
        } else {
            s_ln[i] = -INFINITY;
            s_lv[i] = kNoV;
        }
    }

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int y0 = by * WARPS;
    const int y = y0 + warp;
    const int xw = bx * SPAN;
    const bool active = y < a.H;
    const T *planes = reinterpret_cast<const T *>(a.planes);
    // element index of this lane's first pixel within a plane (even for 16-bit storage)
    const long long tb = a.origin + (long long)y * a.pitch + xw + lane * G::PIX;
    typedef LaneBase<T, byte_offsets<STORAGE, KM, KEYS, I>() && !MANY> LB;
    const LB lane0(planes, tb);
    const unsigned lt_mask = (1u << lane) - 1u;

    float thn[PX];
    int thv[PX];
    uint32_t thk[PX];   // KEYS: the thresholds as keys
    int off[PX];        // the next free buffer slot of the lane's columns, as an offset from slot 0
    const int off_lim = slot_end;
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        thn[p] = -INFINITY;
        thv[p] = kNoV;
        thk[p] = 0u;
        off[p] = k * LS;
    }
    float *ln0 = s_ln + threadIdx.x;      // slot 0 of the lane's first column; column p is p * THREADS further
    uint16_t *lv0 = s_lv + threadIdx.x;
    uint32_t *lk0 = s_lk + threadIdx.x;
    __syncthreads();

    // epochs at the reference time: offset 0 for every velocity (pixels past W read the zero columns)
    float2 acc0[PX];
#pragma unroll
    for (int p = 0; p < PX; ++p) acc0[p] = make_float2(0.0f, 0.0f);
    if (active) {
        for (int j = 0; j < n0; ++j) {
            const LT *src = reinterpret_cast<const LT *>(planes + (long long)a.epoch_of[j] * a.plane_elems + tb);
#pragma unroll
            for (int p = 0; p < P; ++p)
                G::acc(acc0 + p * G::PIX, gather(src + 32 * p, planes, a.planes_elems, 1), sc_of(s_scale[j]));
        }
    }

    // every lane's buffers into its lists
    auto merge_lists = [&]() {
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            const int n = (off[p] - k * LS) / LS;
            if constexpr (KEYS)
                merge_keys<KM, CAP, LS>(lk0 + p * THREADS, k, n, thk[p]);
            else if constexpr (KM > kKeyMax)
                insert_values<LS>(ln0 + p * THREADS, lv0 + p * THREADS, k, n, thn[p], thv[p]);
            else
                merge_values<KM, CAP, LS>(ln0 + p * THREADS, lv0 + p * THREADS, k, n, thn[p], thv[p]);
            off[p] = k * LS;
        }
    };

    // PRUNE: a bound row holds one value per 32 columns, (W + 31) / 32 + SPAN / 32 of them,
    // the value for a span starting at column x at (x >> 5) + SPAN / 32; the reference
    // epochs' share is fixed.  A warp whose row lies outside the image (its loads read zeros)
    // may add any value of the planes: none is negative, so the sum stays a bound.
    const long long RW = (long long)(a.W + 31) / 32 + SPAN / 32;
    const long long RE = (long long)N * a.H * RW;
    float b0 = 0.0f;
    if constexpr (PRUNE) {
        if (active)
            for (int j = 0; j < n0; ++j)
                b0 = __fadd_ru(b0, __ldg(a.snr2 + ((long long)a.epoch_of[j] * a.H + y) * RW + (xw >> 5) + SPAN / 32));
    }

    // Table build: a group of GL lanes takes one velocity, lane by lane its epochs, and keeps
    // (in time order) those whose shifted band overlaps the image for this CTA.  Leaving the
    // others out, which had read zero rows from L1, took 10 % of the loads at 12 x 4096^2
    // (28 % at 2048^2, more on smaller images).
    const int GL = NJ <= 4 ? 4 : NJ <= 8 ? 8 : NJ <= 16 ? 16 : 32;
    const int gl = lane & (GL - 1), gs = lane & ~(GL - 1);
    const unsigned gmask = (GL == 32 ? 0xffffffffu : (1u << GL) - 1u) << gs;
    const int vchunk = min(a.V, min(ROWS, TAB / max(NJP, 1)));
    // velocities whose bounds are taken at once, 32; MANY: the power of two that holds a chunk, and
    // 32 / bv lanes share a velocity's epochs
    int bv = 32;
    if constexpr (MANY) {
        while (bv / 2 >= vchunk) bv /= 2;
    }
    int v0 = 0, v1 = a.V;   // this CTA's velocities, in processing order
    if constexpr (SPLIT) {
        v0 = (int)((long long)a.V * part / parts);
        v1 = (int)((long long)a.V * (part + 1) / parts);
    }
    for (int c0 = v0; c0 < v1; c0 += vchunk) {
        const int nc = min(vchunk, v1 - c0);
        __syncthreads();
        for (int b = warp * (32 / GL); b < nc; b += WARPS * (32 / GL)) {
            const int vi = b + gs / GL;
            const bool ok = vi < nc;
            int cnt = 0;
            for (int j0 = 0; j0 < NJ; j0 += GL) {
                const int jj = j0 + gl, j = n0 + jj;
                int ep = 0, ox = 0, oy = 0;
                bool keep = false;
                if (ok && jj < NJ) {
                    ep = a.epoch_of[j];
                    const uint32_t o = a.ptab[(long long)(c0 + vi) * NJ + jj];   // packed (dx, dy)
                    ox = (int)(short)(o & 0xffffu);
                    oy = (int)o >> 16;
                    keep = xw + ox + SPAN > 0 && xw + ox < a.W && y0 + oy + WARPS > 0 && y0 + oy < a.H;
                }
                const unsigned m = __ballot_sync(0xffffffffu, keep) & gmask;
                const int at = vi * NJP + cnt + __popc(m & lt_mask);
                if (keep && debug_in(at, TAB, 5)) {
                    long long g = (long long)ep * a.plane_elems + (long long)oy * a.pitch + ox;
                    if (STORAGE != KB_F32 && (ox & 1)) g += a.phase1 - 1;   // odd shift: the phase-1 copy
                    E e;
                    e.idx = (I)LB::offset(g);
                    if constexpr (STORAGE != KB_F32) e.sc = sc_of(s_scale[j]);
                    s_tab[at] = e;
                    if constexpr (PRUNE)   // the CTA's first row; a warp adds warp * RW
                        s_rid[at + vi * (NJR - NJP)] = (I)(((long long)ep * a.H + y0 + oy) * RW + ((xw + ox) >> 5) + SPAN / 32);
                }
                cnt += __popc(m);
            }
            if (ok && gl == 0) s_vid[vi] = a.vorder[c0 + vi] | (cnt << 16);
        }
        __syncthreads();
        if (!active) continue;
        unsigned todo = 0u;   // PRUNE: of the 32 velocities around vi, those to gather
        for (int vi = 0; vi < nc; ++vi) {
            if constexpr (PRUNE) {
                if ((vi & 31) == 0) {
                    // a lane's velocity: its span's bound on nu^2, every step rounded upwards
                    const int mine = vi + (MANY ? lane & (bv - 1) : lane);
                    float b = !MANY || lane < bv ? b0 : 0.0f;
                    if (mine < nc) {
                        const I *rid = s_rid + mine * NJR;
                        const int n = s_vid[mine] >> 16;
                        if constexpr (MANY) {
                            // a bound that has reached nu_min^2 says no more: four epochs, then a look
                            const int by = 32 / bv;
                            for (int jj = lane / bv; jj < n && __fmul_ru(b, 1.0f + 0x1p-14f) < a.nu_min2_slack; jj += 4 * by) {
                                float r4[4];
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    r4[u] = 0.0f;
                                    if (jj + u * by < n) {
                                        const long long r = rid[jj + u * by] + (long long)warp * RW;
                                        r4[u] = __ldg(a.snr2 + max(0LL, min(RE - 1, r)));
                                    }
                                }
#pragma unroll
                                for (int u = 0; u < 4; ++u) b = __fadd_ru(b, r4[u]);
                            }
                        } else {
#pragma unroll 4
                            for (int jj = 0; jj < n; ++jj) {
                                const long long r = rid[jj] + (long long)warp * RW;
                                b = __fadd_ru(b, __ldg(a.snr2 + max(0LL, min(RE - 1, r))));
                            }
                        }
                    }
                    if constexpr (MANY) {
                        for (int o = bv; o < 32; o *= 2) b = __fadd_ru(b, __shfl_xor_sync(0xffffffffu, b, o));
                    }
                    todo = __ballot_sync(0xffffffffu, (!MANY || lane < bv) && mine < nc && !(__fmul_ru(b, 1.0f + 0x1p-14f) < a.nu_min2_slack));
                }
                const unsigned rest = todo >> (vi & 31);
                if (rest == 0u) {
                    vi |= 31;
                    continue;
                }
                vi += __ffs(rest) - 1;
            }
            const int v = s_vid[vi] & 0xffff, nj = s_vid[vi] >> 16;
            const E *tab = s_tab + vi * NJP;
            float2 acc[PX];
#pragma unroll
            for (int p = 0; p < PX; ++p) acc[p] = acc0[p];
            // the kept epochs in batches of C loads in flight, then one of four, then the
            // last one to three together (their loads issued before the first sum)
            int jj = 0;
            for (; jj + C <= nj; jj += C) add_epochs<STORAGE, P, C>(tab + jj, lane0, planes, a.planes_elems, acc);
            if constexpr (C > 4) {
                if (jj + 4 <= nj) {
                    add_epochs<STORAGE, P, 4>(tab + jj, lane0, planes, a.planes_elems, acc);
                    jj += 4;
                }
            }
            if (jj < nj) add_tail<STORAGE, P>(tab + jj, nj - jj, lane0, planes, a.planes_elems, acc);
            // scoring; candidates go to their pixels' buffers (the thresholds stay conservative
            // between merges: a stale one only admits more)
            bool full = false;
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                const float F = acc[p].y;
                const float nu = acc[p].x * rsqrtf(F);
                if constexpr (KEYS) {
                    const uint32_t key = nu_key(nu, v, a.key_bits);
                    if ((F > 0.0f) && (nu >= a.nu_min) && key > thk[p] && debug_in(off[p], off_lim, 6)) {
                        lk0[p * THREADS + off[p]] = key;
                        off[p] += LS;
                        full |= off[p] == off_lim;
                    }
                } else {
                    if ((F > 0.0f) && (nu >= a.nu_min) && better(nu, v, thn[p], thv[p]) && debug_in(off[p], off_lim, 6)) {
                        ln0[p * THREADS + off[p]] = nu;
                        lv0[p * THREADS + off[p]] = (uint16_t)v;
                        off[p] += LS;
                        full |= off[p] == off_lim;
                    }
                }
            }
            if (__any_sync(0xffffffffu, full)) merge_lists();
        }
    }
    if constexpr (SPLIT) {
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
        if (active) merge_lists();
        cluster.sync();   // every CTA's lists are complete
        if (active && warp % parts == part) {
            // the other CTAs' lists are sorted: each is read until an entry no longer counts
#pragma unroll 1
            for (int q = 0; q < parts; ++q) {
                if (q == part) continue;
#pragma unroll
                for (int p = 0; p < PX; ++p) {
                    if constexpr (KEYS) {
                        const uint32_t *rk = cluster.map_shared_rank(lk0 + p * THREADS, q);
                        uint32_t *lk = lk0 + p * THREADS;
                        for (int i = 0; i < k; ++i) {
                            const uint32_t ck = rk[i * LS];
                            if (ck <= lk[(k - 1) * LS]) break;
                            int j = k - 1;
                            for (; j > 0 && lk[(j - 1) * LS] < ck; --j) lk[j * LS] = lk[(j - 1) * LS];
                            lk[j * LS] = ck;
                        }
                    } else {
                        const float *rn = cluster.map_shared_rank(ln0 + p * THREADS, q);
                        const uint16_t *rv = cluster.map_shared_rank(lv0 + p * THREADS, q);
                        float *ln = ln0 + p * THREADS;
                        uint16_t *lv = lv0 + p * THREADS;
                        for (int i = 0; i < k; ++i) {
                            const float cn = rn[i * LS];
                            const int cv = rv[i * LS];
                            if (!better(cn, cv, ln[(k - 1) * LS], lv[(k - 1) * LS])) break;
                            int j = k - 1;
                            for (; j > 0 && better(cn, cv, ln[(j - 1) * LS], lv[(j - 1) * LS]); --j) {
                                ln[j * LS] = ln[(j - 1) * LS];
                                lv[j * LS] = lv[(j - 1) * LS];
                            }
                            ln[j * LS] = cn;
                            lv[j * LS] = (uint16_t)cv;
                        }
                    }
                }
            }
        }
        cluster.sync();   // no CTA leaves, or writes its columns again, before the others have read
        if (!active || warp % parts != part) return;
    } else {
        if (!active) return;
        merge_lists();
    }
    if constexpr (KEYS) {
        // candidates for the rescoring, best first, as the keys themselves (4 bytes each,
        // decoded by the rescoring, which recomputes the sums)
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            const int x = xw + (G::PIX == 1 ? lane + 32 * p : 2 * lane + 64 * (p / 2) + (p & 1));
            if (x >= a.W) continue;
            uint32_t *out = reinterpret_cast<uint32_t *>(a.out) + ((long long)y * a.W + x) * k;
            const uint32_t *lk = s_lk + p * THREADS + threadIdx.x;
            for (int i = 0; i < k; ++i) out[i] = lk[i * LS];
        }
        return;
    }

    // epilogue: recompute Psi, Phi (same operation sequence) and nobs of the kept entries;
    // every off-image epoch added a zero in the main loop, so it adds a zero here too.
    // Four epochs at a time: their offsets, then their gathers, then the sums in order.
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        const int x = xw + (G::PIX == 1 ? lane + 32 * p : 2 * lane + 64 * (p / 2) + (p & 1));
        if (x >= a.W) continue;
        Rec *out = a.out + ((long long)y * a.W + x) * k;
        const float *ln = s_ln + p * THREADS + threadIdx.x;
        const uint16_t *lv = s_lv + p * THREADS + threadIdx.x;
        for (int i = 0; i < k; ++i) {
            Rec r;
            const int v = lv[i * LS];
            if (v == kNoV) {
                r.psi = 0.0f;
                r.phi = 0.0f;
                r.nu = -INFINITY;
                r.meta = kEmptyVidx;
            } else if (a.cand_only) {
                r.psi = 0.0f;
                r.phi = 0.0f;
                r.nu = ln[i * LS];
                r.meta = (uint32_t)v;
            } else {
                const int2 *ov = a.offs + (long long)v * N;
                float2 acc = acc0[p];
                int nobs = n0;
                int j = n0;
                for (; j + 4 <= N; j += 4) {
                    T val[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int2 o = __ldg(ov + j + u);
                        const int xx = x + o.x, yy = y + o.y;
                        val[u] = St::zero();
                        if ((unsigned)xx < (unsigned)a.W && (unsigned)yy < (unsigned)a.H) {
                            val[u] = St::load(planes + (long long)a.epoch_of[j + u] * a.plane_elems + a.origin +
                                              (long long)yy * a.pitch + xx);
                            ++nobs;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc = St::acc(acc, val[u], s_scale[j + u]);
                }
                for (; j < N; ++j) {
                    const int2 o = __ldg(ov + j);
                    const int xx = x + o.x, yy = y + o.y;
                    T val = St::zero();
                    if ((unsigned)xx < (unsigned)a.W && (unsigned)yy < (unsigned)a.H) {
                        val = St::load(planes + (long long)a.epoch_of[j] * a.plane_elems + a.origin +
                                       (long long)yy * a.pitch + xx);
                        ++nobs;
                    }
                    acc = St::acc(acc, val, s_scale[j]);
                }
                r.psi = acc.x;
                r.phi = acc.y;
                r.nu = ln[i * LS];
                r.meta = (uint32_t)v | ((uint32_t)nobs << 16);
            }
            reinterpret_cast<uint4 *>(out)[i] = *reinterpret_cast<uint4 *>(&r);
        }
    }
}

// Resident CTAs per SM the register allocation is held to, by shape.  Lists up to 8
// long: the narrow shapes (FP32 with two pixels per lane, 16-bit with one pixel pair) are
// held to 4 CTAs (64 registers; at 5 CTAs, 48 registers, FP32 spills in the loop: 12 x 4096^2,
// k = 8, 136 ms against 76); 16-bit with two pixel pairs per lane to 3 with 4-epoch batches
// (80 registers) and 2 with 8-epoch batches.  Longer lists: 3.  The wide FP32 shapes: 2.  The
// batch kernel, which keeps its search's arguments in shared memory rather than the parameter
// bank and so needs more registers, is held to 3 for the narrow shapes and 2 for the others.
// FP32's automatic kernels and FP16's value lists fit; a few values of the others live in local
// memory: BF16 (1, 4) 8 bytes of stores, key lists (2, 4) 16, BF16 (1, 8) with lists of 9 to 16 52,
// BF16's batch kernels 4 to 52, pruned FP32 with lists up to 8 8 (its form for many epochs none).
template <int STORAGE, int P, int C, int KM, bool KEYS>
constexpr int min_ctas() {
    constexpr bool narrow = STORAGE == KB_F32 ? P <= 2 : P <= 1;
    if (STORAGE != KB_F32 && P == 2) return (C <= 4 && KM <= kKeyMax && (KEYS || KM <= kShortMax)) ? 3 : 2;
    if (!narrow) return 2;
    return KM > kShortMax ? 3 : 4;
}

template <int STORAGE, int P>
constexpr int min_ctas_batch() {
    return (STORAGE == KB_F32 ? P <= 2 : P <= 1) ? 3 : 2;
}

template <int STORAGE, int P, int C, int KM, typename I, bool PRUNE, bool KEYS, bool SPLIT, bool CUT>
__global__ void __launch_bounds__(THREADS, min_ctas<STORAGE, P, C, KM, KEYS>())
    search_kernel(SearchArgs a) {
    __shared__ float2 s_scale[KB_MAX_EPOCHS];
    extern __shared__ int4 s_dyn4[];
    int bx = blockIdx.x, by = blockIdx.y;
    if (a.swz > 0 && a.swz < (int)gridDim.x) {
        // CTAs start roughly in linear order: deal the tiles out in super-columns of
        // swz tiles, row by row within each (the last super-column may be narrower)
        const int gx = gridDim.x, lin = blockIdx.y * gx + blockIdx.x;
        const int per = a.swz * gridDim.y, s = lin / per, r = lin - s * per;
        const int w = min(a.swz, gx - s * a.swz);
        by = r / w;
        bx = s * a.swz + (r - by * w);
    }
    // SPLIT: a cluster is the grid's whole z extent, so z is the CTA's rank in it
    search_tile<STORAGE, P, C, KM, I, PRUNE, KEYS, SPLIT, CUT>(a, bx, a.by0 + by, s_scale, s_dyn4,
                                                               SPLIT ? blockIdx.z : 0, SPLIT ? gridDim.z : 1);
}

// Persistent batch search: CTAs take (job, tile) work items from an atomic
// counter until the list is exhausted, copying the item's job descriptor into
// shared memory first.  The item list is ordered by cost (largest first), so
// uneven stacks, grids and epoch counts balance across the SMs.
template <int STORAGE, int P, int C, int KM, typename I, bool CUT>
__global__ void __launch_bounds__(THREADS, min_ctas_batch<STORAGE, P>())
    search_batch_kernel(const SearchArgs *jobs, const int4 *items, int n_items, int *counter, int slots) {
    __shared__ float2 s_scale[KB_MAX_EPOCHS];
    __shared__ SearchArgs s_job;
    __shared__ int s_it;
    extern __shared__ int4 s_dyn4[];
    for (;;) {
        if (threadIdx.x == 0) s_it = atomicAdd(counter, 1);
        __syncthreads();
        const int it = s_it;
        if (it >= n_items) break;
        const int4 w = items[it];
        for (int i = threadIdx.x; i < (int)(sizeof(SearchArgs) / sizeof(int)); i += THREADS)
            reinterpret_cast<int *>(&s_job)[i] = CUT && i == (int)(offsetof(SearchArgs, slots) / sizeof(int))
                                                     ? slots
                                                     : reinterpret_cast<const int *>(jobs + w.x)[i];
        __syncthreads();
        search_tile<STORAGE, P, C, KM, I, false, false, false, CUT>(s_job, w.y, w.z, s_scale, s_dyn4);
        __syncthreads();
    }
}

// dynamic shared memory of a CTA with lists of k entries and buffers of cap: the table, and the
// lists with their buffers
template <int STORAGE, int P, int KM, typename I, bool PRUNE = false, bool KEYS = false, bool MANY = false>
size_t tile_smem(int k, int cap) {
    constexpr int PX = P * Gather<STORAGE>::PIX;
    constexpr int TAB = table_entries<STORAGE, I, PRUNE>(), RID = PRUNE ? TAB + (MANY ? TAB / 4 : 0) : 0;
    return (size_t)TAB * table_entry_bytes<STORAGE, I>() + RID * sizeof(I) + TAB / 4 * sizeof(int) +
           (size_t)(k + cap) * THREADS * PX *
               (KEYS ? sizeof(uint32_t) : sizeof(float) + sizeof(uint16_t));
}

// Buffer entries of a launch whose lists are long or keys (njs: its searches' most epochs past the
// reference time).  The resident CTAs' shared memory takes 100, 132, 164, 196 or 228 KB of an
// SM's 256, the L1 gets the rest, and the more epochs a velocity has, the more L1 its early
// epochs need to stay there until the next velocity; the merges that shorter buffers add weigh
// less by the same measure.  The longest buffer is taken unless a shorter one, no shorter than
// `least`, brings the CTAs into the next split down or lets another CTA in.  Measured, ms (split
// in KB, entries):
//   FP32 k = 16, 5 x 1500^2, 512 velocities: 228, 5: 6.0; 196, 4: 6.7; 12 x 4096^2, 512: 77.5 and 67.2;
//     20 x 1900^2, 512: 32.9 and 22.1; 24 x 4096^2, 96: 136.6 and 73.1
//   FP16 k = 16, 12 x 4096^2, 512: 228, 5: 70.0; 196, 3: 76.4; 16 x 1900^2, 512: 19.2 and 19.4;
//     16 x 4096^2, 96: 47.6 and 37.2; 20 x 1900^2, 512: 24.1 and 21.6; 24 x 4096^2, 96: 102.5 and 57.2
//   FP32 k = 14, 20 x 1900^2, 512: 196, 5: 20.0; 164, 3: 20.6; 24 x 4096^2, 96: 65.2 and 52.5
//   FP16 k = 12, 20 x 1900^2, 512: 196, 5: 16.8; 164, 4: 17.0; 24 x 4096^2, 96: 44.9 and 38.9
//   FP32 k = 9, 20 x 1900^2, 512: 164, 5: 15.9; 132, 4: 16.0; 24 x 4096^2, 96: 36.8 and 34.2
//   FP16 k = 9, 24 x 4096^2, 96: 164, 5: 31.2; 132, 3: 33.5; 40 x 4096^2, 64: 58.2 and 52.6
//   BF16 keys, k_c = 12, 4096^2, 24 / 40 / 59: 228, 4: 38.6 / 61.7 / 96.7; 196, 2: 39.7 / 59.0 / 90.9
//   FP16 candidates, k_c = 20, 12 x 2048^2 / 40 x 4096^2: two CTAs, 5: 27.2 / 154; three, 3: 24.0 / 147
//     (128 x 1024^2: 34.1 and 35.1)
// The persistent batch kernel (BATCH), whose searches are mixed, leaves only the 228 KB split in
// 16-bit storage, above 20 epochs (three searches of 0.5 to 1 M pixels, BF16, k = 16, 8 to 20
// epochs: 10.2 ms as it is, 12.6 with buffers of 3; 26 to 38 epochs: 25.9 and 20.4).
template <int STORAGE, int P, int KM, typename I, bool PRUNE, bool KEYS, bool BATCH, typename Kern>
cudaError_t buffer_cap(Kern kern, int k, int njs, int &cap) {
    cap = list_cap<KM, KEYS, P * Gather<STORAGE>::PIX>();
    if (KM <= kShortMax) return cudaSuccess;
    cudaFuncAttributes fa;
    cudaError_t err = cudaFuncGetAttributes(&fa, kern);
    if (err != cudaSuccess) return err;
    constexpr bool F32 = STORAGE == KB_F32;
    const size_t KB = 1024, own = fa.sharedSizeBytes + KB;   // each CTA's static share and the system's
    const int by_regs = 65536 / (((fa.numRegs + 7) & ~7) * THREADS);
    auto bytes = [&](int c) { return tile_smem<STORAGE, P, KM, I, PRUNE, KEYS>(k, c) + own; };
    auto ctas = [&](int c) { return std::min(by_regs, (int)(228 * KB / bytes(c))); };
    auto split = [&](int c) {
        const size_t all = ctas(c) * bytes(c);
        for (int kb = 100; kb < 228; kb += 32)
            if (all <= kb * KB) return kb;
        return 228;
    };
    auto least = [&](int from) {   // the shortest buffer that is worth leaving a split
        constexpr int none = 99;
        if (KEYS) return from == 228 && njs > 32 ? 2 : none;
        if (BATCH && !F32) return from == 228 && njs > 20 ? 2 : none;
        if (njs <= 20 && from == 228) return njs <= 8 ? none : njs <= 12 ? 4 : 3;
        if (from == 228) return 2;
        if (njs <= 20) return none;
        if (from == 196) return F32 || njs > 48 ? 2 : 3;
        return F32 ? (njs <= 32 ? 4 : 3) : njs <= 48 ? none : 3;
    };
    for (int c = cap - 1; c >= 2; --c) {
        if (ctas(c) > ctas(cap) ? c >= 3 && njs <= 64 : ctas(c) == ctas(cap) && split(c) < split(cap) && c >= least(split(cap)))
            cap = c;
    }
    return cudaSuccess;
}

// the shapes of the automatic choice (launch_storage): they have a kernel for buffers of their full
// length, a constant, and one whose slots come with the launch (which takes BF16 3 % longer)
template <int STORAGE, int P, int C, int KM, bool PRUNE, bool KEYS>
constexpr bool auto_shape() {
    return !PRUNE && (KEYS || (STORAGE == KB_F32 ? P == 2 && C == 8 : P == 1 && C == (KM > kShortMax ? 8 : 4)));
}

// CTAs (a cluster) that share a tile's velocities: as many of 2, 4 or 8 as leave the launch
// within one wave of resident CTAs, with at least 16 velocities each.  A launch of a few tiles
// leaves most SMs idle otherwise: 5 x 64 x 64, 256 velocities is 8 tiles and 171 us, with 8 CTAs
// per tile 59; beyond one wave the lists' extra work (each CTA fills its own) is not repaid.
template <int STORAGE, int P, int C, int KM, bool KEYS>
int split_of(const SearchArgs &a, dim3 grid) {
    int s = 1;
    while (s < 8 && (long long)grid.x * grid.y * (2 * s) <= 152LL * min_ctas<STORAGE, P, C, KM, KEYS>() &&
           a.V >= 16 * (2 * s))
        s *= 2;
    return s;
}

// the other shapes' kernels for long lists: with the launch's slots, but for wide 16-bit ones,
// whose CTAs are one or two per SM either way
template <int STORAGE, int P, int KM>
constexpr bool always_cut() { return KM > kShortMax && (STORAGE == KB_F32 || P == 1); }

template <int STORAGE, int P, int C, int KM, typename I, bool PRUNE, bool KEYS = false>
cudaError_t launch_pt(const SearchArgs &search, cudaStream_t st) {
    SearchArgs a = search;
    constexpr int SPAN = 32 * P * Gather<STORAGE>::PIX;
    static_assert(SPAN <= kSpan, "warp span wider than the zero columns");
    dim3 grid((a.W + SPAN - 1) / SPAN, a.nby > 0 ? a.nby : (a.H + WARPS - 1) / WARPS);
    constexpr bool kAuto = auto_shape<STORAGE, P, C, KM, PRUNE, KEYS>(), kLong = KM > kShortMax;
    // the automatic shapes with 32-bit offsets have a form for small launches
    constexpr bool kSplit = kAuto && sizeof(I) == 4 && KM <= kKeyMax;
    constexpr int CAP = list_cap<KM, KEYS, P * Gather<STORAGE>::PIX>();
    int parts = 1, cap = CAP;
    if constexpr (kSplit) {
        if (a.variant == 0) parts = split_of<STORAGE, P, C, KM, KEYS>(a, grid);
    }
    constexpr bool kCut = !kAuto && always_cut<STORAGE, P, KM>();
    auto kern = search_kernel<STORAGE, P, C, KM, I, PRUNE, KEYS, false, kCut>;
    cudaError_t err = cudaSuccess;
    if (parts == 1 && (kAuto || kCut)) err = buffer_cap<STORAGE, P, KM, I, PRUNE, KEYS, false>(kern, a.k, a.N - a.n0, cap);
    if (err != cudaSuccess) return err;
    if constexpr (kLong && kAuto) {
        if (cap < CAP) kern = search_kernel<STORAGE, P, C, KM, I, PRUNE, KEYS, false, true>;
    }
    if constexpr (kSplit) {
        if (parts > 1) kern = search_kernel<STORAGE, P, C, KM, I, PRUNE, KEYS, true, false>;
    }
    size_t smem = tile_smem<STORAGE, P, KM, I, PRUNE, KEYS>(a.k, cap);
    if constexpr (many_epochs<STORAGE, KM, PRUNE, true>()) {
        if (a.N - a.n0 > kPruneMany) {
            // 4 CTAs (and the system's 1 KB of each) within the 164 KB split of shared memory
            kern = search_kernel<STORAGE, P, C, KM, I, PRUNE, KEYS, false, true>;
            do
                smem = tile_smem<STORAGE, P, KM, I, PRUNE, KEYS, true>(a.k, cap);
            while (smem > 40 * 1024 && --cap > 1);
        }
    }
    a.slots = a.k + cap;
    err = allow_smem(kern);
    // Shared-memory carveout: the driver's choice (-1) unless the caller sets one
    // (kb_set_search_carveout); it trades resident CTAs against the L1 that the
    // early epochs' gathers reuse across velocities.
    if (err == cudaSuccess)
        err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, a.carveout);
    if (err != cudaSuccess) return err;
    if (parts > 1) {
        grid.z = parts;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = parts;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, a);
    }
    kern<<<grid, THREADS, smem, st>>>(a);
    return cudaGetLastError();
}

// the merge by the lists' length (candidate lists reach 24: k = 16, BF16)
template <int STORAGE, int P, int C, typename I, bool PRUNE>
cudaError_t launch_one(const SearchArgs &a, cudaStream_t st) {
    if (a.k > kKeyMax) return launch_pt<STORAGE, P, C, kListMax, I, PRUNE>(a, st);
    if (a.k > kShortMax) return launch_pt<STORAGE, P, C, kKeyMax, I, PRUNE>(a, st);
    return launch_pt<STORAGE, P, C, kShortMax, I, PRUNE>(a, st);
}

// the candidate search of the FP64 rescoring in key form (automatic shape, no pruning)
template <int STORAGE, int P, int C>
cudaError_t launch_keys(const SearchArgs &a, cudaStream_t st) {
    if (search_idx32(a, true)) return launch_pt<STORAGE, P, C, kKeyMax, int, false, true>(a, st);
    return launch_pt<STORAGE, P, C, kKeyMax, long long, false, true>(a, st);
}

// key form where it keeps at least 11 of nu's 23 fraction bits (up to 4096 velocities)
bool key_lists(int V, int k) { return k <= kKeyMax && V <= 4096; }
bool use_keys(const SearchArgs &a) { return a.cand_only && !a.snr2 && key_lists(a.V, a.k); }

// 32-bit offsets when every plane of both phases (and the bound planes) is in their reach
template <int STORAGE, int P, int C, bool PRUNE = false>
cudaError_t launch_idx(const SearchArgs &a, cudaStream_t st) {
    const long long rspan = PRUNE ? (long long)a.N * a.H * ((a.W + 31) / 32 + P * Gather<STORAGE>::PIX) : 0;
    const bool elements = PRUNE && STORAGE == KB_F32 && a.k <= kShortMax && a.N - a.n0 > kPruneMany;   // MANY
    if (search_idx32(a, elements) && rspan < (1LL << 31) - 1) return launch_one<STORAGE, P, C, int, PRUNE>(a, st);
    return launch_one<STORAGE, P, C, long long, PRUNE>(a, st);
}

// Shapes: (loads per lane P, epochs per load batch C); a 16-bit load is two pixels.  search_shape
// makes the choice.  Automatic: FP32 (2, 8), 12 x 4096^2, k = 8: 76 ms; 16-bit value lists up to 8
// long (1, 4), 12 x 2048^2, 1024 velocities, k = 8, BF16 / FP16: 18.6 / 18.8 ms, (1, 8) 20.8 / 20.7;
// longer ones (1, 8), 12 x 1800^2, 1024 velocities, k = 12, BF16: 18.7 ms, (1, 4) 21.9, (2, 4) 20.8,
// (2, 8) 23.2.  Key lists take two pairs per lane, value lists one, whose merges fit the registers
// beside the loop (pruned short ones two, as their bound planes' span has it).
template <int STORAGE>
cudaError_t launch_storage(const SearchArgs &a, cudaStream_t st) {
    const bool own = a.variant == 0, keys = own && use_keys(a), pruned = own && a.snr2;
    const int shape = search_shape(a.storage, a.variant, a.k, keys, pruned);
    if constexpr (STORAGE == KB_F32) {
        if (pruned) return launch_idx<STORAGE, 2, 8, true>(a, st);
        if (keys) return launch_keys<STORAGE, 2, 8>(a, st);
        switch (shape) {
            case 1: return launch_idx<STORAGE, 4, 4>(a, st);
            case 2: return launch_idx<STORAGE, 2, 4>(a, st);
            case 3: return launch_idx<STORAGE, 4, 8>(a, st);
            default: return launch_idx<STORAGE, 2, 8>(a, st);
        }
    } else {
        if (pruned) return shape == 2 ? launch_idx<STORAGE, 1, 4, true>(a, st) : launch_idx<STORAGE, 2, 4, true>(a, st);
        if (keys) return launch_keys<STORAGE, 2, 4>(a, st);
        switch (shape) {
            case 1: return launch_idx<STORAGE, 2, 4>(a, st);
            case 2: return launch_idx<STORAGE, 1, 4>(a, st);
            case 3: return launch_idx<STORAGE, 2, 8>(a, st);
            default: return launch_idx<STORAGE, 1, 8>(a, st);
        }
    }
}

template <int STORAGE, int P, int C, int KM, typename I>
cudaError_t launch_batch_pt(const SearchArgs *jobs, const int4 *items, int n_items, int *counter, int kmax,
                            int njs, int carve, int sm_count, cudaStream_t st) {
    constexpr bool kAuto = auto_shape<STORAGE, P, C, KM, false, false>(), kLong = KM > kShortMax;
    constexpr int CAP = list_cap<KM, false, P * Gather<STORAGE>::PIX>();
    constexpr bool kCut = !kAuto && always_cut<STORAGE, P, KM>();
    auto kern = search_batch_kernel<STORAGE, P, C, KM, I, kCut>;
    int cap = CAP;
    cudaError_t err = cudaSuccess;
    if (kAuto || kCut) err = buffer_cap<STORAGE, P, KM, I, false, false, true>(kern, kmax, njs, cap);
    if (err != cudaSuccess) return err;
    if constexpr (kLong && kAuto) {
        if (cap < CAP) kern = search_batch_kernel<STORAGE, P, C, KM, I, true>;
    }
    const size_t smem = tile_smem<STORAGE, P, KM, I>(kmax, cap);
    err = allow_smem(kern);
    if (err == cudaSuccess)
        err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, carve);
    int per_sm = 0;
    if (err == cudaSuccess) err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, THREADS, smem);
    if (err != cudaSuccess) return err;
    // persistent grid: every SM filled with as many CTAs as it can hold
    const int grid = sm_count * (per_sm > 0 ? per_sm : 1);
    kern<<<grid, THREADS, smem, st>>>(jobs, items, n_items, counter, kmax + cap);
    return cudaGetLastError();
}

template <int STORAGE, int P, int C, typename I>
cudaError_t launch_batch_one(const SearchArgs *jobs, const int4 *items, int n_items, int *counter, int kmax,
                             int njs, int carve, int sm_count, cudaStream_t st) {
    if (kmax > kKeyMax)
        return launch_batch_pt<STORAGE, P, C, kListMax, I>(jobs, items, n_items, counter, kmax, njs, carve, sm_count, st);
    if (kmax > kShortMax)
        return launch_batch_pt<STORAGE, P, C, kKeyMax, I>(jobs, items, n_items, counter, kmax, njs, carve, sm_count, st);
    return launch_batch_pt<STORAGE, P, C, kShortMax, I>(jobs, items, n_items, counter, kmax, njs, carve, sm_count, st);
}

template <int STORAGE, int P, int C>
cudaError_t launch_batch_idx(const SearchArgs *jobs, const int4 *items, int n_items, int *counter, int kmax,
                             int njs, int carve, bool idx64, int sm_count, cudaStream_t st) {
    if (idx64)
        return launch_batch_one<STORAGE, P, C, long long>(jobs, items, n_items, counter, kmax, njs, carve, sm_count, st);
    return launch_batch_one<STORAGE, P, C, int>(jobs, items, n_items, counter, kmax, njs, carve, sm_count, st);
}

template <int STORAGE>
cudaError_t launch_batch_storage(const SearchArgs *jobs, const int4 *items, int n_items, int *counter, int variant,
                                 int kmax, int njs, int carve, bool idx64, int sm_count, cudaStream_t st) {
    if constexpr (STORAGE == KB_F32) {
        switch (variant) {
            case 1: return launch_batch_idx<STORAGE, 4, 4>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
            case 2: return launch_batch_idx<STORAGE, 2, 4>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
            case 3: return launch_batch_idx<STORAGE, 4, 8>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
            default: return launch_batch_idx<STORAGE, 2, 8>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
        }
    } else {
        switch (variant) {
            case 2: return launch_batch_idx<STORAGE, 1, 4>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
            case 3: return launch_batch_idx<STORAGE, 2, 8>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
            case 4: return launch_batch_idx<STORAGE, 1, 8>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
            default: return launch_batch_idx<STORAGE, 2, 4>(jobs, items, n_items, counter, kmax, njs, carve, idx64, sm_count, st);
        }
    }
}

}  // namespace

template <>
cudaError_t launch_search_storage<KB_SEARCH_STORAGE>(const SearchArgs &a, cudaStream_t st) {
    return launch_storage<KB_SEARCH_STORAGE>(a, st);
}
template <>
cudaError_t launch_search_batch_storage<KB_SEARCH_STORAGE>(const SearchArgs *jobs, const int4 *items, int n_items,
                                                           int *counter, int variant, int kmax, int njs, int carve, bool idx64,
                                                           int sm_count, cudaStream_t st) {
    return launch_batch_storage<KB_SEARCH_STORAGE>(jobs, items, n_items, counter, variant, kmax, njs, carve, idx64, sm_count, st);
}
template <>
cudaError_t debug_word_storage<KB_SEARCH_STORAGE>(unsigned long long *word, bool reset) {
#ifdef KB_DEBUG
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(word, g_debug_word, sizeof(*word));
    if (e == cudaSuccess && reset) {
        const unsigned long long zero = 0;
        e = cudaMemcpyToSymbol(g_debug_word, &zero, sizeof(zero));
    }
    return e;
#else
    (void)word;
    (void)reset;
    return cudaErrorNotSupported;
#endif
}

#ifdef KB_SEARCH_COMMON

cudaError_t debug_word(unsigned long long *word, bool reset) {
    unsigned long long w[3] = {0, 0, 0};
    cudaError_t e = debug_word_storage<KB_F32>(&w[0], reset);
    if (e == cudaSuccess) e = debug_word_storage<KB_BF16>(&w[1], reset);
    if (e == cudaSuccess) e = debug_word_storage<KB_F16>(&w[2], reset);
    *word = w[0] ? w[0] : w[1] ? w[1] : w[2];
    return e;
}

int search_shape(int storage, int variant, int k, bool keys, bool pruned) {
    if (variant >= 1 && variant <= 4) return variant;
    if (storage == KB_F32) return 4;                  // (2, 8)
    if (keys) return 1;                               // (2, 4)
    if (pruned) return k > kShortMax ? 2 : 1;         // (1, 4), (2, 4)
    return k > kShortMax ? 4 : 2;                     // (1, 8), (1, 4)
}

int search_span(int storage, int shape) {
    // loads per lane P of the shape, times 32 lanes, times pixels per load
    static const int p32[5] = {0, 4, 2, 4, 2}, p16[5] = {0, 2, 1, 2, 1};
    return storage == KB_F32 ? 32 * p32[shape] : 64 * p16[shape];
}

bool search_key_lists(int V, int k) { return key_lists(V, k); }

cudaError_t launch_search_batch(const SearchArgs *jobs, const int4 *items, int n_items, int *counter, int storage,
                                int variant, int kmax, int njs, int carve, bool idx64, int sm_count, cudaStream_t st) {
    switch (storage) {
        case KB_F32: return launch_search_batch_storage<KB_F32>(jobs, items, n_items, counter, variant, kmax, njs, carve, idx64, sm_count, st);
        case KB_BF16: return launch_search_batch_storage<KB_BF16>(jobs, items, n_items, counter, variant, kmax, njs, carve, idx64, sm_count, st);
        case KB_F16: return launch_search_batch_storage<KB_F16>(jobs, items, n_items, counter, variant, kmax, njs, carve, idx64, sm_count, st);
        default: return cudaErrorInvalidValue;
    }
}

bool search_keys(const SearchArgs &a) { return a.variant == 0 && use_keys(a); }

cudaError_t launch_search(const SearchArgs &a, cudaStream_t st) {
    switch (a.storage) {
        case KB_F32: return launch_search_storage<KB_F32>(a, st);
        case KB_BF16: return launch_search_storage<KB_BF16>(a, st);
        case KB_F16: return launch_search_storage<KB_F16>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

#endif  // KB_SEARCH_COMMON

}  // namespace kb
