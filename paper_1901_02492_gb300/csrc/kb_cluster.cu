// Sec. 3.3 de-duplication of candidate trajectories: DBSCAN over (x0, y0, vx, vy).
//
// Distance, core points, clusters, border and noise points are as documented at
// kb_cluster in include/kb.h.  The GPU form:
//   - a first pass packs each candidate into 16 bytes (x0, y0, vx, vy) and
//     computes its cell of a 4-D uniform grid of cells a little wider than eps
//     (in the weighted coordinates), so that every neighbour of a point lies in
//     the 3^4 cells around its own; the cells live in an open-addressing hash
//     table, and the points of a cell are gathered into one contiguous run
//     (counted while they are inserted; the runs' places come from an atomic
//     cursor, so their order is arbitrary and no result depends on it);
//   - a warp takes one point: its lanes look up the 81 cells side by side, then
//     share the candidates of all of them, 32 at a time.  A thread per point
//     walking linked lists spent its time in the dense groups around bright
//     sources, one dependent load after the other: 262,144 candidates of a
//     12 x 2048^2 search, core pass 1.92 -> 0.23 ms, unions 3.75 -> 0.32 ms, borders
//     0.24 -> 0.09 ms;
//   - distances are first taken in FP32, whose error is far below the margin it is
//     given; only pairs within 2^-16 of eps take the FP64 distance (this GPU has two
//     FP64 lanes per SM and cycle), and pairs already in one cluster take none;
//   - neighbour counts (stopping at min_samples) give the core points;
//   - a lock-free union-find over the core points, always hooking the larger
//     root under the smaller, so every cluster ends rooted at its lowest core
//     index whatever the order of the unions;
//   - border points take the root of their nearest core neighbour (smallest d2,
//     then lowest index), noise points their own index;
//   - per group, an atomic maximum of the ordered nu bits, then an atomic
//     minimum of the index among the members that reach it.
// The squared distance is evaluated with explicitly rounded FP64 operations in a
// fixed order (no contraction into FMA), so neighbour decisions are exact and
// deterministic.  Every loop is bounded; a bound that is reached sets the status
// word instead of spinning.
#include <math.h>

#include <algorithm>

#include "kb_internal.h"

namespace kb {
namespace {

constexpr int kThreads = 256;
constexpr uint8_t kAlone = 2;   // valid[i] of a point without another in its 81 cells

// Points are packed as (x0, y0, bits of vx, bits of vy).
__device__ __forceinline__ double dist2(int4 a, int4 b, double w_pos, double w_vel) {
    const double ax = __dmul_rn((double)((long long)a.x - (long long)b.x), w_pos);
    const double ay = __dmul_rn((double)((long long)a.y - (long long)b.y), w_pos);
    const double au = __dmul_rn(__dsub_rn((double)__int_as_float(a.z), (double)__int_as_float(b.z)), w_vel);
    const double av = __dmul_rn(__dsub_rn((double)__int_as_float(a.w), (double)__int_as_float(b.w)), w_vel);
    return __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(ax, ax), __dmul_rn(ay, ay)), __dmul_rn(au, au)),
                     __dmul_rn(av, av));
}

// dist2(a, b) <= eps2.  In FP32 the coordinate differences of the start pixels are exact (below
// 2^24, else rounded), each product and sum is rounded once, so d is within 2^-20 of dist2;
// the FP64 form decides the pairs within 2^-16 of eps2, and all of them where eps2 is outside
// the range in which FP32 keeps that accuracy (NaN limits: no comparison holds).
__device__ __forceinline__ bool within(const ClusterArgs &a, int4 p, int4 q) {
    const float wp = (float)a.w_pos, wv = (float)a.w_vel;
    const float ax = (float)(p.x - q.x) * wp, ay = (float)(p.y - q.y) * wp;
    const float au = (__int_as_float(p.z) - __int_as_float(q.z)) * wv;
    const float av = (__int_as_float(p.w) - __int_as_float(q.w)) * wv;
    const float d = ((ax * ax + ay * ay) + au * au) + av * av;
    if (d < a.eps2_lo) return true;
    if (d > a.eps2_hi) return false;
    return dist2(p, q, a.w_pos, a.w_vel) <= a.eps2;
}

// Grid cell of a candidate; false when a coordinate is too far from the origin
// in units of the cell width (the caller's weights and eps are unusable then).
__device__ __forceinline__ bool cell_of(const kb_result &r, const ClusterArgs &a, int4 &c) {
    const double f0 = (double)r.x0 * a.w_pos * a.inv_side, f1 = (double)r.y0 * a.w_pos * a.inv_side;
    const double f2 = (double)r.vx * a.w_vel * a.inv_side, f3 = (double)r.vy * a.w_vel * a.inv_side;
    const double lim = 1073741824.0;   // 2^30
    if (!(fabs(f0) < lim && fabs(f1) < lim && fabs(f2) < lim && fabs(f3) < lim)) return false;
    c = make_int4((int)floor(f0), (int)floor(f1), (int)floor(f2), (int)floor(f3));
    return true;
}

__device__ __forceinline__ unsigned hash4(int4 c, unsigned mask) {
    unsigned long long h = (unsigned long long)(unsigned)c.x * 0x9E3779B97F4A7C15ull;
    h ^= (unsigned long long)(unsigned)c.y * 0xC2B2AE3D27D4EB4Full;
    h ^= (unsigned long long)(unsigned)c.z * 0x165667B19E3779F9ull;
    h ^= (unsigned long long)(unsigned)c.w * 0xD6E8FEB86659FD93ull;
    h ^= h >> 31;
    h *= 0x94D049BB133111EBull;
    h ^= h >> 29;
    return (unsigned)h & mask;
}

__device__ __forceinline__ int4 point_of(const kb_result &r) {
    return make_int4(r.x0, r.y0, __float_as_int(r.vx), __float_as_int(r.vy));
}

__device__ __forceinline__ bool same_cell(const ClusterArgs &a, int o, int4 c) {
    const int4 d = a.cells[o];
    return d.x == c.x && d.y == c.y && d.z == c.z && d.w == c.w;
}

// The first candidate of cell c, or -1.
__device__ int find_cell(const ClusterArgs &a, int4 c) {
    unsigned s = hash4(c, a.T - 1);
    for (int probe = 0; probe < a.T; ++probe) {
        const int o = a.owner[s];
        if (o < 0) return -1;
        if (same_cell(a, o, c)) return o;
        s = (s + 1) & (a.T - 1);
    }
    return -1;
}

__device__ __forceinline__ unsigned long long nu_key(double nu) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(nu);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__device__ int find_root(volatile int *parent, int x, int n, int *status) {
    for (int it = 0; it <= n; ++it) {
        const int p = parent[x];
        if (p == x) return x;
        const int g = parent[p];
        if (g != p) parent[x] = g;   // path halving: g is an ancestor of x
        x = p;
    }
    atomicExch(status, 2);
    return x;
}

__global__ void init_kernel(ClusterArgs a) {
    const int stride = gridDim.x * blockDim.x;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < a.T; s += stride) {
        a.owner[s] = -1;
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
        a.cnt[i] = 0;
        a.parent[i] = i;
        a.bestidx[i] = 0x7fffffff;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.count = 0u;
        *a.status = 0;
        *a.cursor = 0;
    }
}

__global__ void prep_kernel(ClusterArgs a) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        const kb_result r = a.cand[i];
        int4 c = make_int4(0, 0, 0, 0);
        bool ok = r.vidx >= 0;
        if (ok && !cell_of(r, a, c)) {
            atomicExch(a.status, 1);
            ok = false;
        }
        a.cells[i] = c;
        a.valid[i] = ok ? 1 : 0;
    }
}

__global__ void insert_kernel(ClusterArgs a) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        if (!a.valid[i]) continue;
        const int4 c = a.cells[i];
        unsigned s = hash4(c, a.T - 1);
        bool placed = false;
        for (int probe = 0; probe < a.T && !placed; ++probe) {
            const int o = atomicCAS(&a.owner[s], -1, i);
            if (o == -1 || same_cell(a, o, c)) {
                const int first = o == -1 ? i : o;
                a.first[i] = first;
                a.rank[i] = atomicAdd(&a.cnt[first], 1);
                placed = true;
            } else {
                s = (s + 1) & (a.T - 1);
            }
        }
        if (!placed) {   // no slot left: the point takes no part
            atomicExch(a.status, 2);
            a.valid[i] = 0;
        }
    }
}

// the place of every cell's run
__global__ void place_kernel(ClusterArgs a) {
    const int lane = threadIdx.x & 31;
    for (int s0 = blockIdx.x * blockDim.x + threadIdx.x - lane; s0 < a.n; s0 += gridDim.x * blockDim.x) {
        const int s = s0 + lane, c = s < a.n ? a.cnt[s] : 0;
        int end = c;   // one atomic for the warp's cells
#pragma unroll
        for (int o = 1; o < 32; o *= 2) {
            const int e = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += e;
        }
        int base = 0;
        if (lane == 31) base = atomicAdd(a.cursor, end);
        base = __shfl_sync(0xffffffffu, base, 31);
        if (c > 0) a.start[s] = base + end - c;
    }
}

__global__ void gather_kernel(ClusterArgs a) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        if (!a.valid[i]) continue;
        const int at = a.start[a.first[i]] + a.rank[i];
        a.run_pts[at] = point_of(a.cand[i]);
        a.run_idx[at] = i;
    }
}

// Offers the candidates of the 3^4 cells around i's cell to the warp, up to 32 at a time: each
// lane calls f(at, on) with the place of its candidate in the runs (on: it has one); f returns
// the same value in every lane, false to stop.  All lanes call it together.  EACH: 32 cells after
// the other (the unions, whose points have neighbours); else a lane's three lookups go side by
// side, in FIRST where the first ones find nothing, and a point alone in all 81 cells costs no scan:
// the function returns false then, without calling f, and the later passes leave the point out.
// The lookups are chains of dependent loads, which only more warps hide: the kernels are held to 32
// registers (8 CTAs per SM).  1e6 candidates far apart: 5.1 -> 1.8 ms, with 40 registers 2.7.
enum Lookup { EACH, FIRST, ALL };
template <Lookup HOW, class F>
__device__ __forceinline__ bool for_neighbours(const ClusterArgs &a, int i, int lane, F f) {
    const int4 c = a.cells[i];
    auto lookup = [&](int d, int &count, int &start) {
        count = 0;
        start = 0;
        if (d < 81) {
            const int s = find_cell(a, make_int4(c.x + d % 3 - 1, c.y + (d / 3) % 3 - 1, c.z + (d / 9) % 3 - 1, c.w + d / 27 - 1));
            if (s >= 0) {
                count = a.cnt[s];
                start = a.start[s];
            }
        }
    };
    auto offer = [&](int count, int start) {   // false: f stopped
        int end = count;                       // candidates of the cells up to this lane's
#pragma unroll
        for (int o = 1; o < 32; o *= 2) {
            const int e = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += e;
        }
        const int total = __shfl_sync(0xffffffffu, end, 31);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            int cell = 0;   // the first lane whose end is above t
#pragma unroll
            for (int o = 16; o >= 1; o /= 2)
                if (__shfl_sync(0xffffffffu, end, cell + o - 1) <= t) cell += o;
            cell = min(cell, 31);
            const int first = __shfl_sync(0xffffffffu, end - count, cell), place = __shfl_sync(0xffffffffu, start, cell);
            if (!f(place + t - first, t < total)) return false;
        }
        return true;
    };
    if constexpr (HOW == EACH) {
        for (int d0 = 0; d0 < 81; d0 += 32) {
            int count, start;
            lookup(d0 + lane, count, start);
            if (!offer(count, start)) return true;
        }
        return true;
    }
    int c0, s0, c1 = 0, s1 = 0, c2 = 0, s2 = 0;
    lookup(lane, c0, s0);
    const bool side = HOW == ALL || __reduce_add_sync(0xffffffffu, c0) == 0;
    if (side) {
        lookup(32 + lane, c1, s1);
        lookup(64 + lane, c2, s2);
        if (__reduce_add_sync(0xffffffffu, c0 + c1 + c2) <= 1) return false;
    }
    if (!offer(c0, s0)) return true;
    if (!side) lookup(32 + lane, c1, s1);
    if (!offer(c1, s1)) return true;
    if (!side) lookup(64 + lane, c2, s2);
    offer(c2, s2);
    return true;
}

__global__ void __launch_bounds__(kThreads, 8) core_kernel(ClusterArgs a) {
    const int lane = threadIdx.x & 31, warps = gridDim.x * (blockDim.x / 32);
    for (int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; i < a.n; i += warps) {
        const bool ok = a.valid[i] != 0;
        int cnt = 0;
        if (ok) {
            const int4 p = point_of(a.cand[i]);
            const bool near = for_neighbours<FIRST>(a, i, lane, [&](int at, bool on) {
                cnt += __popc(__ballot_sync(0xffffffffu, on && within(a, p, a.run_pts[at])));
                return cnt < a.min_samples;
            });
            if (!near) {   // its own neighbour, and nobody's else: the later passes leave it alone
                cnt = 1;
                if (lane == 0) a.valid[i] = kAlone;
            }
        }
        if (lane == 0) {
            a.core[i] = (ok && cnt >= a.min_samples) ? 1 : 0;
            a.bestnu[i] = 0ull;
        }
    }
}

__global__ void __launch_bounds__(kThreads, 8) union_kernel(ClusterArgs a) {
    volatile int *parent = a.parent;
    const int lane = threadIdx.x & 31, warps = gridDim.x * (blockDim.x / 32);
    for (int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; i < a.n; i += warps) {
        if (!a.core[i] || a.valid[i] == kAlone) continue;
        const int4 p = point_of(a.cand[i]);
        for_neighbours<EACH>(a, i, lane, [&](int at, bool on) {
            const int j = on ? a.run_idx[at] : i;
            if (j < i && a.core[j]) {
                int u = find_root(parent, i, a.n, a.status), v = find_root(parent, j, a.n, a.status);
                if (u != v && within(a, p, a.run_pts[at])) {
                    for (int it = 0; it <= 2 * a.n + 2; ++it) {
                        u = find_root(parent, u, a.n, a.status);
                        v = find_root(parent, v, a.n, a.status);
                        if (u == v) break;
                        if (u < v) {
                            const int t = u;
                            u = v;
                            v = t;
                        }
                        // u > v: hook the larger root under the smaller
                        if (atomicCAS(&a.parent[u], u, v) == u) break;
                        if (it == 2 * a.n + 2) atomicExch(a.status, 2);
                    }
                }
            }
            __syncwarp();
            return true;
        });
    }
}

__global__ void __launch_bounds__(kThreads, 8) label_kernel(ClusterArgs a) {
    volatile int *parent = a.parent;
    const int lane = threadIdx.x & 31, warps = gridDim.x * (blockDim.x / 32);
    for (int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; i < a.n; i += warps) {
        int lab = -1;
        if (a.valid[i]) {
            int best = i;
            if (!a.core[i] && a.valid[i] != kAlone) {
                // the nearest core neighbour (smallest d2, then lowest index)
                const int4 p = point_of(a.cand[i]);
                int bj = 0x7fffffff;
                double bd = INFINITY;
                for_neighbours<ALL>(a, i, lane, [&](int at, bool on) {
                    const int j = on ? a.run_idx[at] : i;
                    if (on && a.core[j] && within(a, p, a.run_pts[at])) {
                        const double d2 = dist2(p, a.run_pts[at], a.w_pos, a.w_vel);
                        if (d2 < bd || (d2 == bd && j < bj)) {
                            bj = j;
                            bd = d2;
                        }
                    }
                    return true;
                });
#pragma unroll
                for (int o = 16; o > 0; o /= 2) {
                    const double od = __shfl_xor_sync(0xffffffffu, bd, o);
                    const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
                    if (od < bd || (od == bd && oj < bj)) {
                        bd = od;
                        bj = oj;
                    }
                }
                if (bj != 0x7fffffff) best = bj;
            }
            if (lane == 0) {
                lab = a.core[best] ? find_root(parent, best, a.n, a.status) : i;
                atomicMax(&a.bestnu[lab], nu_key(a.cand[i].nu));
            }
        }
        if (lane == 0) {
            a.label[i] = lab;
            if (a.core_out) a.core_out[i] = a.core[i];
        }
    }
}

__global__ void pick_kernel(ClusterArgs a) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        const int lab = a.label[i];
        if (lab >= 0 && nu_key(a.cand[i].nu) == a.bestnu[lab]) atomicMin(&a.bestidx[lab], i);
    }
}

__global__ void keep_kernel(ClusterArgs a) {
    unsigned mine = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        const int lab = a.label[i];
        const bool k = lab >= 0 && a.bestidx[lab] == i;
        a.keep[i] = k ? 1 : 0;
        mine += k;
    }
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(a.count, mine);
}

}  // namespace

cudaError_t launch_cluster(const ClusterArgs &a, int sm_count, cudaStream_t st) {
    const int cap = 8 * (sm_count > 0 ? sm_count : 152);
    auto grid = [&](long long m) { return (int)std::max(1LL, std::min<long long>((m + kThreads - 1) / kThreads, cap)); };
    init_kernel<<<grid(std::max<long long>(a.T, a.n)), kThreads, 0, st>>>(a);
    if (a.n > 0) {
        prep_kernel<<<grid(a.n), kThreads, 0, st>>>(a);
        insert_kernel<<<grid(a.n), kThreads, 0, st>>>(a);
        place_kernel<<<grid(a.n), kThreads, 0, st>>>(a);
        gather_kernel<<<grid(a.n), kThreads, 0, st>>>(a);
        core_kernel<<<grid(32LL * a.n), kThreads, 0, st>>>(a);
        union_kernel<<<grid(32LL * a.n), kThreads, 0, st>>>(a);
        label_kernel<<<grid(32LL * a.n), kThreads, 0, st>>>(a);
        pick_kernel<<<grid(a.n), kThreads, 0, st>>>(a);
        keep_kernel<<<grid(a.n), kThreads, 0, st>>>(a);
    }
    return cudaGetLastError();
}

}  // namespace kb
