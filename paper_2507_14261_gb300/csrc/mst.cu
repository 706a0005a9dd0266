// MST extraction (the Kruskal step at the end of Algorithm 1), the FP64
// tree weight, and the gradient of the tree weight.
//
// Kruskal's algorithm on a graph whose edges are totally ordered returns
// the unique MST under that order; Boruvka's algorithm returns the same
// tree (cut property). The device runs edge-centric Boruvka rounds under
// the order (w, min id, max id):
//   1. every edge joining two components offers (w, min id) to both
//      components with a 64-bit atomicMin, then, among the edges that
//      matched the winner, the max id with a second atomicMin: together
//      the lexicographic minimum of the 96-bit key, found without sorting;
//   2. each component hooks to the component across its minimum edge;
//      two components that chose the same edge form the only possible
//      cycle and the smaller id stays root; the others record their edge;
//   3. pointer jumping makes every component point to its new root and the
//      vertices are relabelled.
// The edge set is the kNN graph (edge i -> nbr[i*k + r], weight
// dist[i*k + r]; both directions of a mutual pair are the same edge) plus
// the m inter-component edges. Tree edges are written in the order
// (round, component id), which is deterministic.
#include <cuda_runtime.h>

#include <cstring>

#include "famst_internal.cuh"

namespace famst {
namespace {

constexpr int JUMP_LIMIT = 1 << 22;

struct EdgeSrc {
    const int32_t *nbr;
    const float *dist;
    int k;
    int64_t nk;
    const int32_t *eu, *ev;
    const float *ew;
    int64_t m;
    const int64_t *m_dev;   // optional device-side count of E edges (<= m)
    __device__ __forceinline__ int64_t total() const {
        return nk + (m_dev ? (*m_dev < m ? *m_dev : m) : m);
    }
    __device__ __forceinline__ void get(int64_t e, int &a, int &b, float &w) const {
        if (e < nk) {
            // (a 64-bit division takes several times the 32-bit one)
            a = e >> 32 ? int(e / k) : int(uint32_t(e) / uint32_t(k));
            b = nbr[e];
            w = dist[e];
        } else {
            int64_t q = e - nk;
            a = eu[q];
            b = ev[q];
            w = ew[q];
        }
    }
};

__global__ void bv_init_kernel(int32_t *comp, int64_t n) {
    int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (v < n) comp[v] = int32_t(v);
}

// The smallest key of every component: in the late rounds, where few components
// remain, millions of edges would hit the same few addresses. The result is
// the same minimum whatever the order.
// A key that is not below the value seen is dropped (the value only falls, so
// a stale one drops less, never too much); the first two components among the
// others are reduced over the warp, the rest go out one by one. (A reduction
// per group of equal components, by match and masked reductions, ran once for
// every distinct component of the warp: 1.18 ms for the first round over 42M
// kNN edges, now 0.40.)
__device__ __forceinline__ void warp_min_to(unsigned long long *__restrict__ best, int c,
                                            unsigned long long key, int lane) {
    const bool pass = c >= 0 && key < __ldcg(best + c);
    unsigned todo = __ballot_sync(0xffffffffu, pass);
#pragma unroll 1
    for (int r = 0; r < 2 && todo; ++r) {
        const int lead = __ffs(todo) - 1;
        const int c0 = __shfl_sync(0xffffffffu, c, lead);
        const bool mine = pass && c == c0;
        const unsigned long long m = warp_min_u64(mine ? key : ~0ull);
        if (lane == lead) atomicMin(best + c0, m);
        todo &= ~__ballot_sync(0xffffffffu, mine);
    }
    if (todo >> lane & 1u) atomicMin(best + c, key);
}

constexpr int BV_U = 4;
__global__ void bv_min1_kernel(EdgeSrc es, const int32_t *__restrict__ comp,
                               unsigned long long *__restrict__ best1, const int *__restrict__ done,
                               int32_t *__restrict__ ou = nullptr, int32_t *__restrict__ ov = nullptr,
                               float *__restrict__ ow = nullptr,
                               unsigned long long *__restrict__ ocount = nullptr) {
    if (done && *done) return;
    const int64_t total = es.total();
    const int lane = threadIdx.x & 31;
    // whole warps step together (the warp-wide reductions need every lane), BV_U
    // edges per lane at a time: their loads are in flight together, and the
    // edges between components are appended with one atomic for all of them
    // (one per 32 edges queued up on the counter: 0.83 ms for the 32M edges of 1M
    // points, now 0.32; all rounds 2.5 -> 1.06, the second pass 0.76 -> 0.62)
    const int64_t stride = int64_t(gridDim.x) * blockDim.x * BV_U;
    for (int64_t e0 = (int64_t(blockIdx.x) * blockDim.x + (threadIdx.x & ~31)) * BV_U; e0 < total;
         e0 += stride) {
        int a[BV_U], b[BV_U], ca[BV_U], cb[BV_U];
        float w[BV_U];
#pragma unroll
        for (int i = 0; i < BV_U; ++i) {
            const int64_t e = e0 + 32 * i + lane;
            a[i] = b[i] = 0;
            w[i] = 0.0f;
            if (e < total) es.get(e, a[i], b[i], w[i]);
        }
#pragma unroll
        for (int i = 0; i < BV_U; ++i) {   // (beyond the end: 0, 0, not between components)
            ca[i] = comp[a[i]];
            cb[i] = comp[b[i]];
        }
        unsigned bal[BV_U];
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < BV_U; ++i) {
            const bool inter = ca[i] != cb[i];
            const unsigned long long key1 = (uint64_t(__float_as_uint(w[i])) << 32) |
                                            uint32_t(a[i] < b[i] ? a[i] : b[i]);
            warp_min_to(best1, inter ? ca[i] : -1, key1, lane);
            warp_min_to(best1, inter ? cb[i] : -1, key1, lane);
            bal[i] = __ballot_sync(0xffffffffu, inter);
            cnt += __popc(bal[i]);
        }
        if (ocount && cnt) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(ocount, (unsigned long long)cnt);
            base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
            for (int i = 0; i < BV_U; ++i) {
                if (bal[i] >> lane & 1u) {
                    const unsigned long long idx = base + __popc(bal[i] & ((1u << lane) - 1u));
                    ou[idx] = a[i];
                    ov[idx] = b[i];
                    ow[idx] = w[i];
                }
                base += __popc(bal[i]);
            }
        }
    }
}

__global__ void bv_min2_kernel(EdgeSrc es, const int32_t *__restrict__ comp,
                               const unsigned long long *__restrict__ best1,
                               unsigned int *__restrict__ best2, const int *__restrict__ done) {
    if (done && *done) return;
    const int64_t total = es.total(), step = int64_t(gridDim.x) * blockDim.x;
    for (int64_t e0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e0 < total;
         e0 += BV_U * step) {
        int a[BV_U], b[BV_U], ca[BV_U], cb[BV_U];
        float w[BV_U];
#pragma unroll
        for (int i = 0; i < BV_U; ++i) {
            a[i] = b[i] = 0;
            w[i] = 0.0f;
            if (e0 + i * step < total) es.get(e0 + i * step, a[i], b[i], w[i]);
        }
#pragma unroll
        for (int i = 0; i < BV_U; ++i) {
            ca[i] = comp[a[i]];
            cb[i] = comp[b[i]];
        }
#pragma unroll
        for (int i = 0; i < BV_U; ++i) {
            if (ca[i] == cb[i]) continue;
            const unsigned long long key1 = (uint64_t(__float_as_uint(w[i])) << 32) |
                                            uint32_t(a[i] < b[i] ? a[i] : b[i]);
            const unsigned int mx = unsigned(a[i] < b[i] ? b[i] : a[i]);
            if (best1[ca[i]] == key1) atomicMin(best2 + ca[i], mx);
            if (best1[cb[i]] == key1) atomicMin(best2 + cb[i], mx);
        }
    }
}

// First round (every vertex its own component): a vertex's minimum incident
// edge under (w, min, max) is its first kNN entry -- the list is the exact
// top-k by (w, id), so no edge at v, kNN or inter-component, is lighter, and
// at equal w the smallest id comes first. No edge scan is needed.
__global__ void bv_first_kernel(const int32_t *__restrict__ nbr, const float *__restrict__ dist,
                                int k, int64_t n, unsigned long long *__restrict__ best1,
                                unsigned int *__restrict__ best2) {
    const int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int j = nbr[v * k];
    if (j < 0) {
        best1[v] = KEY_NONE;
        best2[v] = 0xffffffffu;
        return;
    }
    const int mn = int(v) < j ? int(v) : j, mx = int(v) < j ? j : int(v);
    best1[v] = (uint64_t(__float_as_uint(dist[v * k])) << 32) | uint32_t(mn);
    best2[v] = unsigned(mx);
}

__global__ void bv_hook_kernel(const int32_t *__restrict__ comp, int64_t n,
                               const unsigned long long *__restrict__ best1,
                               const unsigned int *__restrict__ best2, int32_t *__restrict__ newp,
                               int32_t *__restrict__ flag, int32_t *__restrict__ rmn,
                               int32_t *__restrict__ rmx, float *__restrict__ rw) {
    int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c >= n) return;
    flag[c] = 0;
    if (comp[c] != c) return;  // not a component root
    unsigned long long b1 = best1[c];
    if (b1 == KEY_NONE) {
        newp[c] = int32_t(c);
        return;
    }
    int mn = int(uint32_t(b1));
    int mx = int(best2[c]);
    int cm = comp[mn], cx = comp[mx];
    int other = cm == int(c) ? cx : cm;
    bool mutual = best1[other] == b1 && best2[other] == unsigned(mx);
    if (mutual && c < other) {
        newp[c] = int32_t(c);
        return;
    }
    newp[c] = other;
    flag[c] = 1;
    rmn[c] = mn;
    rmx[c] = mx;
    rw[c] = __uint_as_float(uint32_t(b1 >> 32));
}

__global__ void bv_jump_kernel(const int32_t *__restrict__ comp, int64_t n, int32_t *newp_,
                               int limit, int *dstatus) {
    int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c >= n || comp[c] != c) return;
    volatile int32_t *newp = newp_;
    int guard = 0;
    while (guard++ < limit) {
        int p = newp[c];
        int g = newp[p];
        if (g == p) return;
        newp[c] = g;
    }
    set_status(dstatus, STATUS_LOOP_LIMIT);
}

__global__ void bv_relabel_kernel(int32_t *__restrict__ comp, int64_t n,
                                  const int32_t *__restrict__ newp) {
    int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (v < n) comp[v] = newp[comp[v]];
}

__global__ void bv_record_kernel(const int32_t *__restrict__ flag,
                                 const int32_t *__restrict__ pos, int64_t n, int64_t base,
                                 const int32_t *__restrict__ rmn, const int32_t *__restrict__ rmx,
                                 const float *__restrict__ rw, int32_t *__restrict__ tu,
                                 int32_t *__restrict__ tv, float *__restrict__ tw) {
    int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c >= n || !flag[c]) return;
    int64_t o = base + pos[c];
    if (o >= n - 1) return;  // a spanning tree has n-1 edges; never write past them
    tu[o] = rmn[c];
    tv[o] = rmx[c];
    tw[o] = rw[c];
}

// ------------------------------------------------------- FP64 weights

constexpr int WR_NT = 256;
constexpr int WR_IPT = 8;
constexpr int WR_TILE = WR_NT * WR_IPT;

// fixed-order block reduction of two double values per thread
__device__ void block_sum2(double &a, double &b) {
    __shared__ double sa[WR_NT], sb[WR_NT];
    sa[threadIdx.x] = a;
    sb[threadIdx.x] = b;
    __syncthreads();
    for (int s = WR_NT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sa[threadIdx.x] += sa[threadIdx.x + s];
            sb[threadIdx.x] += sb[threadIdx.x + s];
        }
        __syncthreads();
    }
    a = sa[0];
    b = sb[0];
}

// The FP64 value of a float without the conversion unit: the FP64 pipe (two
// lanes an SM here) bounds the lengths below, and conversions go through it.
// Normal numbers only need their exponent rebased and their fields moved;
// zeros and subnormals (exponent 0), infinities and NaN (255) take the
// instruction (both ends are at or above 0x7f000000 after the subtraction).
__device__ __forceinline__ double widen(float f) {
    const uint32_t b = __float_as_uint(f), e = b & 0x7f800000u;
    if (e - 0x00800000u >= 0x7f000000u) return double(f);
    return __hiloint2double(int((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)),
                            int(b << 29));
}

// FP64 length of every edge: p = fma(x_t - y_t, x_t - y_t, p) over t = 0 ..
// d - 1. One thread per edge. (The sums over edges are a separate pass, so
// that a small tree still fills the chip: 2k x 16, 47 us in one block.)
template <int VEC>
__global__ void edge_len64_kernel(const float *__restrict__ X, int d,
                                  const int32_t *__restrict__ tu, const int32_t *__restrict__ tv,
                                  int64_t m, double *__restrict__ len) {
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= m) return;
    const float *a = X + int64_t(tu[e]) * d, *b = X + int64_t(tv[e]) * d;
    double p = 0.0;
    if constexpr (VEC == 4) {
        const float4 *a4 = reinterpret_cast<const float4 *>(a);
        const float4 *b4 = reinterpret_cast<const float4 *>(b);
#pragma unroll 2
        for (int q = 0; q < d / 4; ++q) {
            const float4 x = __ldg(a4 + q), y = __ldg(b4 + q);
            const double d0 = widen(x.x) - widen(y.x), d1 = widen(x.y) - widen(y.y);
            const double d2 = widen(x.z) - widen(y.z), d3 = widen(x.w) - widen(y.w);
            p = fma(d0, d0, p);
            p = fma(d1, d1, p);
            p = fma(d2, d2, p);
            p = fma(d3, d3, p);
        }
    } else {
        for (int t = 0; t < d; ++t) {
            const double dl = widen(a[t]) - widen(b[t]);
            p = fma(dl, dl, p);
        }
    }
    len[e] = sqrt(p);
}

__global__ void weight_partial_kernel(const float *__restrict__ tw, const double *__restrict__ len,
                                      int64_t m, double *__restrict__ part) {
    int64_t base = int64_t(blockIdx.x) * WR_TILE + int64_t(threadIdx.x) * WR_IPT;
    double s32 = 0.0, s64 = 0.0;
    for (int r = 0; r < WR_IPT; ++r) {
        int64_t e = base + r;
        if (e >= m) break;
        s32 += double(tw[e]);
        if (len) s64 += len[e];
    }
    block_sum2(s32, s64);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = s32;
        part[2 * blockIdx.x + 1] = s64;
    }
}

__global__ void weight_final_kernel(const double *__restrict__ part, int64_t nb,
                                    double *__restrict__ W) {
    double s32 = 0.0, s64 = 0.0;
    for (int64_t b = threadIdx.x; b < nb; b += WR_NT) {
        s32 += part[2 * b];
        s64 += part[2 * b + 1];
    }
    block_sum2(s32, s64);
    if (threadIdx.x == 0) {
        W[0] = s32;
        W[1] = s64;
    }
}

// ----------------------------------------------------------- backward
//
// Bound: HBM and the latency of its dependent loads. Every vertex's row is
// read once for itself and once per incident edge (about 3 n d floats for a
// tree, 1.5 GB at 1M x 128) and the gradient is written once. A warp owns a
// vertex: its row stays in registers, lane l holding the coordinates l,
// l + 32, ... of both rows, which are the canonical distance's own partials,
// so the edge's length comes out of the loads the gradient needs anyway; no
// pass over the edges computes or stores lengths, and the finiteness check
// rides along. The incidences are placed by counting and ranked inside their
// vertex (ascending edge index) instead of radix sorted, where that is cheap.
//
// A rank reads its vertex's whole list: the reads of all ranks are the sum of the
// squared degrees, and the longest list is one thread's chain. The radix sort's
// cost does not depend on the degrees. Trees of hubs with h leaves each, whole
// call, ranks / radix sort, us: 1M x 16 h = 4 313 / 452, 90 466 / 484, 128 527 /
// 499, 500 1133 / 631, 2000 3577 / 1316; 100,000 x 64 h = 4 118 / 209, 256 306 /
// 363, 500 494 / 507, 1000 575 / 520; 10,000 x 16 h = 500 267 / 313, 2000 840 / 833.
constexpr int INC_RANK_MAX = 2048;   // about 20 us for a single such list
inline bool rank_pays(int64_t m, uint64_t sum_sq, int64_t max_deg) {
    return max_deg <= INC_RANK_MAX && sum_sq <= uint64_t(40000000 + 70 * m);
}

// What incidence_count_kernel leaves behind the degrees.
struct IncTotals {
    unsigned long long sum_sq;   // of the degrees (those beyond INC_RANK_MAX count less)
    int32_t max_deg;
};
inline int64_t totals_at(int64_t n) { return (n + 2) / 2 * 2; }   // 8-byte aligned, behind n + 1 degrees
constexpr int64_t TOTALS_WORDS = 4;

// Range check, degrees and each incidence's arrival number at its vertex; the
// a-th arrival adds 2 a + 1 to the sum of squares.
__global__ void incidence_count_kernel(const int32_t *__restrict__ tu,
                                       const int32_t *__restrict__ tv, int64_t m, int64_t n,
                                       int32_t *__restrict__ deg, int2 *__restrict__ slot,
                                       IncTotals *__restrict__ totals, int *dstatus) {
    __shared__ int bmax;
    __shared__ unsigned bsum;   // 512 arrivals of at most 2^20
    if (threadIdx.x == 0) {
        bmax = 0;
        bsum = 0;
    }
    __syncthreads();
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    int mx = 0;
    unsigned sum = 0;
    if (e < m) {
        const int u = tu[e], v = tv[e];
        if (u < 0 || v < 0 || int64_t(u) >= n || int64_t(v) >= n) {
            set_status(dstatus, STATUS_BAD_ID);
        } else {
            const int su = atomicAdd(&deg[u], 1), sv = atomicAdd(&deg[v], 1);
            slot[e] = make_int2(su, sv);
            mx = (su > sv ? su : sv) + 1;
            sum = min(2u * unsigned(su) + 1u, 1u << 20) + min(2u * unsigned(sv) + 1u, 1u << 20);
        }
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&bmax, mx);
        atomicAdd(&bsum, sum);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&totals->max_deg, bmax);
        atomicAdd(&totals->sum_sq, (unsigned long long)bsum);
    }
}

__global__ void incidence_fill_kernel(const int32_t *__restrict__ tu,
                                      const int32_t *__restrict__ tv, int64_t m,
                                      const int32_t *__restrict__ off,
                                      const int2 *__restrict__ slot, int32_t *__restrict__ inc) {
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= m) return;
    const int2 s = slot[e];
    inc[off[tu[e]] + s.x] = int(2 * e);
    inc[off[tv[e]] + s.y] = int(2 * e + 1);
}

// adj: per vertex, its edges' other ends in ascending edge index
__global__ void incidence_rank_kernel(const int32_t *__restrict__ tu,
                                      const int32_t *__restrict__ tv, int64_t m,
                                      const int32_t *__restrict__ off,
                                      const int32_t *__restrict__ inc, int32_t *__restrict__ adj) {
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= m) return;
    const int u = tu[e], v = tv[e];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int a = side ? v : u, code = int(2 * e) + side;
        const int j0 = off[a], j1 = off[a + 1];
        int r = 0;
        for (int j = j0; j < j1; ++j) r += __ldg(inc + j) < code;
        adj[j0 + r] = side ? u : v;
    }
}

// The radix sort's input (large degrees) and its adj entries.
__global__ void incidence_kernel(const int32_t *__restrict__ tu, const int32_t *__restrict__ tv,
                                 int64_t m, uint32_t *__restrict__ keys,
                                 int32_t *__restrict__ vals) {
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= m) return;
    keys[2 * e] = uint32_t(tu[e]);
    vals[2 * e] = int32_t(2 * e);
    keys[2 * e + 1] = uint32_t(tv[e]);
    vals[2 * e + 1] = int32_t(2 * e + 1);
}

__global__ void incidence_adj_kernel(const int32_t *__restrict__ tu,
                                     const int32_t *__restrict__ tv, int64_t m2,
                                     const int32_t *__restrict__ inc, int32_t *__restrict__ adj) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= m2) return;
    const int code = inc[i];
    adj[i] = (code & 1) ? tu[code >> 1] : tv[code >> 1];
}

// gX[v][t] = gW * sum over v's edges, ascending edge index, of
// (x_v[t] - x_other[t]) / w_e  (w_e = 0 contributes 0).
// Narrow rows (d <= 16): G lanes per vertex, G the power of two that holds d
// (the canonical butterfly's wider steps would add zeros).
template <int G>
__global__ void grad_narrow_kernel(const float *__restrict__ X, int64_t n, int d,
                                   const int32_t *__restrict__ off,
                                   const int32_t *__restrict__ adj, float gW,
                                   float *__restrict__ gX, int *dstatus) {
    const int64_t v = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) / G;
    if (v >= n) return;   // whole groups
    const int lane = threadIdx.x & 31, g = lane % G;
    const unsigned gmask = ((1u << G) - 1u) << (lane - g);
    const float x = g < d ? X[v * d + g] : 0.0f;
    if (!isfinite(x)) set_status(dstatus, STATUS_NONFINITE);
    float acc = 0.0f;
    const int j1 = off[v + 1];
    for (int j = off[v]; j < j1; ++j) {
        const float y = g < d ? __ldg(X + int64_t(adj[j]) * d + g) : 0.0f;
        const float dl = __fsub_rn(x, y);
        float p = __fmaf_rn(dl, dl, 0.0f);
#pragma unroll
        for (int o = G / 2; o >= 1; o >>= 1) p = __fadd_rn(p, __shfl_xor_sync(gmask, p, o));
        const float w = __fsqrt_rn(p);
        if (w > 0.0f) acc = __fadd_rn(acc, __fdiv_rn(dl, w));
    }
    if (g < d) gX[v * d + g] = __fmul_rn(gW, acc);
}

// A warp takes GRAD_V consecutive vertices: their offsets and the ends of
// their edges come with one load each, and while a vertex is summed the next
// one's row and its first two neighbours' rows are on their way (a tree
// vertex has two edges on average), so a warp waits for the chain offset ->
// edge end -> row once per GRAD_V vertices instead of once per vertex.
// A lane holds XR coordinates; rows wider than 32 XR (WIDE) take the
// coordinates in chunks of 32 XR and evaluate each edge's length again per
// chunk.
constexpr int GRAD_V = 8;
template <int XR, bool WIDE>
__global__ void __launch_bounds__(256) grad_rows_kernel(const float *__restrict__ X, int64_t n, int d,
                                 const int32_t *__restrict__ off, const int32_t *__restrict__ adj,
                                 float gW, float *__restrict__ gX, int *dstatus) {
    const int64_t vb = ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * GRAD_V;
    if (vb >= n) return;
    const int lane = threadIdx.x & 31;
    const int nv = n - vb < GRAD_V ? int(n - vb) : GRAD_V;
    const int o = off[vb + (lane < nv ? lane : nv)];
    const int base = __shfl_sync(0xffffffffu, o, 0), last = __shfl_sync(0xffffffffu, o, nv);
    const int aj = base + lane < last ? adj[base + lane] : 0;
    auto end_of = [&](int j) {   // the other end of entry j (warp-uniform)
        const int a = __shfl_sync(0xffffffffu, aj, (j - base) & 31);
        return j - base < 32 ? a : __ldg(adj + j);
    };
    bool bad = false;
    for (int c0 = 0; c0 < d; c0 += 32 * XR) {
        float xn[XR], yn[2][XR];
        const float *yp[2] = {X, X};
        auto row = [&](const float *r, float(&f)[XR]) {
#pragma unroll
            for (int q = 0; q < XR; ++q) {
                const int t = c0 + lane + 32 * q;
                f[q] = t < d ? __ldg(r + t) : 0.0f;
            }
        };
        auto fetch = [&](int i) {   // vertex vb + i and its first two neighbours
            const int j0 = __shfl_sync(0xffffffffu, o, i), j1 = __shfl_sync(0xffffffffu, o, i + 1);
            row(X + (vb + i) * d, xn);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (j0 + e < j1) {
                    yp[e] = X + int64_t(end_of(j0 + e)) * d;
                    row(yp[e], yn[e]);
                }
            }
        };
        fetch(0);
        for (int i = 0; i < nv; ++i) {
            const int j0 = __shfl_sync(0xffffffffu, o, i), j1 = __shfl_sync(0xffffffffu, o, i + 1);
            float xs[XR], acc[XR], y[2][XR];
            const float *yc[2] = {yp[0], yp[1]};
            const float *xr = X + (vb + i) * d;
#pragma unroll
            for (int q = 0; q < XR; ++q) {
                xs[q] = xn[q];
                y[0][q] = yn[0][q];
                y[1][q] = yn[1][q];
                acc[q] = 0.0f;
                bad |= !isfinite(xs[q]);
            }
            if (i + 1 < nv) fetch(i + 1);
            auto add = [&](const float *yr, const float(&yv)[XR]) {
                float p = 0.0f;
                if constexpr (WIDE) {
                    for (int t = lane; t < d; t += 32) {
                        const float dl = __fsub_rn(__ldg(xr + t), __ldg(yr + t));
                        p = __fmaf_rn(dl, dl, p);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < XR; ++q) {
                        const float dl = __fsub_rn(xs[q], yv[q]);
                        p = __fmaf_rn(dl, dl, p);
                    }
                }
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) p = __fadd_rn(p, __shfl_xor_sync(0xffffffffu, p, s));
                const float w = __fsqrt_rn(p);
                if (w > 0.0f) {
#pragma unroll
                    for (int q = 0; q < XR; ++q)
                        acc[q] = __fadd_rn(acc[q], __fdiv_rn(__fsub_rn(xs[q], yv[q]), w));
                }
            };
            if (j0 < j1) add(yc[0], y[0]);
            if (j0 + 1 < j1) add(yc[1], y[1]);
            // (the other edges two at a time, both rows in flight: a hub of 1000
            // edges of 64 coordinates 0.4 -> 0.3 us an edge; not with one coordinate
            // per lane, where it takes 39 registers instead of 32)
            if constexpr (XR > 1) {
#pragma unroll 1
                for (int j = j0 + 2; j < j1; j += 2) {
                    const float *yr[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        yr[e] = X + int64_t(end_of(j + e < j1 ? j + e : j)) * d;
                        row(yr[e], y[e]);
                    }
                    add(yr[0], y[0]);
                    if (j + 1 < j1) add(yr[1], y[1]);
                }
            } else {
                for (int j = j0 + 2; j < j1; ++j) {
                    const float *yr = X + int64_t(end_of(j)) * d;
                    row(yr, y[0]);
                    add(yr, y[0]);
                }
            }
#pragma unroll
            for (int q = 0; q < XR; ++q) {
                const int t = c0 + lane + 32 * q;
                if (t < d) gX[(vb + i) * d + t] = __fmul_rn(gW, acc[q]);
            }
        }
    }
    if (bad) set_status(dstatus, STATUS_NONFINITE);
}

// Record the round's tree edges at base + pos (base and the round's count
// live on the device), then advance base and raise `done` when a round
// added no edge: the later rounds of a fixed budget become no-ops.
__global__ void bv_record_dev_kernel(const int32_t *__restrict__ flag,
                                     const int32_t *__restrict__ pos, int64_t n,
                                     const long long *__restrict__ base,
                                     const int32_t *__restrict__ rmn, const int32_t *__restrict__ rmx,
                                     const float *__restrict__ rw, int32_t *__restrict__ tu,
                                     int32_t *__restrict__ tv, float *__restrict__ tw,
                                     int64_t cap, const int *__restrict__ done) {
    if (*done) return;
    int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c >= n || !flag[c]) return;
    int64_t o = *base + pos[c];
    if (o >= cap) return;
    tu[o] = rmn[c];
    tv[o] = rmx[c];
    tw[o] = rw[c];
}

__global__ void bv_advance_kernel(long long *base, const int32_t *__restrict__ added, int *done,
                                  int *rounds) {
    if (*done) return;
    if (*added == 0) {
        *done = 1;
    } else {
        *base += *added;
        *rounds += 1;
    }
}

__global__ void bv_gate_kernel(const int *__restrict__ done, int32_t *__restrict__ flag, int64_t n) {
    // a finished forest records nothing more
    if (!*done) return;
    int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c < n) flag[c] = 0;
}

inline unsigned blocks_for(int64_t count, int th) { return unsigned((count + th - 1) / th); }

}  // namespace

size_t boruvka_workspace(int64_t n, int64_t ecap) {
    size_t b = align256(size_t(n) * 8) + align256(size_t(n) * 4) * 8 + scan_workspace(n) + 256;
    if (ecap > 0) b += align256(size_t(ecap) * 4) * 6 + 256;
    return b;
}

// Boruvka with no host synchronisation: a fixed budget of rounds, the
// edge count of E and the termination live on the device (for CUDA-graph
// capture). Finds the minimum spanning forest of the candidate graph.
famst_status boruvka_dev(const Exec &ex, Arena &ar, int64_t n, const int32_t *nbr,
                         const float *dist, int k, const int32_t *eu, const int32_t *ev,
                         const float *ew, int64_t m_cap, const int64_t *m_dev, MstOut out,
                         int64_t out_cap, int max_rounds, long long *edges_dev, int *rounds_dev) {
    if (n <= 1) return FAMST_OK;
    unsigned long long *best1 = ar.take<unsigned long long>(size_t(n));
    unsigned int *best2 = ar.take<unsigned int>(size_t(n));
    int32_t *comp = ar.take<int32_t>(size_t(n));
    int32_t *newp = ar.take<int32_t>(size_t(n));
    int32_t *flag = ar.take<int32_t>(size_t(n));
    int32_t *pos = ar.take<int32_t>(size_t(n));
    int32_t *rmn = ar.take<int32_t>(size_t(n));
    int32_t *rmx = ar.take<int32_t>(size_t(n));
    float *rw = ar.take<float>(size_t(n));
    int32_t *added = ar.take<int32_t>(1);
    int *done = ar.take<int>(1);
    if (!best1 || !best2 || !comp || !newp || !flag || !pos || !rmn || !rmx || !rw || !added ||
        !done)
        return FAMST_ERR_OOM;
    EdgeSrc es{nbr, dist, k, n * int64_t(k), eu, ev, ew, m_cap, m_dev};
    const int th = 256;
    int64_t nedges = es.nk + m_cap;
    unsigned egrid = blocks_for(nedges, th);
    unsigned ecap = unsigned(ex.num_sms) * 32;
    if (egrid > ecap) egrid = ecap;
    if (egrid == 0) egrid = 1;
    if (cudaMemsetAsync(done, 0, sizeof(int), ex.stream) != cudaSuccess ||
        cudaMemsetAsync(edges_dev, 0, sizeof(long long), ex.stream) != cudaSuccess ||
        cudaMemsetAsync(rounds_dev, 0, sizeof(int), ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    FAMST_LAUNCH(ex, bv_init_kernel, blocks_for(n, th), th, 0, comp, n);
    for (int r = 0; r < max_rounds; ++r) {
        if (cudaMemsetAsync(best1, 0xff, size_t(n) * 8, ex.stream) != cudaSuccess ||
            cudaMemsetAsync(best2, 0xff, size_t(n) * 4, ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
        FAMST_LAUNCH(ex, bv_min1_kernel, egrid, th, 0, es, comp, best1, done);
        FAMST_LAUNCH(ex, bv_min2_kernel, egrid, th, 0, es, comp, best1, best2, done);
        FAMST_LAUNCH(ex, bv_hook_kernel, blocks_for(n, th), th, 0, comp, n, best1, best2, newp,
                     flag, rmn, rmx, rw);
        FAMST_LAUNCH(ex, bv_gate_kernel, blocks_for(n, th), th, 0, done, flag, n);
        FAMST_LAUNCH(ex, bv_jump_kernel, blocks_for(n, th), th, 0, comp, n, newp,
                     ex.loop_limit > 0 ? ex.loop_limit : JUMP_LIMIT, ex.dstatus);
        FAMST_LAUNCH(ex, bv_relabel_kernel, blocks_for(n, th), th, 0, comp, n, newp);
        size_t mark = ar.off;
        famst_status st = exclusive_scan_i32(ex, ar, flag, pos, n, added);
        ar.off = mark;
        if (st != FAMST_OK) return st;
        FAMST_LAUNCH(ex, bv_record_dev_kernel, blocks_for(n, th), th, 0, flag, pos, n, edges_dev,
                     rmn, rmx, rw, out.tu, out.tv, out.tw, out_cap, done);
        FAMST_LAUNCH(ex, bv_advance_kernel, 1, 1, 0, edges_dev, added, done, rounds_dev);
    }
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

famst_status bv_state_init(const Exec &ex, Arena &ar, int64_t n, BvState *S, int64_t ecap) {
    S->n = n;
    if (ecap > 0) {
        S->ecap = ecap;
        for (int i = 0; i < 2; ++i) {
            S->cu[i] = ar.take<int32_t>(size_t(ecap));
            S->cv[i] = ar.take<int32_t>(size_t(ecap));
            S->cw[i] = ar.take<float>(size_t(ecap));
            if (!S->cu[i] || !S->cv[i] || !S->cw[i]) return FAMST_ERR_OOM;
        }
        S->ccount = ar.take<unsigned long long>(2);
        if (!S->ccount) return FAMST_ERR_OOM;
    }
    S->best1 = ar.take<unsigned long long>(size_t(n));
    S->best2 = ar.take<unsigned int>(size_t(n));
    S->comp = ar.take<int32_t>(size_t(n));
    S->newp = ar.take<int32_t>(size_t(n));
    S->flag = ar.take<int32_t>(size_t(n));
    S->pos = ar.take<int32_t>(size_t(n));
    S->rmn = ar.take<int32_t>(size_t(n));
    S->rmx = ar.take<int32_t>(size_t(n));
    S->rw = ar.take<float>(size_t(n));
    S->total = ar.take<int32_t>(1);
    if (!S->best1 || !S->best2 || !S->comp || !S->newp || !S->flag || !S->pos || !S->rmn ||
        !S->rmx || !S->rw || !S->total)
        return FAMST_ERR_OOM;
    FAMST_LAUNCH(ex, bv_init_kernel, blocks_for(n, 256), 256, 0, S->comp, n);
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

// One Boruvka round over the kNN-style edges (i -> nbr[i*k + r]) plus
// (eu, ev): every component's minimum outgoing edge under (w, min, max)
// is hooked and recorded at out[base ...]; *added_host (pinned) receives
// the number of edges added. Synchronises.
famst_status bv_round(const Exec &ex, Arena &ar, BvState &S, const int32_t *nbr, const float *dist,
                      int k, const int32_t *eu, const int32_t *ev, const float *ew, int64_t m,
                      MstOut out, int64_t base, int32_t *added_host) {
    const int64_t n = S.n;
    EdgeSrc es{nbr, dist, k, n * int64_t(k), eu, ev, ew, m, nullptr};
    if (S.cur >= 0)   // the previous scan's edges between components
        es = EdgeSrc{nullptr, nullptr, 1, 0, S.cu[S.cur], S.cv[S.cur], S.cw[S.cur], S.ecap,
                      reinterpret_cast<const int64_t *>(S.ccount + S.cur)};
    const int th = 256;
    int64_t nedges = es.nk + es.m;
    unsigned egrid = blocks_for(nedges, th);
    unsigned ecap = unsigned(ex.num_sms) * 32;
    if (egrid > ecap) egrid = ecap;
    if (egrid == 0) egrid = 1;
    if (S.round == 0 && S.knn_exact && k >= 1) {
        FAMST_LAUNCH(ex, bv_first_kernel, blocks_for(n, th), th, 0, nbr, dist, k, n, S.best1,
                     S.best2);
    } else {
        if (cudaMemsetAsync(S.best1, 0xff, size_t(n) * 8, ex.stream) != cudaSuccess ||
            cudaMemsetAsync(S.best2, 0xff, size_t(n) * 4, ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
        if (S.ecap > 0 && S.round >= 2) {   // early rounds keep most edges: no copy
            const int nxt = S.cur == 0 ? 1 : 0;
            if (cudaMemsetAsync(S.ccount + nxt, 0, 8, ex.stream) != cudaSuccess)
                return FAMST_ERR_CUDA;
            FAMST_LAUNCH(ex, bv_min1_kernel, egrid, th, 0, es, S.comp, S.best1, nullptr, S.cu[nxt],
                         S.cv[nxt], S.cw[nxt], S.ccount + nxt);
            FAMST_LAUNCH(ex, bv_min2_kernel, egrid, th, 0, es, S.comp, S.best1, S.best2, nullptr);
            S.cur = nxt;
        } else {
            FAMST_LAUNCH(ex, bv_min1_kernel, egrid, th, 0, es, S.comp, S.best1, nullptr, nullptr,
                         nullptr, nullptr, nullptr);
            FAMST_LAUNCH(ex, bv_min2_kernel, egrid, th, 0, es, S.comp, S.best1, S.best2, nullptr);
        }
    }
    ++S.round;
    FAMST_LAUNCH(ex, bv_hook_kernel, blocks_for(n, th), th, 0, S.comp, n, S.best1, S.best2, S.newp,
                 S.flag, S.rmn, S.rmx, S.rw);
    FAMST_LAUNCH(ex, bv_jump_kernel, blocks_for(n, th), th, 0, S.comp, n, S.newp,
                 ex.loop_limit > 0 ? ex.loop_limit : JUMP_LIMIT, ex.dstatus);
    FAMST_LAUNCH(ex, bv_relabel_kernel, blocks_for(n, th), th, 0, S.comp, n, S.newp);
    size_t mark = ar.off;  // the scan's scratch is reused by every round
    famst_status st = exclusive_scan_i32(ex, ar, S.flag, S.pos, n, S.total);
    ar.off = mark;
    if (st != FAMST_OK) return st;
    FAMST_LAUNCH(ex, bv_record_kernel, blocks_for(n, th), th, 0, S.flag, S.pos, n, base, S.rmn,
                 S.rmx, S.rw, out.tu, out.tv, out.tw);
    if (cudaMemcpyAsync(added_host, S.total, 4, cudaMemcpyDeviceToHost, ex.stream) != cudaSuccess ||
        cudaStreamSynchronize(ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

famst_status boruvka(const Exec &ex, Arena &ar, int64_t n, const int32_t *nbr, const float *dist,
                     int k, const int32_t *eu, const int32_t *ev, const float *ew, int64_t m,
                     MstOut out, int64_t *tree_edges, int *rounds, int32_t *pinned_host,
                     bool knn_exact, bool compact) {
    *tree_edges = 0;
    *rounds = 0;
    if (n <= 1) return FAMST_OK;
    BvState S;
    famst_status st = bv_state_init(ex, ar, n, &S, compact ? n * int64_t(k) + m : 0);
    if (st != FAMST_OK) return st;
    S.knn_exact = knn_exact;
    int64_t got = 0;
    // at least half the components disappear every round that adds edges:
    // 64 rounds cover any n; the context's loop limit can lower the budget
    const int budget = ex.loop_limit > 0 && ex.loop_limit < 64 ? ex.loop_limit : 64;
    int32_t added = 0;
    for (int r = 0; r < budget && got < n - 1; ++r) {
        st = bv_round(ex, ar, S, nbr, dist, k, eu, ev, ew, m, out, got, pinned_host);
        if (st != FAMST_OK) return st;
        *rounds = r + 1;
        added = *pinned_host;
        if (added == 0) break;
        got += added;
    }
    *tree_edges = got;
    // the budget ran out while rounds still added edges: not a disconnected graph
    if (got < n - 1 && added > 0) return FAMST_ERR_TIMEOUT;
    return FAMST_OK;
}

size_t tree_weight_workspace(int64_t m) {
    return align256(size_t((m + WR_TILE - 1) / WR_TILE + 1) * 16) + align256(size_t(m) * 8);
}

famst_status tree_weight(const Exec &ex, Arena &ar, const float *X, int d, bool vec4,
                         const int32_t *tu, const int32_t *tv, const float *tw, int64_t m,
                         double *W_dev) {
    int64_t nb = (m + WR_TILE - 1) / WR_TILE;
    if (nb == 0) nb = 1;
    double *part = ar.take<double>(size_t(nb) * 2);
    if (!part) return FAMST_ERR_OOM;
    double *len = nullptr;
    if (X && m > 0) {
        len = ar.take<double>(size_t(m));
        if (!len) return FAMST_ERR_OOM;
        if (vec4)
            FAMST_LAUNCH(ex, edge_len64_kernel<4>, blocks_for(m, 128), 128, 0, X, d, tu, tv, m, len);
        else
            FAMST_LAUNCH(ex, edge_len64_kernel<1>, blocks_for(m, 128), 128, 0, X, d, tu, tv, m, len);
    }
    FAMST_LAUNCH(ex, weight_partial_kernel, unsigned(nb), WR_NT, 0, tw, len, m, part);
    FAMST_LAUNCH(ex, weight_final_kernel, 1, WR_NT, 0, part, nb, W_dev);
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

size_t mst_backward_workspace(int64_t n, int64_t m) {
    return align256(size_t(m) * 8) + align256(size_t(2 * m) * 4) * 3 +
           align256(size_t(totals_at(n) + TOTALS_WORDS) * 4) + align256(size_t(n + 1) * 4) +
           radix_sort_workspace(2 * m) + scan_workspace(n + 1);
}

// pinned_host: four pinned host words (the totals, the status word). Ids are
// checked before they are used; synchronises once.
famst_status mst_backward(const Exec &ex, Arena &ar, const float *X, int64_t n, int d,
                          const int32_t *tu, const int32_t *tv, int64_t m, float gW, float *gX,
                          int32_t *pinned_host) {
    int2 *slot = ar.take<int2>(size_t(m > 0 ? m : 1));
    int32_t *inc = ar.take<int32_t>(size_t(m > 0 ? 2 * m : 1));
    int32_t *adj = ar.take<int32_t>(size_t(m > 0 ? 2 * m : 1));
    const int64_t tot = totals_at(n);
    int32_t *deg = ar.take<int32_t>(size_t(tot + TOTALS_WORDS));
    int32_t *off = ar.take<int32_t>(size_t(n + 1));
    if (!slot || !inc || !adj || !deg || !off) return FAMST_ERR_OOM;
    const int th = 256;
    IncTotals *totals = reinterpret_cast<IncTotals *>(deg + tot);
    if (cudaMemsetAsync(deg, 0, size_t(tot + TOTALS_WORDS) * 4, ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    if (m > 0)
        FAMST_LAUNCH(ex, incidence_count_kernel, blocks_for(m, th), th, 0, tu, tv, m, n, deg, slot,
                     totals, ex.dstatus);
    famst_status st = exclusive_scan_i32(ex, ar, deg, off, n + 1, nullptr);
    if (st != FAMST_OK) return st;
    if (m > 0) {
        IncTotals h;
        if (cudaMemcpyAsync(pinned_host, totals, 12, cudaMemcpyDeviceToHost, ex.stream) !=
                cudaSuccess ||
            cudaMemcpyAsync(pinned_host + 3, ex.dstatus, 4, cudaMemcpyDeviceToHost, ex.stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
        if (pinned_host[3] != 0) return FAMST_OK;   // an id out of range: the caller reads the status
        std::memcpy(&h, pinned_host, 12);
        if (rank_pays(m, h.sum_sq, h.max_deg)) {
            FAMST_LAUNCH(ex, incidence_fill_kernel, blocks_for(m, th), th, 0, tu, tv, m, off, slot,
                         inc);
            FAMST_LAUNCH(ex, incidence_rank_kernel, blocks_for(m, th), th, 0, tu, tv, m, off, inc,
                         adj);
        } else {
            uint32_t *keys = ar.take<uint32_t>(size_t(2 * m));
            if (!keys) return FAMST_ERR_OOM;
            FAMST_LAUNCH(ex, incidence_kernel, blocks_for(m, th), th, 0, tu, tv, m, keys, inc);
            int bits = 0;
            while ((int64_t(1) << bits) < n) ++bits;
            st = radix_sort_pairs(ex, ar, keys, inc, 2 * m, bits);
            if (st != FAMST_OK) return st;
            FAMST_LAUNCH(ex, incidence_adj_kernel, blocks_for(2 * m, th), th, 0, tu, tv, 2 * m, inc,
                         adj);
        }
    }
#define FAMST_GRADN(GV)                                                                         \
    FAMST_LAUNCH(ex, grad_narrow_kernel<GV>, blocks_for(n * GV, th), th, 0, X, n, d, off, adj, gW, \
                 gX, ex.dstatus)
#define FAMST_GRAD(XRV, WIDEV)                                                                  \
    FAMST_LAUNCH(ex, (grad_rows_kernel<XRV, WIDEV>),                                            \
                 blocks_for((n + GRAD_V - 1) / GRAD_V * 32, th), th, 0, X, n, d, off, adj, gW, gX, \
                 ex.dstatus)
    if (d <= 4) FAMST_GRADN(4);
    else if (d <= 8) FAMST_GRADN(8);
    else if (d <= 16) FAMST_GRADN(16);
    else if (d <= 32) FAMST_GRAD(1, false);
    else if (d <= 64) FAMST_GRAD(2, false);
    else if (d <= 128) FAMST_GRAD(4, false);
    else if (d <= 256) FAMST_GRAD(8, false);
    else FAMST_GRAD(8, true);
#undef FAMST_GRADN
#undef FAMST_GRAD
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

}  // namespace famst
