// The nearest-pair variant of Algorithm 3: for every component pair i < j,
// the lambda pairs (u in C_i, v in C_j) with the smallest canonical distance
// under the edge order (w, min id, max id) -- "the lambda nearest
// cross-component edges" -- instead of the lambda shortest of lambda^2
// random samples. A component pair with fewer than lambda cross pairs
// repeats its farthest pair in the remaining slots.
//
// The work is all cross pairs, |C_i| |C_j| per component pair (n^2 / 2 over
// all pairs when the components cover the points): a GEMM over the points
// sorted by component, whose output is nearly all discarded. Large clouds:
//  * the centred BF16 rows are gathered into component order; a work item is
//    128 rows of one component against a run of 256-row key tiles of the
//    later components, one CTA each: TMA stages the operand blocks, one
//    thread issues tcgen05.mma (128 x 256 FP32 accumulators in TMEM, two of
//    them), sixteen warps read the accumulators back;
//  * per (row, 16 columns) one threshold T on ||h_y||^2 - 2 h_x.h_y says
//    which pairs may reach the component pair's bound thr (T folds in the
//    row's norm, the rounding bounds of both rows and the accumulation
//    error), so a discarded pair costs an fma and a comparison;
//  * thr[i, j] starts as the lambda-th smallest canonical distance of up to
//    1024 distinct pairs and falls as the survivors' upper bounds enter the
//    component pair's lambda slots: at any time the slots hold upper bounds
//    of lambda distinct pairs, so no pair above their maximum is needed. The
//    first rows of every component go first, in a launch of their own: the
//    rest then meets bounds that a part of each component pair has set,
//    instead of all its CTAs passing the sample's bound at once. With many
//    component pairs that launch stores nothing and only lowers the bounds:
//    most survivors pass before them (nearest_plan.h);
//  * the survivors (a few hundred per component pair) are filtered with the
//    final thr, grouped by component pair, and decided on canonical FP32
//    distances by a warp per component pair.
// Bound: the key tiles' way from L2 (64 KB per 128 x 256 x 128 tile, 1.0 ms
// for 100k x 128 in 50 components without an epilogue) and the epilogue's
// latency (TMEM load, score, compare: 1.8 ms with it, 2.5 ms with the
// survivors; eight epilogue warps instead of sixteen: 3.2 ms). The whole call
// there: 33.1 ms with the warp kernel below, 3.1 ms; 1M x 128 points in 1000
// components, lambda 10: 2514 and 689 ms.
// Small clouds, many small components (nearest_plan.h), inputs with so many
// ties that the survivors overflow their buffer, and points whose squares leave
// the FP32 range take the warp kernel below:
//  * a work item is a block of 32 consecutive members of one component C_i;
//    its warp stages their BF16 rows in shared memory once and then streams
//    the members of every later component C_j (j > i), eight per step, as
//    the B columns of mma.sync m16n8k16;
//  * rigorous bounds on the canonical distance (staged_rows.cuh) rule pairs
//    out against the warp's current lambda-th best (before lambda pairs are
//    known: the lambda-th smallest upper bound of the step), survivors are
//    decided on canonical FP32 distances four at a time, and the warp keeps
//    a sorted top-lambda list of (w, min id, max id) keys, one entry per
//    lane, for each (item, C_j);
//  * a second kernel merges, per component pair, the lists of its C_i
//    blocks into the final lambda edges, written in Algorithm 3's layout.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "famst_internal.cuh"
#include "mbarrier.cuh"
#include "nearest_plan.h"
#include "staged_rows.cuh"
#include "tcgen05.cuh"

namespace famst {
namespace {

using namespace staged;

constexpr int NP_WARPS = 4;   // warps per block

template <int NKS>
struct NpStage : StageRows<NKS> {
    // per warp: the block's rows, their (eb, n2) and ids, the step's eight
    // (id, eb, n2) of the B columns
    static constexpr int WARP_BYTES = StageRows<NKS>::ROWS_BYTES + 32 * 8 + 32 * 4 + 8 * 16;
    static constexpr int SMEM = NP_WARPS * WARP_BYTES;
};

// (w, min id, max id) as two words: hi = w bits << 32 | min id, lo = max id
__device__ __forceinline__ bool pkey_less(uint64_t ah, uint32_t al, uint64_t bh, uint32_t bl) {
    return ah < bh || (ah == bh && al < bl);
}
__device__ __forceinline__ uint64_t pkey_hi(float w, int a, int b) {
    return (uint64_t(__float_as_uint(w)) << 32) | uint32_t(a < b ? a : b);
}

// Insert (kh, kl, u, v) into the warp's sorted list (lane r holds entry r,
// entries beyond `have` hold +inf keys); warp-uniform arguments.
__device__ __forceinline__ void list_insert(uint64_t &eh, uint32_t &el, int &eu, int &ev,
                                            uint64_t kh, uint32_t kl, int u, int v, int lambda,
                                            int &have, int lane) {
    const unsigned before = __ballot_sync(0xffffffffu, lane < have && pkey_less(eh, el, kh, kl));
    const int pos = __popc(before);
    if (pos >= lambda) return;
    const uint64_t ph = shfl_up_u64(eh, 1);
    const uint32_t pl = __shfl_up_sync(0xffffffffu, el, 1);
    const int pu = __shfl_up_sync(0xffffffffu, eu, 1);
    const int pv = __shfl_up_sync(0xffffffffu, ev, 1);
    if (lane > pos && lane < lambda) {
        eh = ph;
        el = pl;
        eu = pu;
        ev = pv;
    } else if (lane == pos) {
        eh = kh;
        el = kl;
        eu = u;
        ev = v;
    }
    if (have < lambda) ++have;
}

// Up to four canonical distances of pairs (ua[j], vb[j]) computed together
// and inserted into the list.
template <int XR>
__device__ __forceinline__ void pairs_batch(const float *__restrict__ X, int d, int nq,
                                            const int (&ua)[4], const int (&vb)[4],
                                            uint64_t &eh, uint32_t &el, int &eu, int &ev,
                                            int lambda, int &have, int lane) {
    if constexpr (XR > 0) {
        float xa[4][XR], xb[4][XR];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < XR; ++q) {
                const int t = lane + 32 * q;
                const bool ok = j < nq && t < d;
                xa[j][q] = ok ? __ldg(X + int64_t(ua[j]) * d + t) : 0.0f;
                xb[j][q] = ok ? __ldg(X + int64_t(vb[j]) * d + t) : 0.0f;
            }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= nq) break;
            float p = 0.0f;
#pragma unroll
            for (int q = 0; q < XR; ++q) {
                const float dl = __fsub_rn(xb[j][q], xa[j][q]);
                p = __fmaf_rn(dl, dl, p);
            }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) p = __fadd_rn(p, __shfl_xor_sync(0xffffffffu, p, o));
            const float w = __fsqrt_rn(p);
            const int a = ua[j], b = vb[j];
            list_insert(eh, el, eu, ev, pkey_hi(w, a, b), uint32_t(a < b ? b : a), a, b, lambda,
                        have, lane);
        }
    } else {
        for (int j = 0; j < nq; ++j) {
            const float w = canon_w<0>(X, d, ua[j], vb[j], lane);
            const int a = ua[j], b = vb[j];
            list_insert(eh, el, eu, ev, pkey_hi(w, a, b), uint32_t(a < b ? b : a), a, b, lambda,
                        have, lane);
        }
    }
}

// ------------------------------------------------ all pairs on tcgen05

constexpr int NT_M = 128;      // rows of an item (TMEM lanes)
constexpr int NT_N = 256;      // rows of a key tile (accumulator columns)
constexpr int NT_A = NT_M * TC_BK * 2, NT_B = NT_N * TC_BK * 2;
constexpr int NT_EPI = 16;     // epilogue warps, four per TMEM lane quarter
constexpr int NT_COLS = NT_N / (NT_EPI / 4);   // columns of one
constexpr int NT_QUEUE = 96;   // queued survivors per epilogue warp
constexpr int NT_FLUSH = 16;   // queued survivors at which a tile ends with a flush
constexpr int NT_THREADS = 64 + 32 * NT_EPI;
constexpr int NT_SAMPLES = 1024;
constexpr int NT_SW = 4;       // warps of a component pair's sample
constexpr unsigned long long NT_TOO_MANY = 1ull << 62;   // above any survivor buffer
constexpr unsigned long long NT_GAVE_UP = 1ull << 63;    // a wait ran out: pairs are missing

struct NtItem {
    int32_t row0, row_end;   // sorted rows row0 .. min(row0 + 127, row_end - 1), of component i
    int32_t i;
    int32_t kt0, kt1;        // key tiles
};

struct NtArgs {
    const NtItem *items;
    int nkb, stages;
    int64_t n, t;
    int lambda;
    const float *nyq;        // ||h||^2 (1 - aerr'), rounded down; +inf beyond n
    const float *n2, *eb;    // in component order
    const int32_t *colcomp;  // component of a sorted row (t beyond n)
    const int4 *chunk;       // per 16 sorted rows: first and last component, largest eb
    const int4 *hchunk;      // the same per NT_COLS
    unsigned *thr;           // per component pair: bound on its lambda-th distance (float bits)
    unsigned *slots;         // per component pair: lambda upper bounds (float bits)
    unsigned long long *count, cap;   // survivors found, room for them
    unsigned long long limit;         // with more the search has failed
    int32_t *su, *sv;        // survivors: sorted rows, lower bound
    float *sl;
    float aerr, eps;
    int *status;
};

// The rows of H in component order with their norms and error bounds, one
// warp per sorted row (npad rows: the last ones are padding).
__global__ void nt_gather_kernel(const __nv_bfloat16 *__restrict__ H, int ld,
                                 const float *__restrict__ heb, const float *__restrict__ hn2,
                                 const int32_t *__restrict__ members,
                                 const int32_t *__restrict__ comp_off, int64_t t, int64_t n,
                                 int64_t npad, float aerr, __nv_bfloat16 *__restrict__ Hs,
                                 float *__restrict__ n2, float *__restrict__ eb,
                                 float *__restrict__ nyq, int32_t *__restrict__ colcomp,
                                 unsigned long long *__restrict__ count) {
    const int64_t pos = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (pos >= npad) return;
    if (pos >= n) {
        if (lane == 0) {
            n2[pos] = eb[pos] = 0.0f;
            nyq[pos] = __int_as_float(0x7f800000);
            colcomp[pos] = int32_t(t);
        }
        return;
    }
    const int64_t r = members[pos];
    for (int c = lane; c < ld / 8; c += 32)
        reinterpret_cast<uint4 *>(Hs + pos * ld)[c] =
            __ldg(reinterpret_cast<const uint4 *>(H + r * ld) + c);
    if (lane == 0) {
        int64_t lo = 0, hi = t;   // comp_off[lo] <= pos < comp_off[hi]
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (comp_off[mid] <= pos) lo = mid; else hi = mid;
        }
        colcomp[pos] = int32_t(lo);
        const float v = hn2[r];
        // the thresholds' squares need room in the FP32 range: beyond it the
        // survivors count as too many, and the warp kernel takes the call
        if (!(v < 1e36f)) *count = NT_TOO_MANY;
        n2[pos] = v;
        eb[pos] = heb[r];
        nyq[pos] = __fmul_rd(v, 1.0f - (aerr + 0x1p-20f));
    }
}

__global__ void nt_chunk_kernel(const int32_t *__restrict__ colcomp, const float *__restrict__ eb,
                                int64_t n, int64_t nchunks, int len, int64_t t,
                                int4 *__restrict__ chunk) {
    const int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c >= nchunks) return;
    int4 v = make_int4(int(t), int(t), 0, 0);
    float m = 0.0f;
    if (len * c < n) {
        const int64_t last = len * c + len - 1 < n ? len * c + len - 1 : n - 1;
        v.x = colcomp[len * c];
        v.y = colcomp[last];
        for (int64_t q = len * c; q <= last; ++q) m = fmaxf(m, eb[q]);
    }
    v.z = __float_as_int(m);
    chunk[c] = v;
}

// thr = the lambda-th smallest canonical distance of up to NT_SAMPLES
// distinct cross pairs (sample s: member s mod |C_i| with member (s div |C_i|
// + s mod |C_i|) mod |C_j|), +inf when there are fewer than lambda pairs; the
// slots start at +inf. One block per component pair, its warps taking the
// samples in turn; no more samples than a 1024th of the pairs (but 64), so
// that small components do not pay more for the sample than for their tiles.
template <int XR>
__global__ void __launch_bounds__(NT_SW * 32)
nt_sample_kernel(const float *__restrict__ X, int d, const int32_t *__restrict__ members,
                 const int32_t *__restrict__ comp_off, int64_t t, int lambda,
                 unsigned *__restrict__ thr, unsigned *__restrict__ slots) {
    __shared__ unsigned best[NT_SW][32];
    const int64_t npairs = t * (t - 1) / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t p = blockIdx.x; p < npairs; p += gridDim.x) {
        int64_t i, j;
        pair_of(p, t, i, j);
        const int a0 = comp_off[i], b0 = comp_off[j];
        const unsigned A = unsigned(comp_off[i + 1] - a0), B = unsigned(comp_off[j + 1] - b0);
        const uint64_t N = uint64_t(A) * B;
        uint64_t want = N / 1024 < 64 ? 64 : N / 1024;
        want = want > NT_SAMPLES ? NT_SAMPLES : want;
        const unsigned r = unsigned(N < want ? N : want);
        uint64_t eh = ~0ull;
        uint32_t el = ~0u;
        int eu = -1, ev = -1, have = 0;
        for (unsigned s0 = 4 * warp; s0 < r; s0 += 4 * NT_SW) {
            int qa[4], qb[4];
#pragma unroll
            for (unsigned e = 0; e < 4; ++e) {
                const unsigned s = s0 + e < r ? s0 + e : s0;
                const unsigned a = s % A, b = (s / A + a) % B;
                qa[e] = members[a0 + a];
                qb[e] = members[b0 + b];
            }
            pairs_batch<XR>(X, d, int(min(4u, r - s0)), qa, qb, eh, el, eu, ev, lambda, have, lane);
        }
        best[warp][lane] = lane < have ? uint32_t(eh >> 32) : 0x7f800000u;
        __syncthreads();
        if (warp == 0) {   // the lambda-th of the warps' ascending lists
            unsigned v = 0x7f800000u;
            int head = 0;   // lane w < NT_SW walks list w
            for (int q = 0; q < lambda; ++q) {
                const unsigned mine =
                    lane < NT_SW && head < lambda ? best[lane][head] : 0x7f800000u;
                v = __reduce_min_sync(0xffffffffu, mine);
                const unsigned who = __ballot_sync(0xffffffffu, mine == v);
                if (lane == __ffs(who) - 1) ++head;
            }
            if (lane == 0) thr[p] = v;
            if (lane < lambda) slots[p * lambda + lane] = 0x7f800000u;
        }
        __syncthreads();
    }
}

// Enter the upper bound hi (float bits) of one more pair into its component
// pair's slots if it is below their maximum, and lower thr to the new maximum.
// A slot only ever falls, so a maximum of stale reads is a valid bound.
__device__ __forceinline__ void nt_slot_insert(unsigned *slots, unsigned *thr, int lambda,
                                               unsigned hi) {
    for (int tries = 0; tries < 64; ++tries) {
        unsigned m1 = 0, m2 = 0;   // largest, second largest
        int at = 0;
        for (int r = 0; r < lambda; ++r) {
            const unsigned v = __ldcg(slots + r);
            if (r == 0 || v > m1) {
                m2 = r == 0 ? 0u : m1;
                m1 = v;
                at = r;
            } else if (v > m2) {
                m2 = v;
            }
        }
        if (hi >= m1) return;
        if (atomicCAS(slots + at, m1, hi) == m1) {
            const unsigned m = m2 > hi ? m2 : hi;
            if (m < 0x7f800000u) atomicMin(thr, m);
            return;
        }
    }
}

// scores ny - 2 dot of two columns
__device__ __forceinline__ void nt_scores(uint32_t d0, uint32_t d1, unsigned long long ny, float &s0,
                                          float &s1) {
    unsigned long long d, r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(d0), "r"(d1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(d), "l"(f2_pack(-2.0f, -2.0f)), "l"(ny));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(s0), "=f"(s1) : "l"(r));
}

__global__ void __launch_bounds__(NT_THREADS, 1)
nearest_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  NtArgs args) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *sA = base;
    unsigned char *sB = sA + size_t(args.nkb) * NT_A;
    // per epilogue warp, its queue: dot product, sorted row of the key, lane
    float *qd = reinterpret_cast<float *>(sB + size_t(args.stages) * NT_B);
    int *qp = reinterpret_cast<int *>(qd + NT_EPI * NT_QUEUE);
    int *ql = qp + NT_EPI * NT_QUEUE;
    uint64_t *full = reinterpret_cast<uint64_t *>(ql + NT_EPI * NT_QUEUE);
    uint64_t *empty = full + args.stages;
    uint64_t *a_full = empty + args.stages;
    uint64_t *tfull = a_full + 1;     // [2]
    uint64_t *tempty = tfull + 2;     // [2]
    uint64_t *mma_done = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const NtItem I = args.items[blockIdx.x];
    const int ntiles = I.kt1 - I.kt0;
    if (threadIdx.x == 0)
        *abort_flag = *reinterpret_cast<volatile unsigned long long *>(args.count) > args.limit;
    __syncthreads();
    if (*abort_flag) return;
    if (threadIdx.x == 0) {
        for (int s = 0; s < args.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(a_full, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], NT_EPI);
        }
        mbar_init(mma_done, 1);
        mbar_init_fence();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp == 0) {
        if (lane == 0) {   // TMA producer: the rows once, then the key tiles
            mbar_expect_tx(a_full, uint32_t(args.nkb) * NT_A);
            for (int a = 0; a < args.nkb; ++a)
                tma_load_2d(sA + size_t(a) * NT_A, &tmA, a_full, a * TC_BK, I.row0);
            int it = 0;
            const int total = ntiles * args.nkb;
            for (; it < total; ++it) {
                const int s = it % args.stages, r = it / args.stages;
                if (!mbar_wait(&empty[s], (r & 1) ^ 1, abort_flag, args.status)) break;
                mbar_expect_tx(&full[s], NT_B);
                tma_load_2d(sB + size_t(s) * NT_B, &tmB, &full[s], (it % args.nkb) * TC_BK,
                            (I.kt0 + it / args.nkb) * NT_N);
            }
            // drain: every issued copy must land before the CTA leaves
            mbar_drain(a_full, 0);
            for (int s = 0; s < args.stages && s < it; ++s) {
                const int last = s + ((it - 1 - s) / args.stages) * args.stages;
                mbar_drain(&full[s], (last / args.stages) & 1);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {   // MMA issuer
            constexpr uint32_t IDESC = idesc_bf16(NT_M, NT_N);
            int it = 0;
            bool ok = mbar_wait(a_full, 0, abort_flag, args.status);
            tc_fence_after();
            for (int g = 0; g < ntiles && ok; ++g) {
                const int b = g & 1, use = g >> 1;
                if (!mbar_wait(&tempty[b], (use & 1) ^ 1, abort_flag, args.status)) break;
                tc_fence_after();
                uint32_t acc = 0;
                for (int kb = 0; kb < args.nkb; ++kb, ++it) {
                    const int s = it % args.stages, r = it / args.stages;
                    if (!mbar_wait(&full[s], r & 1, abort_flag, args.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t as = smem_u32(sA + size_t(kb) * NT_A);
                    const uint32_t bs = smem_u32(sB + size_t(s) * NT_B);
#pragma unroll
                    for (int kk = 0; kk < TC_BK / 16; ++kk) {
                        umma_f16(tmem + uint32_t(b * NT_N), sdesc_sw128(as + kk * 32),
                                 sdesc_sw128(bs + kk * 32), IDESC, acc);
                        acc = 1;
                    }
                    umma_commit(&empty[s]);
                }
                if (!ok) break;
                umma_commit(&tfull[b]);
            }
            umma_commit(mma_done);
            mbar_drain(mma_done, 0);
        }
        __syncwarp();
    } else {
        // epilogue: thread = row of its TMEM lane quarter, NT_COLS columns
        const float inf = __int_as_float(0x7f800000);
        const int quarter = warp & 3;
        const int col0 = ((warp - 2) >> 2) * NT_COLS;
        const int row = quarter * 32 + lane;
        const int64_t ru = int64_t(I.row0) + row;
        const bool valid = ru < I.row_end;
        const int q0 = (warp - 2) * NT_QUEUE;
        const float nx = valid ? args.n2[ru] : 0.0f, ebx = valid ? args.eb[ru] : 0.0f;
        const float nxl = __fmul_rd(nx, 1.0f - (args.aerr + 0x1p-20f));
        const float rel = __fdiv_ru(1.0f + 0x1p-21f, 1.0f - args.eps);
        // pair rank of (i, c) is pbase + c
        const int64_t pbase = int64_t(I.i) * args.t - int64_t(I.i) * (I.i + 1) / 2 - I.i - 1;
        int cur = -1;            // component whose bound is in curthr
        float curthr = -inf, nthr = inf;   // nthr: re-read during the previous tile
        unsigned long long seen = 0;
        int cnt = 0;
        auto thr_of = [&](int c) { return __uint_as_float(__ldcg(args.thr + pbase + c)); };
        // pairs with ||h_y||^2 (1 - aerr') - 2 h_x.h_y above this lie beyond th
        auto limit = [&](float th, int ebmax) {
            const float gg = __fadd_ru(__fmaf_ru(th, rel, ebx), __int_as_float(ebmax));
            return valid ? __fadd_ru(__fsub_ru(__fmul_ru(__fmul_ru(gg, gg), 1.0f + 0x1p-20f), nxl),
                                     1e-30f)
                         : -inf;
        };
        // the bound of one component, as last read
        auto bound_of = [&](int c) {
            if (c <= I.i || c >= args.t) return -inf;
            if (c != cur) {
                cur = c;
                curthr = thr_of(c);
                nthr = inf;
            }
            return curthr;
        };
        // the queued pairs, one per lane: those within their component pair's
        // bound go to the survivors and into its slots
        auto flush = [&]() {
            __syncwarp();
#pragma unroll 1
            for (int q = 0; q < cnt; q += 32) {
                const bool have = q + lane < cnt;
                const int at0 = q0 + (have ? q + lane : 0);
                const float dt = qd[at0];
                const int pos = qp[at0], ln = ql[at0];
                const float nxr = __shfl_sync(0xffffffffu, nx, ln);
                const float ebr = __shfl_sync(0xffffffffu, ebx, ln);
                const int c = __ldg(args.colcomp + pos);
                if (!have || c <= I.i || c >= args.t) continue;
                float lo, hi;
                dist_bounds(dt, nxr, __ldg(args.n2 + pos), ebr, __ldg(args.eb + pos), args.aerr,
                            args.eps, lo, hi);
                const float th = thr_of(c);
                if (!(lo <= __fmul_ru(th, 1.0f + 0x1p-22f))) continue;
                const unsigned long long at = atomicAdd(args.count, 1ull);
                if (at < args.cap) {
                    args.su[at] = I.row0 + quarter * 32 + ln;
                    args.sv[at] = pos;
                    args.sl[at] = lo;
                }
                if (hi < th)
                    nt_slot_insert(args.slots + (pbase + c) * args.lambda, args.thr + pbase + c,
                                   args.lambda, __float_as_uint(hi));
            }
            __syncwarp();
            cnt = 0;
        };
        for (int g = 0; g < ntiles; ++g) {
            const int b = g & 1, use = g >> 1;
            const bool got = mbar_wait(&tfull[b], use & 1, abort_flag, args.status);
            if (!__all_sync(0xffffffffu, got)) break;
            tc_fence_after();
            const uint32_t tb = tmem + (uint32_t(quarter * 32) << 16) + uint32_t(b * NT_N + col0);
            const int64_t key0 = int64_t(I.kt0 + g) * NT_N + col0;
            const int4 hc = __ldg(args.hchunk + key0 / NT_COLS);
            // the bound in use and the survivor count as other CTAs left them
            // (read during one tile, used from the next)
            curthr = fminf(curthr, nthr);
            const float bh = hc.x == hc.y ? bound_of(hc.x) : 0.0f;
            nthr = cur >= 0 ? thr_of(cur) : inf;
            const bool over = seen > args.limit;
            if ((g & 15) == 15) seen = *reinterpret_cast<volatile unsigned long long *>(args.count);
            float T = hc.x == hc.y ? limit(bh, hc.z) : 0.0f;
            // the next tile's norms and its record into L1 meanwhile
            if (g + 1 < ntiles && lane < 3) {
                const void *nx =
                    lane < 2 ? static_cast<const void *>(args.nyq + key0 + NT_N + 32 * lane)
                             : static_cast<const void *>(args.hchunk + (key0 + NT_N) / NT_COLS);
                asm volatile("prefetch.global.L1 [%0];" ::"l"(nx));
            }
            // 16 columns: scores in packed pairs, their minimum against T
            auto process = [&](uint32_t(&v)[16], int ch) {
                const int64_t p0 = key0 + ch * 16;
                if (hc.x != hc.y) {   // these columns span components: per 16
                    const int4 ci = __ldg(args.chunk + (p0 >> 4));
                    float th = -inf;
                    if (ci.x == ci.y) {
                        th = bound_of(ci.x);
                    } else {   // the largest of their bounds
                        for (int c = max(ci.x, I.i + 1); c <= ci.y && c < args.t; ++c)
                            th = fmaxf(th, thr_of(c));
                    }
                    T = th >= 0.0f ? limit(th, ci.z) : -inf;
                }
                float sc[16];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const ulonglong2 ny =
                        __ldg(reinterpret_cast<const ulonglong2 *>(args.nyq + p0 + 4 * q));
                    nt_scores(v[4 * q], v[4 * q + 1], ny.x, sc[4 * q], sc[4 * q + 1]);
                    nt_scores(v[4 * q + 2], v[4 * q + 3], ny.y, sc[4 * q + 2], sc[4 * q + 3]);
                }
                float m[5];
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    m[q] = fminf(fminf(sc[3 * q], sc[3 * q + 1]), sc[3 * q + 2]);
                const float mn = fminf(fminf(fminf(m[0], m[1]), m[2]), fminf(fminf(m[3], m[4]), sc[15]));
                if (!__any_sync(0xffffffffu, mn <= T)) return;
                unsigned bits = 0;
#pragma unroll
                for (int c = 0; c < 16; ++c) bits |= sc[c] <= T ? 1u << c : 0u;
#pragma unroll 1
                while (true) {   // one per lane and turn
                    const unsigned who = __ballot_sync(0xffffffffu, bits != 0u);
                    if (!who) break;
                    if (cnt + __popc(who) > NT_QUEUE) flush();
                    if (bits) {
                        const int c = __ffs(bits) - 1;
                        bits &= bits - 1u;
                        uint32_t d[8];   // the dot product of column c, by its bits
#pragma unroll
                        for (int x = 0; x < 8; ++x) d[x] = (c & 1) ? v[2 * x + 1] : v[2 * x];
#pragma unroll
                        for (int w = 1; w < 4; ++w)
#pragma unroll
                            for (int x = 0; x < (8 >> w); ++x)
                                d[x] = (c >> w) & 1 ? d[2 * x + 1] : d[2 * x];
                        const int at = q0 + cnt + __popc(who & ((1u << lane) - 1u));
                        qd[at] = __uint_as_float(d[0]);
                        qp[at] = int(p0) + c;
                        ql[at] = lane;
                    }
                    cnt += __popc(who);
                }
            };
            // too many survivors end the search (the caller starts over on the
            // warp kernel); this CTA's tiles still flow, later CTAs leave at once
            if (!__any_sync(0xffffffffu, over) && (hc.x != hc.y || bh >= 0.0f)) {
                uint32_t va[16], vb[16];
                __syncwarp();
                tmem_ld16(tb, va);
#pragma unroll 1
                for (int ch = 0; ch < NT_COLS / 16; ch += 2) {
                    tmem_ld_wait16(va);
                    __syncwarp();
                    tmem_ld16(tb + (ch + 1) * 16, vb);
                    process(va, ch);
                    tmem_ld_wait16(vb);
                    __syncwarp();
                    if (ch + 2 < NT_COLS / 16) tmem_ld16(tb + (ch + 2) * 16, va);
                    process(vb, ch + 1);
                }
                // many survivors tighten the bounds at once; a few wait (the
                // tensor pipe waits for the slowest of the warps)
                if (cnt >= NT_FLUSH) flush();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
        }
        __syncwarp();
        flush();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    // (beside the count, which the host reads anyway)
    if (threadIdx.x == 0 && *abort_flag) atomicMax(args.count, NT_GAVE_UP);
}

// Between the launch that only lowers the bounds and the search: the slots
// start again (the search meets the same pairs once more, and a slot has to
// hold a pair of its own), the bounds stay.
__global__ void nt_restart_kernel(unsigned *__restrict__ slots, int64_t nslots,
                                  unsigned long long *__restrict__ count,
                                  unsigned long long limit) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < nslots) slots[i] = 0x7f800000u;
    if (i == 0 && *count <= limit) *count = 0;
}

// Survivors within the final bounds, counted per component pair (slot: the
// arrival number, -1 for the others), then grouped.
__global__ void nt_count_kernel(const int32_t *__restrict__ su, const int32_t *__restrict__ sv,
                                const float *__restrict__ sl, int64_t count, int64_t t,
                                const int32_t *__restrict__ colcomp,
                                const unsigned *__restrict__ thr, int32_t *__restrict__ cnt,
                                int32_t *__restrict__ slot) {
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= count) return;
    const int64_t i = colcomp[su[e]], c = colcomp[sv[e]];
    const int64_t p = i * t - i * (i + 1) / 2 - i - 1 + c;
    slot[e] = sl[e] <= __fmul_ru(__uint_as_float(thr[p]), 1.0f + 0x1p-22f) ? atomicAdd(cnt + p, 1)
                                                                            : -1;
}

__global__ void nt_scatter_kernel(const int32_t *__restrict__ su, const int32_t *__restrict__ sv,
                                  int64_t count, int64_t t, const int32_t *__restrict__ colcomp,
                                  const int32_t *__restrict__ members,
                                  const int32_t *__restrict__ off, const int32_t *__restrict__ slot,
                                  int2 *__restrict__ grouped) {
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= count || slot[e] < 0) return;
    const int u = su[e], v = sv[e];
    const int64_t i = colcomp[u], c = colcomp[v];
    const int64_t p = i * t - i * (i + 1) / 2 - i - 1 + c;
    grouped[int64_t(off[p]) + slot[e]] = make_int2(members[u], members[v]);
}

// The lambda smallest (w, min id, max id) of a component pair's survivors,
// one warp per component pair.
template <int XR>
__global__ void nt_select_kernel(const float *__restrict__ X, int d,
                                 const int2 *__restrict__ grouped, const int32_t *__restrict__ off,
                                 int64_t t, int lambda, int32_t *__restrict__ eu_out,
                                 int32_t *__restrict__ ev_out, float *__restrict__ ew_out,
                                 int32_t *__restrict__ eci, int32_t *__restrict__ ecj,
                                 int *status) {
    const int64_t npairs = t * (t - 1) / 2;
    const int64_t w0 = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
    const int lane = threadIdx.x & 31;
    for (int64_t p = w0; p < npairs; p += nw) {
        int64_t i, j;
        pair_of(p, t, i, j);
        uint64_t eh = ~0ull;
        uint32_t el = ~0u;
        int eu = 0, ev = 0, have = 0;
        if (off[p] == off[p + 1]) {   // the nearest pair always survives: a bug, never an id of -1
            if (lane == 0) set_status(status, STATUS_INTERNAL);
            eh = 0;
            have = 1;
        }
        for (int e0 = off[p]; e0 < off[p + 1]; e0 += 4) {
            int qa[4], qb[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int2 g = grouped[min(e0 + e, off[p + 1] - 1)];
                qa[e] = g.x;
                qb[e] = g.y;
            }
            pairs_batch<XR>(X, d, min(4, off[p + 1] - e0), qa, qb, eh, el, eu, ev, lambda, have,
                            lane);
        }
        // fewer pairs than lambda: repeat the farthest
        const int src = lane < have ? lane : have - 1;
        const int ru = __shfl_sync(0xffffffffu, eu, src);
        const int rv = __shfl_sync(0xffffffffu, ev, src);
        const float rw = __uint_as_float(uint32_t(shfl_idx_u64(eh, src) >> 32));
        if (lane < lambda) {
            const int64_t o = p * lambda + lane;
            eu_out[o] = ru;
            ev_out[o] = rv;
            ew_out[o] = rw;
            eci[o] = int32_t(i);
            ecj[o] = int32_t(j);
        }
    }
}

// ------------------------------------------------------- warp kernel

// One warp per work item (component i, block of 32 of its members): the
// top-lambda list of every later component j goes to out[(item, j - i - 1)].
// item_off[i] = first item of component i (t + 1 entries), out_off[i] =
// first output slot (in lists) of component i's items.
template <int NKS, int XR>
__global__ void __launch_bounds__(NP_WARPS * 32)
    nearest_pairs_kernel(const float *__restrict__ X, int d, const __nv_bfloat16 *__restrict__ H,
                         const float *__restrict__ heb, const float *__restrict__ hn2,
                         const int32_t *__restrict__ members, const int32_t *__restrict__ comp_off,
                         const int64_t *__restrict__ item_off, const int64_t *__restrict__ out_off,
                         int64_t t, int64_t items, int lambda, int32_t *__restrict__ ou,
                         int32_t *__restrict__ ov, float *__restrict__ ow, float aerr, float eps,
                         unsigned long long *__restrict__ stats) {
    using S = NpStage<NKS>;
    extern __shared__ __align__(128) char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    char *wb = smem + warp * S::WARP_BYTES;
    const uint32_t sbuf = smem_addr(wb);
    float2 *s_en = reinterpret_cast<float2 *>(wb + S::ROWS_BYTES);          // 32 (eb, n2) of u
    int32_t *s_u = reinterpret_cast<int32_t *>(wb + S::ROWS_BYTES + 256);   // 32 ids of u
    float4 *s_v = reinterpret_cast<float4 *>(wb + S::ROWS_BYTES + 384);     // 8 (id, eb, n2) of v
    const float inf = __int_as_float(0x7f800000);
    const int g4 = lane >> 2, t4 = lane & 3;
    unsigned long long pairs = 0, canon = 0;
    const int64_t nw = int64_t(gridDim.x) * NP_WARPS;
    for (int64_t q = int64_t(blockIdx.x) * NP_WARPS + warp; q < items; q += nw) {
        // component i of item q: the last i with item_off[i] <= q
        int64_t lo_i = 0, hi_i = t;   // item_off[lo_i] <= q < item_off[hi_i]
        while (hi_i - lo_i > 1) {
            const int64_t mid = (lo_i + hi_i) >> 1;
            if (item_off[mid] <= q) lo_i = mid; else hi_i = mid;
        }
        const int64_t i = lo_i;
        const int64_t b = q - item_off[i];
        const int u0 = comp_off[i] + int(b) * 32;
        const int nu = min(32, comp_off[i + 1] - u0);
        int myu = -1;
        float2 ue = make_float2(inf, 0.0f);
        if (lane < nu) {
            myu = members[u0 + lane];
            ue = make_float2(__ldg(heb + myu), __ldg(hn2 + myu));
        }
        s_en[lane] = ue;
        s_u[lane] = myu;
        stage_rows<NKS>(H, myu, sbuf, lane);
        int64_t slot = out_off[i] + b * (t - 1 - i);
        for (int64_t j = i + 1; j < t; ++j, ++slot) {
            uint64_t eh = ~0ull;
            uint32_t el = ~0u;
            int eu = -1, ev = -1, have = 0;
            const int v0 = comp_off[j], v1 = comp_off[j + 1];
            for (int vc = v0; vc < v1; vc += 8) {
                const int nvb = min(8, v1 - vc);
                if (lane < nvb) {
                    const int v = members[vc + lane];
                    s_v[lane] = make_float4(__int_as_float(v), __ldg(heb + v), __ldg(hn2 + v), 0.0f);
                }
                __syncwarp();
                uint32_t b0[NKS], b1[NKS];
                {
                    const bool has = g4 < nvb;
                    const __nv_bfloat16 *hf =
                        H + int64_t(has ? __float_as_int(s_v[g4].x) : 0) * S::LD;
#pragma unroll
                    for (int ks = 0; ks < NKS; ++ks) {
                        b0[ks] = has ? ldg_u32(hf + 16 * ks + 2 * t4) : 0u;
                        b1[ks] = has ? ldg_u32(hf + 16 * ks + 8 + 2 * t4) : 0u;
                    }
                }
                float acc[2][4];
                round_dots<NKS>(sbuf, b0, b1, lane, acc);
                // this lane: pairs (u slot 16 T + g4 + 8 (e2 >> 1), v slot 2 t4 + (e2 & 1))
                float lo[2][4], hi[2][4];
#pragma unroll
                for (int T = 0; T < 2; ++T)
#pragma unroll
                    for (int e2 = 0; e2 < 4; ++e2) {
                        const int ui = 16 * T + g4 + 8 * (e2 >> 1), vj = 2 * t4 + (e2 & 1);
                        lo[T][e2] = inf;
                        hi[T][e2] = inf;
                        if (ui < nu && vj < nvb) {
                            const float2 a = s_en[ui];
                            const float4 c = s_v[vj];
                            dist_bounds(acc[T][e2], a.y, c.z, a.x, c.y, aerr, eps, lo[T][e2],
                                        hi[T][e2]);
                        }
                    }
                if (lane == 0) pairs += unsigned(nu * nvb);
                // threshold: the list's lambda-th weight; while the list is not
                // full, the lambda-th smallest upper bound of this step (lambda
                // pairs at most that far exist, so a pair above it is beaten)
                float thr = have == lambda ? __uint_as_float(uint32_t(__shfl_sync(
                                                 0xffffffffu, uint32_t(eh >> 32), lambda - 1)))
                                           : inf;
                if (have < lambda) {
                    float hv[8];
#pragma unroll
                    for (int T = 0; T < 2; ++T)
#pragma unroll
                        for (int e2 = 0; e2 < 4; ++e2) hv[4 * T + e2] = hi[T][e2];
                    float kth = inf;
                    for (int r = 0; r < lambda; ++r) {
                        float m = inf;
                        int at = -1;
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            if (hv[e] < m) {
                                m = hv[e];
                                at = e;
                            }
                        float wm = m;
#pragma unroll
                        for (int o = 16; o >= 1; o >>= 1)
                            wm = fminf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
                        kth = wm;
                        if (!(wm < inf)) break;
                        // remove one occurrence: the lowest lane holding it
                        const unsigned holders = __ballot_sync(0xffffffffu, m == wm && at >= 0);
                        if (lane == __ffs(holders) - 1) {
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                if (e == at) hv[e] = inf;
                        }
                    }
                    thr = fminf(thr, kth);
                }
                const float bound = __fmul_ru(thr, 1.0f + 0x1p-22f);
                // survivors among the valid pairs only (the bound is +inf while a
                // step has fewer than lambda pairs)
                unsigned my = 0;
#pragma unroll
                for (int T = 0; T < 2; ++T)
#pragma unroll
                    for (int e2 = 0; e2 < 4; ++e2) {
                        const int ui = 16 * T + g4 + 8 * (e2 >> 1), vj = 2 * t4 + (e2 & 1);
                        if (ui < nu && vj < nvb && lo[T][e2] <= bound) my |= 1u << (4 * T + e2);
                    }
                {
                    int cnt = __popc(my);
#pragma unroll
                    for (int o = 16; o >= 1; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
                    if (lane == 0) canon += unsigned(cnt);
                }
#pragma unroll 1
                while (true) {
                    int qa[4], qb[4], nq = 0;
#pragma unroll 1
                    while (nq < 4) {
                        const unsigned any = __ballot_sync(0xffffffffu, my != 0u);
                        if (!any) break;
                        const int sl = __ffs(any) - 1;
                        const int bit = __ffs(__shfl_sync(0xffffffffu, my, sl)) - 1;
                        if (lane == sl) my &= my - 1u;
                        const int ui = 16 * (bit >> 2) + (sl >> 2) + 8 * ((bit & 3) >> 1);
                        const int vj = 2 * (sl & 3) + (bit & 1);
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (e == nq) {
                                qa[e] = s_u[ui];
                                qb[e] = __float_as_int(s_v[vj].x);
                            }
                        ++nq;
                    }
                    if (nq == 0) break;
                    pairs_batch<XR>(X, d, nq, qa, qb, eh, el, eu, ev, lambda, have, lane);
                }
                __syncwarp();   // s_v is rewritten by the next step
            }
            // the list, padded by repeating its last entry
            const int src = lane < have ? lane : have - 1;
            const int ru = __shfl_sync(0xffffffffu, eu, src);
            const int rv = __shfl_sync(0xffffffffu, ev, src);
            const float rw = __uint_as_float(uint32_t(shfl_idx_u64(eh, src) >> 32));
            if (lane < lambda) {
                ou[slot * lambda + lane] = ru;
                ov[slot * lambda + lane] = rv;
                ow[slot * lambda + lane] = rw;
            }
        }
        __syncwarp();   // the block's rows stay until every component j is done
    }
    if (stats && lane == 0) {
        atomicAdd(stats, pairs);
        atomicAdd(stats + 1, canon);
    }
}

// Per component pair (i, j): merge the lists of C_i's blocks (nb_i lists of
// lambda entries) into the lambda smallest (w, min id, max id), written as
// edges (pair rank) * lambda + r with u in C_i, v in C_j. One warp per pair.
__global__ void nearest_merge_kernel(const int32_t *__restrict__ comp_off,
                                     const int64_t *__restrict__ out_off, int64_t t, int lambda,
                                     const int32_t *__restrict__ ou, const int32_t *__restrict__ ov,
                                     const float *__restrict__ ow, int32_t *__restrict__ eu,
                                     int32_t *__restrict__ ev, float *__restrict__ ew,
                                     int32_t *__restrict__ eci, int32_t *__restrict__ ecj) {
    const int lane = threadIdx.x & 31;
    const int64_t npairs = t * (t - 1) / 2;
    const int64_t w0 = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t p = w0; p < npairs; p += nw) {
        int64_t i, j;
        pair_of(p, t, i, j);
        const int64_t nb = (comp_off[i + 1] - comp_off[i] + 31) / 32;
        const int64_t total = nb * lambda;
        // the lists of this pair sit at out_off[i] + b (t - 1 - i) + (j - i - 1)
        uint64_t bh = ~0ull;
        uint32_t bl = ~0u;
        int bu = -1, bv = -1;
        for (int r = 0; r < lambda; ++r) {
            // the r-th smallest: every lane scans its share, warp minimum
            uint64_t mh = ~0ull;
            uint32_t ml = ~0u;
            int64_t at = -1;
            for (int64_t e = lane; e < total; e += 32) {
                const int64_t b = e / lambda, rr = e - b * lambda;
                const int64_t s = (out_off[i] + b * (t - 1 - i) + (j - i - 1)) * lambda + rr;
                const int a = ou[s], c = ov[s];
                const uint64_t h = pkey_hi(ow[s], a, c);
                const uint32_t l = uint32_t(a < c ? c : a);
                // strictly after the previous pick: a pair sits in one block's
                // list only, so equal keys are a list's padding repeats
                const bool after = r == 0 || pkey_less(bh, bl, h, l);
                if (after && pkey_less(h, l, mh, ml)) {
                    mh = h;
                    ml = l;
                    at = s;
                }
            }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                const uint64_t oh = shfl_xor_u64(mh, o);
                const uint32_t ol = __shfl_xor_sync(0xffffffffu, ml, o);
                const int64_t oa = int64_t(shfl_xor_u64(uint64_t(at), o));
                if (pkey_less(oh, ol, mh, ml) || (oh == mh && ol == ml && oa < at)) {
                    mh = oh;
                    ml = ol;
                    at = oa;
                }
            }
            if (at >= 0) {
                bh = mh;
                bl = ml;
                bu = ou[at];
                bv = ov[at];
            }
            // fewer distinct pairs than lambda: repeat the last one
            if (lane == 0) {
                const int64_t e = p * lambda + r;
                eu[e] = bu;
                ev[e] = bv;
                ew[e] = __uint_as_float(uint32_t(bh >> 32));
                eci[e] = int32_t(i);
                ecj[e] = int32_t(j);
            }
        }
    }
}

template <int NKS, int XR>
famst_status launch_np(const Exec &ex, const float *X, int d, const HalfRows &hr,
                       const int32_t *members, const int32_t *comp_off, const int64_t *item_off,
                       const int64_t *out_off, int64_t t, int64_t items, int lambda, int32_t *ou,
                       int32_t *ov, float *ow, float aerr, float eps,
                       unsigned long long *stats) {
    using S = NpStage<NKS>;
    auto *fn = nearest_pairs_kernel<NKS, XR>;
    if (set_smem_attr(fn, S::SMEM, ex.stream) != cudaSuccess) return FAMST_ERR_CUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, NP_WARPS * 32, S::SMEM) !=
            cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    const int64_t want = (items + NP_WARPS - 1) / NP_WARPS;
    const int64_t cap = int64_t(ex.num_sms) * per_sm;
    const unsigned grid = unsigned(want < cap ? (want > 0 ? want : 1) : cap);
    FAMST_LAUNCH(ex, fn, grid, NP_WARPS * 32, S::SMEM, X, d, hr.h, hr.eb, hr.n2, members,
                 comp_off, item_off, out_off, t, items, lambda, ou, ov, ow, aerr, eps, stats);
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

}  // namespace

namespace {

// Below this the sampling, grouping and selection around the tile pass
// (about 0.3 ms of launches) cost more than the warp kernel's whole run:
// 4100 x 128 in 10 components 1.47 ms warp kernel, 0.48 ms tiles.
constexpr int64_t NT_MIN_N = 1024;

size_t nt_workspace(int64_t n, int64_t t, int lambda) {
    const int64_t npairs = nearest_pairs(t), cap = nearest_plan(n, t, lambda).cap;
    const int64_t npad = (n + NT_N - 1) / NT_N * NT_N;
    const int64_t items = (n / NT_M + t) * 2 + 16 * 1024;
    return align256(size_t(npad) * 256 * 2) + align256(size_t(npad) * 4) * 4 +
           align256(size_t(npad / 16) * 16) + align256(size_t(npad / NT_COLS) * 16) +
           align256(size_t(npairs) * 4) +
           align256(size_t(npairs) * lambda * 4) + align256(size_t(npairs + 1) * 4) * 2 +
           scan_workspace(npairs + 1) + align256(size_t(cap) * 4) * 4 + align256(size_t(cap) * 8) +
           align256(size_t(items) * sizeof(NtItem)) + 1024;
}

// The tensor-core pass; *done = false (and nothing written) when the survivors
// overflowed their buffer.
template <int XR>
famst_status nearest_tc(const Exec &ex, Arena &ar, const float *X, int d, const HalfRows &hr,
                        const int32_t *members, const int32_t *comp_off,
                        const int32_t *comp_off_host, int64_t t, int lambda, float aerr, float eps,
                        int32_t *eu, int32_t *ev, float *ew, int32_t *eci, int32_t *ecj,
                        bool *done) {
    *done = false;
    const int64_t n = comp_off_host[t], npairs = nearest_pairs(t);
    const NearestPlan plan = nearest_plan(n, t, lambda);
    const int64_t cap = plan.cap;
    const bool bounds_first = plan.bounds_first;
    const int64_t ntile = (n + NT_N - 1) / NT_N, npad = ntile * NT_N;
    // items: 128 rows of a component against a run of the tiles that hold
    // later components; runs of about a sixteenth of an SM's share, so that
    // the last round is short
    int64_t total = 0;
    for (int64_t i = 0; i + 1 < t; ++i)
        total += (int64_t(comp_off_host[i + 1] - comp_off_host[i]) + NT_M - 1) / NT_M *
                 (ntile - comp_off_host[i + 1] / NT_N);
    // the first launch: a few runs per SM
    int64_t total1 = 0;
    for (int64_t i = 0; i + 1 < t; ++i) total1 += ntile - comp_off_host[i + 1] / NT_N;
    const int64_t run1 = std::max<int64_t>(4, total1 / (4 * int64_t(ex.num_sms)));
    const int64_t run = std::max<int64_t>(8, total / (16 * int64_t(ex.num_sms)));
    std::vector<NtItem> items;
    auto add = [&](int64_t i, int64_t r, int64_t len) {
        const int64_t k0 = comp_off_host[i + 1] / NT_N;
        const int64_t parts = (ntile - k0 + len - 1) / len;
        for (int64_t q = 0; q < parts; ++q) {
            NtItem I;
            I.row0 = int32_t(r);
            I.row_end = comp_off_host[i + 1];
            I.i = int32_t(i);
            I.kt0 = int32_t(k0 + (ntile - k0) * q / parts);
            I.kt1 = int32_t(k0 + (ntile - k0) * (q + 1) / parts);
            items.push_back(I);
        }
    };
    // (bounds_first: the first launch only lowers the bounds, and the search
    // goes over all rows)
    for (int64_t i = 0; i + 1 < t; ++i) add(i, comp_off_host[i], run1);
    const size_t first = items.size();
    for (int64_t i = 0; i + 1 < t; ++i)
        for (int64_t r = comp_off_host[i] + (bounds_first ? 0 : NT_M); r < comp_off_host[i + 1];
             r += NT_M)
            add(i, r, run);
    __nv_bfloat16 *Hs = ar.take<__nv_bfloat16>(size_t(npad) * hr.ld);
    float *n2 = ar.take<float>(size_t(npad));
    float *eb = ar.take<float>(size_t(npad));
    float *nyq = ar.take<float>(size_t(npad));
    int32_t *colcomp = ar.take<int32_t>(size_t(npad));
    int4 *chunk = ar.take<int4>(size_t(npad / 16));
    int4 *hchunk = ar.take<int4>(size_t(npad / NT_COLS));
    unsigned *thr = ar.take<unsigned>(size_t(npairs));
    unsigned *slots = ar.take<unsigned>(size_t(npairs) * lambda);
    int32_t *cnt = ar.take<int32_t>(size_t(npairs + 1));
    int32_t *off = ar.take<int32_t>(size_t(npairs + 1));
    int32_t *su = ar.take<int32_t>(size_t(cap));
    int32_t *sv = ar.take<int32_t>(size_t(cap));
    float *sl = ar.take<float>(size_t(cap));
    int32_t *slot = ar.take<int32_t>(size_t(cap));
    int2 *grouped = ar.take<int2>(size_t(cap));
    NtItem *d_items = ar.take<NtItem>(items.size());
    unsigned long long *count = ar.take<unsigned long long>(1);
    if (!Hs || !n2 || !eb || !nyq || !colcomp || !chunk || !hchunk || !thr || !slots || !cnt || !off || !su ||
        !sv || !sl || !slot || !grouped || !d_items || !count)
        return FAMST_ERR_OOM;
    if (cudaMemcpyAsync(d_items, items.data(), items.size() * sizeof(NtItem),
                        cudaMemcpyHostToDevice, ex.stream) != cudaSuccess ||
        cudaMemsetAsync(count, 0, 8, ex.stream) != cudaSuccess ||
        cudaMemsetAsync(cnt, 0, size_t(npairs + 1) * 4, ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    FAMST_LAUNCH(ex, nt_gather_kernel, unsigned((npad * 32 + 255) / 256), 256, 0, hr.h, hr.ld,
                 hr.eb, hr.n2, members, comp_off, t, n, npad, aerr, Hs, n2, eb, nyq, colcomp, count);
    FAMST_LAUNCH(ex, nt_chunk_kernel, unsigned((npad / 16 + 255) / 256), 256, 0, colcomp, eb, n,
                 npad / 16, 16, t, chunk);
    FAMST_LAUNCH(ex, nt_chunk_kernel, unsigned((npad / NT_COLS + 63) / 64), 64, 0, colcomp, eb, n,
                 npad / NT_COLS, NT_COLS, t, hchunk);
    const int64_t pw = (npairs * 32 + 127) / 128, pcap = int64_t(ex.num_sms) * 16;
    const unsigned pgrid = unsigned(pw < pcap ? pw : pcap);
    FAMST_LAUNCH(ex, nt_sample_kernel<XR>, unsigned(npairs < pcap ? npairs : pcap), NT_SW * 32, 0,
                 X, d, members, comp_off, t, lambda, thr, slots);
    CUtensorMap mA, mB;
    if (!make_map(&mA, Hs, n, hr.ld, NT_M) || !make_map(&mB, Hs, n, hr.ld, NT_N))
        return FAMST_ERR_CUDA;
    NtArgs a{};
    a.items = d_items;
    a.nkb = hr.ld / TC_BK;
    const size_t fixed = 1024 + size_t(a.nkb) * NT_A + size_t(NT_EPI) * NT_QUEUE * 12 + 512;
    a.stages = int(std::min<size_t>(6, (size_t(227) * 1024 - fixed) / NT_B));
    const size_t smem = fixed + size_t(a.stages) * NT_B;
    a.n = n;
    a.t = t;
    a.lambda = lambda;
    a.nyq = nyq;
    a.n2 = n2;
    a.eb = eb;
    a.colcomp = colcomp;
    a.chunk = chunk;
    a.hchunk = hchunk;
    a.thr = thr;
    a.slots = slots;
    a.count = count;
    a.cap = (unsigned long long)cap;
    a.su = su;
    a.sv = sv;
    a.sl = sl;
    a.aerr = aerr;
    a.eps = eps;
    a.status = ex.dstatus;
    if (set_smem_attr(nearest_tc_kernel, smem, ex.stream) != cudaSuccess) return FAMST_ERR_CUDA;
    a.limit = a.cap;
    if (bounds_first) {
        a.cap = 0;
        a.limit *= 8;
    }
    FAMST_LAUNCH(ex, nearest_tc_kernel, unsigned(first), NT_THREADS, smem, mA, mB, a);
    if (bounds_first) {
        FAMST_LAUNCH(ex, nt_restart_kernel, unsigned((npairs * lambda + 255) / 256), 256, 0, slots,
                     npairs * lambda, count, a.limit);
        a.cap = a.limit = (unsigned long long)cap;
    }
    if (items.size() > first) {
        a.items = d_items + first;
        FAMST_LAUNCH(ex, nearest_tc_kernel, unsigned(items.size() - first), NT_THREADS, smem, mA, mB,
                     a);
    }
    unsigned long long got = 0;
    if (cudaMemcpyAsync(&got, count, 8, cudaMemcpyDeviceToHost, ex.stream) != cudaSuccess ||
        cudaStreamSynchronize(ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    if (got >= NT_GAVE_UP) return FAMST_ERR_TIMEOUT;
    if (got > (unsigned long long)cap) return FAMST_OK;
    const unsigned sgrid = unsigned((got + 255) / 256);
    if (got > 0)
        FAMST_LAUNCH(ex, nt_count_kernel, sgrid, 256, 0, su, sv, sl, int64_t(got), t, colcomp, thr,
                     cnt, slot);
    famst_status st = exclusive_scan_i32(ex, ar, cnt, off, npairs + 1, nullptr);
    if (st != FAMST_OK) return st;
    if (got > 0)
        FAMST_LAUNCH(ex, nt_scatter_kernel, sgrid, 256, 0, su, sv, int64_t(got), t, colcomp,
                     members, off, slot, grouped);
    FAMST_LAUNCH(ex, nt_select_kernel<XR>, pgrid, 128, 0, X, d, grouped, off, t, lambda, eu, ev, ew,
                 eci, ecj, ex.dstatus);
    *done = true;
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

}  // namespace

size_t connect_nearest_workspace(int64_t n, int64_t t, int lambda) {
    const size_t warp = 2 * align256(size_t(t + 1) * 8) + nearest_warp_bytes(n, t, lambda) + 1024;
    const bool tensor = n >= NT_MIN_N && nearest_plan(n, t, lambda).tensor;
    return std::max(warp, tensor ? nt_workspace(n, t, lambda) : 0);
}

// comp_off_host: the t + 1 member offsets on the host (the list layout is
// planned there). hr: BF16 rows of the points (ld <= 256).
famst_status connect_nearest(const Exec &ex, Arena &ar, const float *X, int d,
                             const HalfRows &hr, const int32_t *members,
                             const int32_t *comp_off, const int32_t *comp_off_host, int64_t t,
                             int lambda, int32_t *eu, int32_t *ev, float *ew, int32_t *eci,
                             int32_t *ecj, unsigned long long *stats) {
    if (t < 2) return FAMST_OK;
    if (!hr.h || hr.ld > 256) return FAMST_ERR_UNSUPPORTED;
    const float aerr = float(hr.ld * std::ldexp(1.0, -19) + std::ldexp(1.0, -20));
    const float eps = float((d + 16) * std::ldexp(1.0, -24) * 1.1);
    if (comp_off_host[t] >= NT_MIN_N && nearest_plan(comp_off_host[t], t, lambda).tensor &&
        encode_fn()) {
        const size_t mark = ar.off;
        bool done = false;
        const famst_status s =
            d <= 64 ? nearest_tc<2>(ex, ar, X, d, hr, members, comp_off, comp_off_host, t, lambda,
                                    aerr, eps, eu, ev, ew, eci, ecj, &done)
            : d <= 128 ? nearest_tc<4>(ex, ar, X, d, hr, members, comp_off, comp_off_host, t,
                                       lambda, aerr, eps, eu, ev, ew, eci, ecj, &done)
                       : nearest_tc<0>(ex, ar, X, d, hr, members, comp_off, comp_off_host, t,
                                       lambda, aerr, eps, eu, ev, ew, eci, ecj, &done);
        ar.off = mark;
        if (s != FAMST_OK || done) return s;
    }
    std::vector<int64_t> item_off(size_t(t + 1)), out_off(size_t(t + 1));
    item_off[0] = 0;
    out_off[0] = 0;
    for (int64_t i = 0; i < t; ++i) {
        const int64_t nb = (comp_off_host[i + 1] - comp_off_host[i] + 31) / 32;
        item_off[size_t(i + 1)] = item_off[size_t(i)] + nb;
        out_off[size_t(i + 1)] = out_off[size_t(i)] + nb * (t - 1 - i);
    }
    const int64_t items = item_off[size_t(t)], lists = out_off[size_t(t)];
    int64_t *d_item = ar.take<int64_t>(size_t(t + 1));
    int64_t *d_out = ar.take<int64_t>(size_t(t + 1));
    int32_t *ou = ar.take<int32_t>(size_t(lists) * lambda);
    int32_t *ov = ar.take<int32_t>(size_t(lists) * lambda);
    float *ow = ar.take<float>(size_t(lists) * lambda);
    if (!d_item || !d_out || !ou || !ov || !ow) return FAMST_ERR_OOM;
    if (cudaMemcpyAsync(d_item, item_off.data(), size_t(t + 1) * 8, cudaMemcpyHostToDevice,
                        ex.stream) != cudaSuccess ||
        cudaMemcpyAsync(d_out, out_off.data(), size_t(t + 1) * 8, cudaMemcpyHostToDevice,
                        ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    famst_status st;
    if (hr.ld == 64)
        st = launch_np<4, 2>(ex, X, d, hr, members, comp_off, d_item, d_out, t, items, lambda, ou,
                             ov, ow, aerr, eps, stats);
    else if (hr.ld == 128)
        st = launch_np<8, 4>(ex, X, d, hr, members, comp_off, d_item, d_out, t, items, lambda, ou,
                             ov, ow, aerr, eps, stats);
    else
        st = launch_np<16, 0>(ex, X, d, hr, members, comp_off, d_item, d_out, t, items, lambda,
                              ou, ov, ow, aerr, eps, stats);
    if (st != FAMST_OK) return st;
    // the host vectors must outlive the copies above
    if (cudaStreamSynchronize(ex.stream) != cudaSuccess) return FAMST_ERR_CUDA;
    const int64_t npairs = t * (t - 1) / 2;
    int64_t mg = (npairs * 32 + 255) / 256;
    const int64_t mcap = int64_t(ex.num_sms) * 16;
    FAMST_LAUNCH(ex, nearest_merge_kernel, unsigned(mg < mcap ? mg : mcap), 256, 0, comp_off,
                 d_out, t, lambda, ou, ov, ow, eu, ev, ew, eci, ecj);
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

}  // namespace famst
