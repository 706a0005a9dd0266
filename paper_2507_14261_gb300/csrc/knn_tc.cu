// Phase 1 (Algorithm 1, GetANNs) on tcgen05 tensor cores, exact result.
//
// Score. With centred coordinates x' = fl(x - mean), the squared distance
// is ||x'_i||^2 + s(i,j) with s(i,j) = ||x'_j||^2 - 2 x'_i . x'_j; the first
// term is constant along a row, so rows are ranked by s. The dot products
// run on the tensor cores in BF16 with FP32 accumulation: BF16 mode uses
// xh = bf16(x'); BF16X3 mode adds the two correction products of the
// hi/lo split x' ~ xh + xl (xh.yh + xl.yh + xh.yl), whose error is
// O(2^-16) instead of O(2^-8).
//
// Kernel (one CTA per 128 query rows, 18 warps):
//   warp 0     TMA producer: the query tile's operand rows once (resident),
//              then 256-key tiles, one 64-wide K block per ring stage;
//   warp 1     allocates 512 TMEM columns (two 128 x 256 FP32
//              accumulators) and one lane issues tcgen05.mma (M=128, N=256,
//              K=16 per instruction) with SW128 K-major smem descriptors;
//              tcgen05.commit frees ring stages and publishes accumulators;
//   warps 2..  sixteen epilogue warps, four per TMEM lane quarter: thread r of
//              a warp owns query row r of the quarter and, of every tile, a
//              fourth of the columns (16-column chunks g, g + 4, g + 8, g + 12
//              for the quarter's warp g). It loads 16 columns at a time with
//              tcgen05.ld and forms s = ny_j - 2 acc (key norms from L1).
//              A row keeps no sorted list of ids (32 to 64 scores and ids per
//              thread left room for eight warps, which could not hide the
//              latency of TMEM, norms and branches, and two column halves each
//              kept a full list):
//              - bound: a thread keeps its R smallest scores, a sorted list; a
//                new one goes in by R min/max pairs. The row's T is the largest
//                of its four threads' R-th (shared memory): each list holds R
//                distinct keys' scores at or below it, so at least 4 R keys
//                score <= T. (Tight when the near keys are spread over the four
//                column groups and do not come last: passes without pruned
//                lists take the rows in a scrambled order, tile_rows.cuh.)
//              - log: a key that scores at most the T of the moment is appended
//                to the thread's log of (score, id) in a scratch area of the
//                CTA (about 4 R ln(keys / 4 R) entries per row, L2-resident).
//                The item's first tile is read twice from TMEM, for T and then
//                for the log.
//              - at the end a warp per row keeps the logged keys at or below
//                the final T and lowers it to the k-th key plus the score
//                error's margin: the row's candidates, with s+ = that bound.
//              Bound: the epilogue's issue slots (48 % of peak: min/max pairs,
//              norms and log branches; the tensor cores wait for it). Against
//              sorted id lists in eight warps: 65,537 x 96 overlapping points at
//              k = 32 7.4 -> 4.05 ms, 256 clouds of 500 to 20,000 points
//              (k = 16) 31.2 -> 23.5, 1M x 128 sphere points (k = 32, pruned
//              lists) 9.5 -> 8.05, five masked passes of a 10,000-point EMST
//              1.31 -> 0.92; 100,000 x 128 blobs (k = 16, pruned lists of few
//              tiles, so the first tile's second turn weighs) 1.05 -> 1.18.
// Work items: a query tile with its key tiles (all of them, or a pruned
// list); a long pruned list is split into parts run by separate CTAs, whose
// rows' candidates split_merge_kernel combines.
// Nothing of the n x n score matrix leaves the SM. Every mbarrier wait is
// bounded in time; on expiry the CTA sets an error bit, drains its own
// copies and MMAs, frees its TMEM and returns.
//
// Exactness. Row i keeps every key (but itself) that scores at most s+.
// The rerank kernel computes the canonical FP32 distance of every
// candidate, takes the k smallest (w, id), and certifies the row when a
// rigorous bound on the score error proves that no unkept point can have a
// canonical distance <= the k-th. Uncertified rows are recomputed by the
// FP32 SIMT tiles, so the output equals the exact brute-force kNN.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "famst_internal.cuh"
#include "mbarrier.cuh"
#include "tcgen05.cuh"
#include "tile_rows.cuh"

namespace famst {
namespace {

constexpr int BM = tile::ROWS;   // query rows per CTA (TMEM lanes)
constexpr int BN = tile::KEYS;   // keys per tile (accumulator columns)
constexpr int BK = TC_BK;        // K elements per stage (one 128-byte swizzle atom)
constexpr int A_BLOCK = BM * BK * 2;   // 16 KB
constexpr int B_BLOCK = BN * BK * 2;   // 32 KB
constexpr int CAP = TC_CAND_CAP; // candidates kept per row; a row with more is not certified
constexpr int EPI = 16;          // epilogue warps
constexpr int LOG_CAP = 256;     // log entries per thread; compacted beyond LOG_CAP - 64
constexpr size_t LOG_SLOT = size_t(4) * BM * LOG_CAP;   // entries of one CTA's scratch area
// scratch areas of a launch of nctas CTAs, of which one per SM is resident
inline int log_slots(int64_t nctas, int num_sms) { return int(std::min<int64_t>(nctas, num_sms)); }
// Most work items of a pass: the query tiles, with pruned lists' parts (each of
// more than PRUNE_SPLIT_MIN / 2 key tiles, so that small clouds have none).
inline int64_t max_items(int64_t nq_tiles, int64_t nk_tiles, bool prune) {
    if (!prune) return nq_tiles;
    const int64_t parts = (nk_tiles + PRUNE_SPLIT_MIN - 1) / PRUNE_SPLIT_MIN;
    return std::min(nq_tiles + PRUNE_SPLIT_SLOTS, nq_tiles * std::max<int64_t>(1, parts));
}
constexpr int TC_THREADS = 64 + 32 * EPI;
constexpr int VISITED_ROWS_SHARE = 32;   // uncertified rows redone one by one: up to n / this

// Instruction descriptor, kind::f8f6f4: D F32, A/B E4M3 (format 0), both K-major.
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N) {
    return (1u << 4) | (uint32_t(N >> 3) << 17) | (uint32_t(M >> 4) << 24);
}
// D[tmem] (+)= A[smem] * B[smem]^T, kind::f8f6f4 (E4M3 inputs, FP32 accumulate;
// K = 32 per instruction, 32 bytes of each K-major row as for kind::f16)
__device__ __forceinline__ void umma_f8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                        uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// A row keeps the keys up to its k-th plus what the certificate loses to the
// score's error, eps_dot |x||y|max + eps_row (|x| + |y|max)^2: that is the
// fewest that a row can be certified with, and what it takes where the errors
// are large. (A fixed 4 R keys cost the re-rank 31 to 50 distances a row
// instead of about k + 3: 10.5 against 12.9 ms for 256 clouds of 500 to 20,000
// points at k = 16; and rows whose margin held more were redone exactly.)
struct Select {
    int k, cap;
    float eps_dot, eps_row;
};
// count(t): the row's keys that score at most t, of all up to Tr; lo, hi:
// the least and the largest of them. A bound by bisection: with k + 1 or k + 2
// keys at or below it, plus the margin; where that takes in more than cap,
// one with cap - 8 .. cap (or nearly).
template <class Count>
__device__ __forceinline__ float select_bound(Count count, float lo, float hi, float Tr,
                                              const Select &S, float xn, float ym) {
    const float margin = S.eps_dot * xn * ym + S.eps_row * (xn + ym) * (xn + ym);
    int w0 = S.k + 1, w1 = S.k + 2;
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        float l = lo, u = hi;
#pragma unroll 1
        for (int it = 0; it < 10; ++it) {
            const float mid = 0.5f * l + 0.5f * u;
            const int c = count(mid);
            if (c >= w0) {
                u = mid;
                if (c <= w1) break;
            } else {
                l = mid;
            }
        }
        if (pass > 0) return u;
        hi = fminf(u + margin, Tr);
        if (count(hi) <= S.cap) return hi;
        w0 = S.cap - 8;
        w1 = S.cap;
    }
}

struct TcArgs {
    int n;
    int nk_tiles;
    int nkb;        // 64-wide K blocks of the hi part (d_pad / 64)
    int x3;         // hi/lo split on
    int stages;     // B ring depth
    const float *ny;    // key norms ||x'_j||^2, +inf beyond n (nk_tiles * BN entries)
    int32_t *cand;      // n x cap (TOP1: n)
    int32_t *ccnt;      // candidates of the row
    int cap;            // places per row in cand and side_j / side_s (<= CAP)
    Select sel;         // which of them a row keeps
    const unsigned *ymax;   // largest |y| (float bits) of every cloud
    float *splus;       // n
    int *status;
    const TcTile *tiles;  // null: one cloud, CTA b = query tile b over all keys
    const int32_t *colcomp;  // MASK: component of every (padded) row; pairs in one component are skipped
    const int32_t *klist;    // non-null: CTA key tiles are klist[kt0 .. kt1) instead of kt0 .. kt1
    int cross;               // queries and keys are different sets: no self-exclusion
    const float *rscale;     // FP8 operands: per-row scale s (x' ~ s q), query and key rows
                             // alike (keys padded with 1 to nk_tiles * BN entries)
    const float *thr0;       // non-null: per query row, a score every one of its k nearest
                             // keys stays below (T and s+ are capped by it)
    int nitems;              // > 0: work items (query tiles) handed to the CTAs round-robin
                             // (persistent launch, grid <= nitems); 0: one per CTA
    int spiral;              // 1: an item's key tiles [kt0, kt1) are visited outward from the
                             // query tile's own (q0 / BN, then +1, -1, +2, ...)
    const int32_t *nitems_dev;  // non-null (one item per CTA): CTAs from *nitems_dev on are idle
    int32_t *side_j;         // items that are parts of a split list (TcTile::part = s + 1):
    float *side_s;           //   per slot s and tile row, the candidates' ids and scores
    int32_t *side_cnt;       //   (cap each), their number and the part's s+
    float *side_splus;
    int2 *log;               // nslots scratch areas of LOG_SLOT (score bits, id)
    int *claim;              // per area: 0 free, 1 taken by a resident CTA
    int nslots;              // at least as many as CTAs can be resident (one per SM)
};

// packed scores of two columns: ny - 2 acc
__device__ __forceinline__ void scores2(uint32_t d0, uint32_t d1, unsigned long long ny, float &s0,
                                        float &s1) {
    unsigned long long d, r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(d0), "r"(d1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(d), "l"(f2_pack(-2.0f, -2.0f)), "l"(ny));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(s0), "=f"(s1) : "l"(r));
}

// R = 0: top-1 mode (the best key and its score).
template <int R, bool MASK, bool F8 = false>
__global__ void __launch_bounds__(TC_THREADS, 1)
knn_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              TcArgs args) {
    constexpr bool TOP1 = R == 0;
    constexpr int RL = TOP1 ? 1 : R;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte alignment for the swizzle atoms
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // Work items: query tile `item` with its key tiles. A CTA takes items
    // blockIdx.x, blockIdx.x + gridDim.x, ...; TMEM, barriers and the
    // pipeline state carry over from one item to the next.
    // a launch sized for the most items a table can hold: the CTAs beyond
    // the table's count leave before touching barriers or TMEM
    if (args.nitems_dev && int(blockIdx.x) >= __ldg(args.nitems_dev)) return;
    const int nitems = args.nitems > 0 ? args.nitems : int(gridDim.x);
    struct Item {
        int q0, kt0, kt1, nkb, row_end, shift, part, cloud;
    };
    auto item_of = [&](int item) {
        Item I;
        if (args.tiles) {
            const TcTile T = args.tiles[item];
            I.q0 = T.q0; I.kt0 = T.kt0; I.kt1 = T.kt1; I.nkb = T.nkb; I.row_end = T.row_end;
            I.shift = T.shift;
            I.part = T.part; I.cloud = T.cloud;
        } else {
            I.q0 = item * BM; I.kt0 = 0; I.kt1 = args.nk_tiles; I.nkb = args.nkb;
            I.row_end = args.n; I.shift = 0; I.part = 0; I.cloud = 0;
        }
        return I;
    };
    // key tile of the t-th step of an item
    auto ktile = [&](const Item &I, int t) {
        if (args.klist) return __ldg(args.klist + I.kt0 + t);
        if (!args.spiral) return I.kt0 + t;
        const int c0 = min(max(I.q0 / BN, I.kt0), I.kt1 - 1);
        const int L = c0 - I.kt0, Rt = I.kt1 - 1 - c0, m = min(L, Rt);
        if (t <= 2 * m) return (t & 1) ? c0 + ((t + 1) >> 1) : c0 - (t >> 1);
        return Rt > L ? c0 + (t - m) : c0 - (t - m);
    };
    const int nA_max = (args.x3 ? 2 : 1) * args.nkb;  // resident A blocks (widest item)
    unsigned char *sA = base;
    unsigned char *sB = sA + size_t(nA_max) * A_BLOCK;
    float *t_sh = reinterpret_cast<float *>(sB + size_t(args.stages) * B_BLOCK);   // [4][BM]
    int *j_sh = reinterpret_cast<int *>(t_sh + 4 * BM);                            // [4][BM]
    float *f_sh = reinterpret_cast<float *>(j_sh + 4 * BM);       // [EPI][CAP] scores, then
    int *fj_sh = reinterpret_cast<int *>(f_sh + EPI * CAP);       // [EPI][CAP] ids of a row
    uint64_t *bars = reinterpret_cast<uint64_t *>(fj_sh + EPI * CAP);
    uint64_t *full = bars;                       // [stages]
    uint64_t *empty = bars + args.stages;        // [stages]
    uint64_t *a_full = bars + 2 * args.stages;
    uint64_t *tfull = a_full + 1;                // [2]
    uint64_t *tempty = tfull + 2;                // [2]
    uint64_t *mma_done = tempty + 2;
    uint64_t *a_empty = mma_done + 1;            // the A blocks may be overwritten
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(a_empty + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    int *slot_sh = reinterpret_cast<int *>(tmem_slot + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < args.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(a_full, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], EPI);
        }
        mbar_init(mma_done, 1);
        mbar_init(a_empty, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if constexpr (!TOP1) {   // a free scratch area: there are as many as resident CTAs
            int slot = int(blockIdx.x) % args.nslots, tries = 0;
            while (atomicCAS(args.claim + slot, 0, 1) != 0 && ++tries < (1 << 20))
                slot = slot + 1 == args.nslots ? 0 : slot + 1;
            if (tries == 1 << 20) {
                set_status(args.status, STATUS_LOOP_LIMIT);
                slot = -1;
            }
            *slot_sh = slot;
        }
    }
    if constexpr (!TOP1) {
        __syncthreads();
        if (*slot_sh < 0) return;
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
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA))
                         : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB))
                         : "memory");
            int it = 0, a_issued = 0;   // B blocks and A batches issued
            bool ok = true;
            for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
                const Item I = item_of(item);
                // the previous item's MMAs must be done with the A blocks
                if (a_issued > 0 && !mbar_wait(a_empty, (a_issued - 1) & 1, abort_flag,
                                               args.status)) {
                    ok = false;
                    break;
                }
                const int nA = (args.x3 ? 2 : 1) * I.nkb;
                mbar_expect_tx(a_full, uint32_t(nA) * A_BLOCK);
                // resident A blocks: hi blocks 0..nkb-1, then lo blocks (at column
                // block args.nkb + kb of the operand rows)
                for (int a = 0; a < nA; ++a) {
                    const int col = a < I.nkb ? a : args.nkb + (a - I.nkb);
                    tma_load_2d(sA + size_t(a) * A_BLOCK, &tmA, a_full, col * (F8 ? 2 * BK : BK),
                                I.q0);
                }
                ++a_issued;
                const int nkb_tile = args.x3 ? 2 * I.nkb : I.nkb;   // B blocks per key tile
                const int total = (I.kt1 - I.kt0) * nkb_tile;
                for (int j = 0; j < total; ++j, ++it) {
                    const int s = it % args.stages, r = it / args.stages;
                    if (!mbar_wait(&empty[s], (r & 1) ^ 1, abort_flag, args.status)) {
                        ok = false;
                        break;
                    }
                    const int t = ktile(I, j / nkb_tile), blk = j % nkb_tile;
                    // x3 order per key tile: hi_0, lo_0, hi_1, lo_1, ...
                    const int col =
                        args.x3 ? ((blk & 1) ? args.nkb + (blk >> 1) : (blk >> 1)) : blk;
                    mbar_expect_tx(&full[s], B_BLOCK);
                    tma_load_2d(sB + size_t(s) * B_BLOCK, &tmB, &full[s],
                                col * (F8 ? 2 * BK : BK), t * BN);
                }
            }
            // drain: every issued copy must land before the CTA leaves
            if (a_issued > 0) mbar_drain(a_full, (a_issued - 1) & 1);
            for (int s = 0; s < args.stages && s < it; ++s) {
                int last = s + ((it - 1 - s) / args.stages) * args.stages;  // last use of stage s
                mbar_drain(&full[s], (last / args.stages) & 1);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t IDESC = F8 ? idesc_e4m3(BM, BN) : idesc_bf16(BM, BN);
            int it = 0, g = 0, na = 0;   // B blocks, key tiles and items consumed
            bool ok = true;
            for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x, ++na) {
                const Item I = item_of(item);
                if (!mbar_wait(a_full, na & 1, abort_flag, args.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const int nkb_tile = args.x3 ? 2 * I.nkb : I.nkb;
                for (int t = 0; t < I.kt1 - I.kt0 && ok; ++t, ++g) {
                    const int b = g & 1, use = g >> 1;
                    if (!mbar_wait(&tempty[b], (use & 1) ^ 1, abort_flag, args.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d_tmem = tmem + uint32_t(b * BN);
                    uint32_t acc = 0;
                    for (int blk = 0; blk < nkb_tile; ++blk, ++it) {
                        const int s = it % args.stages, r = it / args.stages;
                        if (!mbar_wait(&full[s], r & 1, abort_flag, args.status)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t bsm = smem_u32(sB + size_t(s) * B_BLOCK);
                        const int kb = args.x3 ? (blk >> 1) : blk;
                        const bool is_lo = args.x3 && (blk & 1);
                        // which resident A blocks multiply this B block
                        const int nq = args.x3 ? (is_lo ? 1 : 2) : 1;
                        for (int q = 0; q < nq; ++q) {
                            // hi B block: A_hi then A_lo; lo B block: A_hi
                            const int ablk = (q == 0) ? kb : I.nkb + kb;
                            const uint32_t asm_ = smem_u32(sA + size_t(ablk) * A_BLOCK);
#pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk) {
                                if constexpr (F8)
                                    umma_f8(d_tmem, sdesc_sw128(asm_ + kk * 32),
                                            sdesc_sw128(bsm + kk * 32), IDESC, acc);
                                else
                                    umma_f16(d_tmem, sdesc_sw128(asm_ + kk * 32),
                                             sdesc_sw128(bsm + kk * 32), IDESC, acc);
                                acc = 1;
                            }
                        }
                        umma_commit(&empty[s]);  // stage s is free once these MMAs finish
                    }
                    if (!ok) break;
                    umma_commit(&tfull[b]);      // accumulator b is complete
                }
                if (!ok) break;
                umma_commit(a_empty);            // this item's A blocks are free once done
            }
            umma_commit(mma_done);
            mbar_drain(mma_done, 0);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue
        const float inf = __int_as_float(0x7f800000);
        const int quarter = warp & 3;               // TMEM lanes 32*quarter ..
        const int grp = (warp - 2) >> 2;            // 16-column chunks grp, grp + 4, ...
        const int row = quarter * 32 + lane;
        volatile float *vt_sh = t_sh;
        int2 *area = TOP1 ? nullptr : args.log + size_t(*slot_sh) * LOG_SLOT;
        int2 *my_log = TOP1 ? nullptr : area + size_t(grp * BM + row) * LOG_CAP;
        int g = 0;   // key tiles consumed (accumulator buffer g & 1)
        for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
        const Item I = item_of(item);
        const int i = I.q0 + row;
        const int ntiles = I.kt1 - I.kt0;
        const bool mine = i < I.row_end;
        const float thr0v = (args.thr0 && i < args.n) ? __ldg(args.thr0 + i) : inf;
        // this thread's R smallest scores, ascending (TOP1: the best score)
        float ls[RL];
#pragma unroll
        for (int p = 0; p < RL; ++p) ls[p] = inf;
        int best_j = -1;
        float T = inf;
        int cnt = 0;        // log entries
        bool over = false;  // the log does not hold every key at or below T
        bool ok = true;
        int my_comp = 0;
        if constexpr (MASK) my_comp = __ldg(args.colcomp + i);
        // FP8: acc = q_i . q_j, so x'_i . x'_j ~ s_i s_j acc
        float m2s = -2.0f;
        if constexpr (F8) m2s = -2.0f * (i < args.n ? __ldg(args.rscale + i) : 1.0f);
        auto put = [&](float v) {   // into the sorted list; its largest drops out
#pragma unroll
            for (int p = 0; p < RL; ++p) {
                const float lo = fminf(ls[p], v);
                v = fmaxf(ls[p], v);
                ls[p] = lo;
            }
        };
        auto row_bound = [&]() {   // of the four lists as last published
            return fmaxf(fmaxf(vt_sh[row], vt_sh[BM + row]),
                         fmaxf(vt_sh[2 * BM + row], vt_sh[3 * BM + row]));
        };
        for (int t = 0; t < ntiles; ++t, ++g) {
            const int b = g & 1, use = g >> 1;
            // every lane waits; the warp proceeds only if all lanes saw the phase
            const bool got = mbar_wait(&tfull[b], use & 1, abort_flag, args.status);
            if (!__all_sync(0xffffffffu, got)) {
                ok = false;
                if (!TOP1 && t == 0) epilogue_bar(32 * EPI);   // the others wait there
                break;
            }
            tc_fence_after();
            const uint32_t tb = tmem + (uint32_t(quarter * 32) << 16) + uint32_t(b * BN + 16 * grp);
            const int key0 = ktile(I, t) * BN + 16 * grp;
            // key norms (and components) of this tile's columns straight from
            // global memory: every lane reads the same addresses (L1 broadcast);
            // the next tile's are prefetched into L1 meanwhile
            if (t + 1 < ntiles && lane < 4) {
                const size_t nxt = size_t(ktile(I, t + 1)) * BN + 16 * grp + 64 * lane;
                asm volatile("prefetch.global.L1 [%0];" ::"l"(args.ny + nxt));
                if constexpr (MASK) asm volatile("prefetch.global.L1 [%0];" ::"l"(args.colcomp + nxt));
            }
            // one pass over the tile: the list, the log, or both
            bool lists = true, logs = t > 0;
            auto process = [&](uint32_t(&v)[16], int ch) {
                const int k0 = key0 + 64 * ch;
                float sc[16];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if constexpr (F8) {   // per-key scales, same layout as the norms
                        const float4 nn = __ldg(reinterpret_cast<const float4 *>(args.ny + k0 + 4 * q));
                        const float4 sk =
                            __ldg(reinterpret_cast<const float4 *>(args.rscale + k0 + 4 * q));
                        sc[4 * q + 0] = fmaf(m2s * sk.x, __uint_as_float(v[4 * q + 0]), nn.x);
                        sc[4 * q + 1] = fmaf(m2s * sk.y, __uint_as_float(v[4 * q + 1]), nn.y);
                        sc[4 * q + 2] = fmaf(m2s * sk.z, __uint_as_float(v[4 * q + 2]), nn.z);
                        sc[4 * q + 3] = fmaf(m2s * sk.w, __uint_as_float(v[4 * q + 3]), nn.w);
                    } else {
                        const ulonglong2 nn =
                            __ldg(reinterpret_cast<const ulonglong2 *>(args.ny + k0 + 4 * q));
                        scores2(v[4 * q], v[4 * q + 1], nn.x, sc[4 * q], sc[4 * q + 1]);
                        scores2(v[4 * q + 2], v[4 * q + 3], nn.y, sc[4 * q + 2], sc[4 * q + 3]);
                    }
                    if constexpr (MASK) {  // same component: not a candidate
                        const int4 cc = __ldg(reinterpret_cast<const int4 *>(args.colcomp + k0 + 4 * q));
                        sc[4 * q + 0] = cc.x == my_comp ? inf : sc[4 * q + 0];
                        sc[4 * q + 1] = cc.y == my_comp ? inf : sc[4 * q + 1];
                        sc[4 * q + 2] = cc.z == my_comp ? inf : sc[4 * q + 2];
                        sc[4 * q + 3] = cc.w == my_comp ? inf : sc[4 * q + 3];
                    }
                }
                float mn = inf;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    mn = fminf(mn, fminf(fminf(sc[4 * q], sc[4 * q + 1]),
                                         fminf(sc[4 * q + 2], sc[4 * q + 3])));
                if constexpr (TOP1) {
                    if (mn < ls[0]) {
                        ls[0] = mn;
                        int at = 0;
#pragma unroll
                        for (int c = 15; c >= 0; --c) at = sc[c] == mn ? c : at;
                        best_j = k0 + at;
                    }
                    return;
                }
                // T is at or above this thread's own R-th: a chunk above T
                // changes neither
                if (!__any_sync(0xffffffffu, mn <= T)) return;
                if (!logs) {   // first tile: every score into the list
#pragma unroll 1
                    for (int q = 0; q < 4; ++q) {   // four columns a turn, by select
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            put(q == 0 ? sc[c] : q == 1 ? sc[4 + c] : q == 2 ? sc[8 + c] : sc[12 + c]);
                    }
                } else {   // the scores at or below T into the log, and into the list
                    unsigned bits = 0;
                    if (mn <= T && mine) {
#pragma unroll
                        for (int c = 0; c < 16; ++c)
                            bits |= (sc[c] <= T && sc[c] < inf) ? 1u << c : 0u;
                        if (!args.cross && i >= k0 && i < k0 + 16) bits &= ~(1u << (i - k0));
                    }
                    // (cnt stays below LOG_CAP: at most 64 columns a tile)
#pragma unroll 1
                    while (bits) {
                        const int c = __ffs(bits) - 1;
                        bits &= bits - 1u;
                        float x[8];   // the score of column c, by its bits
#pragma unroll
                        for (int q = 0; q < 8; ++q) x[q] = (c & 1) ? sc[2 * q + 1] : sc[2 * q];
#pragma unroll
                        for (int w = 1; w < 4; ++w)
#pragma unroll
                            for (int q = 0; q < (8 >> w); ++q)
                                x[q] = (c >> w) & 1 ? x[2 * q + 1] : x[2 * q];
                        my_log[cnt] = make_int2(__float_as_int(x[0]), k0 + c);
                        ++cnt;
                        if (lists) put(x[0]);
                    }
                }
                __syncwarp();
            };
            // two 16-column register buffers: the load of chunk c+1 overlaps the
            // processing of chunk c
            auto pass = [&]() {
                uint32_t va[16], vb[16];
                __syncwarp();
                tmem_ld16(tb, va);
#pragma unroll 1
                for (int ch = 0; ch < 4; ch += 2) {
                    tmem_ld_wait16(va);
                    __syncwarp();
                    tmem_ld16(tb + (ch + 1) * 64, vb);
                    process(va, ch);
                    tmem_ld_wait16(vb);
                    __syncwarp();
                    if (ch + 2 < 4) tmem_ld16(tb + (ch + 2) * 64, va);
                    process(vb, ch + 1);
                }
            };
            // (one copy of the pass: the first tile takes a second turn)
#pragma unroll 1
            while (true) {
                pass();
                if (TOP1) break;
                vt_sh[grp * BM + row] = ls[RL - 1];
                if (t == 0 && lists) epilogue_bar(32 * EPI);
                T = fminf(fminf(T, thr0v), row_bound());
                if (t > 0 || !lists) break;
                lists = false;
                logs = true;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
            if (!TOP1 && cnt > LOG_CAP - 64) {   // room for another tile: drop what T has ruled out
                int w = 0;
                for (int e = 0; e < cnt; ++e) {
                    const int2 x = my_log[e];
                    if (__int_as_float(x.x) <= T) my_log[w++] = x;
                }
                cnt = w;
                if (cnt > LOG_CAP - 64) {   // masses of near ties: the row is not certified
                    over = true;
                    cnt = 0;
                }
            }
            __syncwarp();
        }
        // (on a failed item others may still publish their first bounds)
        if constexpr (TOP1) {   // the best of the row's four threads (smaller id on ties)
            t_sh[grp * BM + row] = ls[0];
            j_sh[grp * BM + row] = best_j;
        } else {
            j_sh[grp * BM + row] = over ? -1 : cnt;
        }
        // the logs are complete; a failure anywhere stops every warp here
        const bool failed = epilogue_bar_any(32 * EPI, !ok);
        if constexpr (TOP1) {
            if (!failed && grp == 0 && mine) {
                float s = t_sh[row];
                int j = j_sh[row];
                for (int q = 1; q < 4; ++q) {
                    const float sq = t_sh[q * BM + row];
                    const int jq = j_sh[q * BM + row];
                    if (jq >= 0 && (j < 0 || sq < s || (sq == s && jq < j))) {
                        s = sq;
                        j = jq;
                    }
                }
                args.cand[i - I.shift] = j >= 0 ? j - I.shift : -1;
                args.splus[i - I.shift] = s;
            }
        } else if (!failed) {
            // candidates: this warp's eight rows one after another
            float *fs = f_sh + (warp - 2) * CAP;
            int *fj = fj_sh + (warp - 2) * CAP;
            const float ym = __uint_as_float(__ldg(args.ymax + I.cloud));
#pragma unroll 1
            for (int q = 0; q < BM / EPI; ++q) {
                const int rr = (warp - 2) * (BM / EPI) + q;
                const int ri = I.q0 + rr;
                if (ri >= I.row_end) break;   // warp-uniform
                float Tr = fmaxf(fmaxf(t_sh[rr], t_sh[BM + rr]),
                                 fmaxf(t_sh[2 * BM + rr], t_sh[3 * BM + rr]));
                if (ntiles == 0) Tr = inf;
                if (args.thr0 && ri < args.n) Tr = fminf(Tr, __ldg(args.thr0 + ri));
                bool lost = false;
                int total = 0;
                int2 pre[4][2];   // the first 64 entries of the four logs, in flight together
                int c4[4];
#pragma unroll
                for (int gq = 0; gq < 4; ++gq) {
                    const int c = j_sh[gq * BM + rr];
                    lost |= c < 0;
                    c4[gq] = c < 0 ? 0 : c;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int e = 32 * h + lane;
                        pre[gq][h] = make_int2(0x7f800000, -1);
                        if (e < c4[gq])
                            pre[gq][h] = area[size_t(gq * BM + rr) * LOG_CAP + e];
                    }
                }
                auto keep = [&](int2 x, bool have) {
                    const bool in = have && __int_as_float(x.x) <= Tr;
                    const unsigned m = __ballot_sync(0xffffffffu, in);
                    const int to = total + __popc(m & ((1u << lane) - 1u));
                    if (in && to < CAP) {
                        fs[to] = __int_as_float(x.x);
                        fj[to] = x.y;
                    }
                    total += __popc(m);
                };
#pragma unroll
                for (int gq = 0; gq < 4; ++gq) {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (32 * h < c4[gq]) keep(pre[gq][h], 32 * h + lane < c4[gq]);
#pragma unroll 1
                    for (int e0 = 64; e0 < c4[gq]; e0 += 32) {
                        const bool have = e0 + lane < c4[gq];
                        int2 x = make_int2(0x7f800000, -1);
                        if (have) x = area[size_t(gq * BM + rr) * LOG_CAP + e0 + lane];
                        keep(x, have);
                    }
                }
                lost |= total > CAP;
                const int kept = min(total, CAP);
                __syncwarp();
                float sv[4];
                float lo = inf, hi = -inf;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const bool have = 32 * h + lane < kept;
                    sv[h] = have ? fs[32 * h + lane] : inf;
                    lo = fminf(lo, sv[h]);
                    hi = have ? fmaxf(hi, sv[h]) : hi;
                }
                float sp = Tr;
                if (!lost && kept > args.sel.k + 1) {
#pragma unroll
                    for (int o = 16; o >= 1; o >>= 1) {
                        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                    }
                    auto count = [&](float t) {
                        int c = 0;
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            c += __popc(__ballot_sync(0xffffffffu, sv[h] <= t));
                        return c;
                    };
                    // (all keys up to Tr are in the log)
                    sp = select_bound(count, lo, hi, Tr, args.sel, sqrtf(__ldg(args.ny + ri)), ym);
                }
                // out: the candidates at or below sp
                const tile::RowSlot slot = tile::row_slot(I.q0, rr, I.shift, I.part);
                const size_t at0 = slot.at * size_t(args.cap);
                int out = 0;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const bool in = 32 * h + lane < kept && sv[h] <= sp;
                    const unsigned m = __ballot_sync(0xffffffffu, in);
                    const int to_row = out + __popc(m & ((1u << lane) - 1u));
                    if (in && to_row < args.cap) {
                        const size_t to = at0 + to_row;
                        const int j = fj[32 * h + lane] - I.shift;
                        if (slot.side) {
                            args.side_j[to] = j;
                            args.side_s[to] = sv[h];
                        } else {
                            args.cand[to] = j;
                        }
                    }
                    out += __popc(m);
                }
                if (out > args.cap) {   // ties at the bound
                    lost = true;
                    out = args.cap;
                }
                if (lane == 0) {
                    if (lost) sp = -inf;   // never certified
                    (slot.side ? args.side_cnt : args.ccnt)[slot.at] = out;
                    (slot.side ? args.side_splus : args.splus)[slot.at] = sp;
                }
                __syncwarp();
            }
        }
        // the next item reuses the logs, the counts and the bounds
        epilogue_bar(32 * EPI);
        if (failed) break;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    if constexpr (!TOP1) {
        if (threadIdx.x == 0) {
            __threadfence();
            atomicExch(args.claim + *slot_sh, 0);
        }
    }
}

// A row's candidates and bound as the kernels behind the tiles take them. A CTA
// that gives up (a bounded wait ran out, or no scratch area was free) leaves its
// rows unset and the status word says so: then no row has candidates, or a bound
// that certifies. (Written by the tile kernel itself, 20 lines behind its loops,
// this cost registers in them: 16 to 40 bytes of spills, 1.6 % of 256 clouds'
// build.) The pivots of such a top-1 pass may be anything; their reader takes
// what is no pivot as pivot 0.
__device__ __forceinline__ void row_result(const int *__restrict__ status,
                                           const int32_t *__restrict__ ccnt,
                                           const float *__restrict__ splus, int64_t r, int &cnt,
                                           float &sp) {
    cnt = ccnt[r];
    sp = splus[r];
    if (__ldg(status) & STATUS_LOOP_LIMIT)
        tile::give_up_row(tile::RowSlot{false, 0}, &cnt, &sp, nullptr, nullptr);
}

// Rows of split query tiles (a warp per row, blockIdx.y = 16 rows of split
// tile blockIdx.x): s+ = the smallest of the parts' s+ (every key of the
// others at or below it is among their candidates), lowered like a whole
// list's; candidates = the parts' candidates at or below it.
__global__ void __launch_bounds__(512)
split_merge_kernel(const int32_t *__restrict__ splitq, const int32_t *__restrict__ nsplit,
                   const int32_t *__restrict__ side_j, const float *__restrict__ side_s,
                   const int32_t *__restrict__ side_cnt, const float *__restrict__ side_splus,
                   int64_t n, Select sel, const float *__restrict__ ny,
                   const unsigned *__restrict__ ymax, int32_t *__restrict__ cand,
                   int32_t *__restrict__ ccnt, float *__restrict__ splus,
                   const int *__restrict__ status) {
    if (int(blockIdx.x) >= __ldg(nsplit)) return;
    if (__ldg(status) & STATUS_LOOP_LIMIT) return;   // (row_result)
    const int q = splitq[3 * blockIdx.x], slot0 = splitq[3 * blockIdx.x + 1];
    const int P = splitq[3 * blockIdx.x + 2];
    const int row = int(blockIdx.y) * 16 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int64_t i = int64_t(q) * BM + row;
    if (i >= n) return;
    const float inf = __int_as_float(0x7f800000);
    float T = inf;
    for (int p = lane; p < P; p += 32) T = fminf(T, side_splus[size_t(slot0 + p) * BM + row]);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) T = fminf(T, __shfl_xor_sync(0xffffffffu, T, o));
    const int cap = sel.cap;
    float lo = inf, hi = -inf;
    int have = 0;   // candidates of the parts up to T
    for (int p = 0; p < P; ++p) {
        const size_t at = size_t(slot0 + p) * BM + row;
        const int c = side_cnt[at];   // <= cap
        for (int e = lane; e < c; e += 32) {
            const float s = side_s[at * cap + e];
            if (s <= T) {
                lo = fminf(lo, s);
                hi = fmaxf(hi, s);
                ++have;
            }
        }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        have += __shfl_xor_sync(0xffffffffu, have, o);
    }
    if (have > sel.k + 1) {
        auto count = [&](float t) {
            int c = 0;
            for (int p = 0; p < P; ++p) {
                const size_t at = size_t(slot0 + p) * BM + row;
                const int cp = side_cnt[at];
                for (int e0 = 0; e0 < cp; e0 += 32)
                    c += __popc(__ballot_sync(
                        0xffffffffu, e0 + lane < cp && side_s[at * cap + e0 + lane] <= t));
            }
            return c;
        };
        T = select_bound(count, lo, hi, T, sel, sqrtf(ny[i]), __uint_as_float(*ymax));
    }
    int total = 0;
    for (int p = 0; p < P; ++p) {
        const size_t at = size_t(slot0 + p) * BM + row;
        const int c = side_cnt[at];
        for (int e0 = 0; e0 < c; e0 += 32) {
            const int e = e0 + lane;
            const bool in = e < c && side_s[at * cap + e] <= T;
            const unsigned m = __ballot_sync(0xffffffffu, in);
            const int to = total + __popc(m & ((1u << lane) - 1u));
            if (in && to < cap) cand[i * cap + to] = side_j[at * cap + e];
            total += __popc(m);
        }
    }
    if (lane == 0) {
        ccnt[i] = total < cap ? total : cap;
        splus[i] = total <= cap ? T : -inf;   // more ties than places: not certified
    }
}

// ------------------------------------------------------------- prep

// per-block column sums (double) over a contiguous range of rows
// (the rows in order, eight loads in flight per thread)
__global__ void colsum_partial_kernel(const float *__restrict__ X, int64_t n, int d, int rows_per,
                                      double *__restrict__ part) {
    int64_t r0 = int64_t(blockIdx.x) * rows_per;
    int64_t r1 = r0 + rows_per < n ? r0 + rows_per : n;
    // FP32 sums within the block's rows (the FP64 pipe is slow on this GPU,
    // and the centre only has to be some fixed point near the data: every
    // bound downstream holds for any centre), FP64 across blocks
    for (int c = threadIdx.x; c < d; c += blockDim.x) {
        float s = 0.0f;
        int64_t r = r0;
        for (; r + 8 <= r1; r += 8) {
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = __ldg(X + (r + q) * d + c);
#pragma unroll
            for (int q = 0; q < 8; ++q) s += v[q];
        }
        for (; r < r1; ++r) s += __ldg(X + r * d + c);
        part[int64_t(blockIdx.x) * d + c] = double(s);
    }
}

// one block per column: strided partial sums, then a tree in shared memory
__global__ void colsum_final_kernel(const double *__restrict__ part, int nb, int d, int64_t n,
                                    float *__restrict__ mean) {
    __shared__ double red[256];
    const int c = blockIdx.x;
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += 256) s += part[int64_t(b) * d + c];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o >= 1; o >>= 1) {
        if (int(threadIdx.x) < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) mean[c] = float(red[0] / double(n));
}

// One warp per row: centred row, BF16 hi (and lo) operand rows, FP32 norm.
// `scrambled`: operand row and key norm at position p are those of row
// scrambled_row(p) (xnorm stays by row).
__global__ void tc_prep_kernel(const float *__restrict__ X, int64_t n, int d, int d_pad, int x3,
                               int scrambled,
                               const float *__restrict__ mean, __nv_bfloat16 *__restrict__ H,
                               float *__restrict__ ny, float *__restrict__ xnorm,
                               unsigned *__restrict__ ymax_bits) {
    __shared__ unsigned bmax;
    if (threadIdx.x == 0) bmax = 0u;
    __syncthreads();
    const int64_t row = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row < n) {
        const int kh = (x3 ? 2 : 1) * d_pad;
        const int64_t src = scrambled ? tile::scrambled_row(int(row), int(n)) : row;
        __nv_bfloat16 *h = H + row * kh;
        const float *x = X + src * d;
        float acc = 0.0f;
        // four coordinates per lane per step (16-byte rows), else one
        const bool v4 = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
        if (v4) {
            for (int t = 4 * lane; t < d_pad; t += 128) {
                float4 xv = make_float4(0.f, 0.f, 0.f, 0.f);
                if (t < d) {
                    const float4 a = __ldg(reinterpret_cast<const float4 *>(x + t));
                    const float4 m = __ldg(reinterpret_cast<const float4 *>(mean + t));
                    xv = make_float4(__fsub_rn(a.x, m.x), __fsub_rn(a.y, m.y), __fsub_rn(a.z, m.z),
                                     __fsub_rn(a.w, m.w));
                }
                const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
                __nv_bfloat16 hi[4], lo[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    hi[q] = __float2bfloat16_rn(xs[q]);
                    lo[q] = __float2bfloat16_rn(__fsub_rn(xs[q], __bfloat162float(hi[q])));
                    acc = fmaf(xs[q], xs[q], acc);
                }
                *reinterpret_cast<uint2 *>(h + t) = *reinterpret_cast<const uint2 *>(hi);
                if (x3) *reinterpret_cast<uint2 *>(h + d_pad + t) = *reinterpret_cast<const uint2 *>(lo);
            }
        } else {
            for (int t = lane; t < d_pad; t += 32) {
                float xc = t < d ? __fsub_rn(x[t], mean[t]) : 0.0f;
                __nv_bfloat16 hi = __float2bfloat16_rn(xc);
                h[t] = hi;
                if (x3) h[d_pad + t] = __float2bfloat16_rn(__fsub_rn(xc, __bfloat162float(hi)));
                acc = fmaf(xc, xc, acc);
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) {
            ny[row] = acc;
            xnorm[src] = acc;
            atomicMax(&bmax, __float_as_uint(sqrtf(acc)));   // one global atomic per block
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && bmax != 0u) atomicMax(ymax_bits, bmax);
}

// One warp per row, FP8 operands: centred row x' = fl(x - mean), scale
// s = 2^e with e the smallest integer such that max |x'| <= 448 s (the
// largest finite E4M3), q = e4m3(x' / s) rounded to nearest (the division by
// a power of two is exact), FP32 norm ||x'||^2 as for the BF16 operands.
// Rows of d_pad bytes, zero beyond d.
__global__ void tc_prep_f8_kernel(const float *__restrict__ X, int64_t n, int d, int d_pad, int scrambled,
                                  const float *__restrict__ mean, uint8_t *__restrict__ Q,
                                  float *__restrict__ rscale, float *__restrict__ ny,
                                  float *__restrict__ xnorm, unsigned *__restrict__ ymax_bits) {
    __shared__ unsigned bmax;
    if (threadIdx.x == 0) bmax = 0u;
    __syncthreads();
    const int64_t row = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row < n) {
        const int64_t src = scrambled ? tile::scrambled_row(int(row), int(n)) : row;
        const float *x = X + src * d;
        float amax = 0.0f, acc = 0.0f;
        for (int t = lane; t < d; t += 32) {
            const float xc = __fsub_rn(__ldg(x + t), __ldg(mean + t));
            amax = fmaxf(amax, fabsf(xc));
            acc = fmaf(xc, xc, acc);
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            acc += __shfl_xor_sync(0xffffffffu, acc, o);
        }
        // smallest e with amax <= 448 2^e (so 2^e < 2 amax / 448), kept to
        // normal FP32 scales; the quotient's rounding is corrected by the
        // exact comparisons with 448 2^e
        int e = 0;
        if (amax > 0.0f) {
            frexpf(amax / 448.0f, &e);   // amax / 448 = f 2^e, 0.5 <= f < 1
            while (e > -126 && ldexpf(448.0f, e - 1) >= amax) e -= 1;
            while (e < 127 && ldexpf(448.0f, e) < amax) e += 1;
        }
        const float sc = ldexpf(1.0f, e);
        uint8_t *q = Q + row * d_pad;
        for (int t = lane; t < d_pad; t += 32) {
            const float xc = t < d ? __fsub_rn(__ldg(x + t), __ldg(mean + t)) : 0.0f;
            q[t] = uint8_t(__nv_cvt_float_to_fp8(ldexpf(xc, -e), __NV_SATFINITE, __NV_E4M3));
        }
        if (lane == 0) {
            rscale[row] = sc;
            ny[row] = acc;
            xnorm[src] = acc;
            atomicMax(&bmax, __float_as_uint(sqrtf(acc)));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && bmax != 0u) atomicMax(ymax_bits, bmax);
}

__global__ void fill_value_kernel(float *p, int64_t from, int64_t to, float v) {
    int64_t i = from + int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < to) p[i] = v;
}

__global__ void fill_inf_kernel(float *p, int64_t from, int64_t to) {
    int64_t i = from + int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < to) p[i] = __int_as_float(0x7f800000);
}

// components over the (scrambled) padded rows, -1 beyond n
__global__ void pad_components_kernel(const int32_t *__restrict__ comp, int64_t n, int64_t npad,
                                      int32_t *__restrict__ cpad) {
    const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (p < npad) cpad[p] = p < n ? comp[tile::scrambled_row(int(p), int(n))] : -1;
}

// Start threshold of the pruned tiles' lists: every key y within tau_r of
// row r (tau_r bounds r's k-th neighbour distance from above) has a tile
// score s~(y) = ||y'||^2 - 2 x'.y' (rounded) with s~ <= ||x' - y'||^2 -
// ||x'||^2 + E <= (tau_r + c)^2 - xn2 (1 - (d+1) u) + E, where c bounds the
// centring rounding and E the tile's score error (the certificate's terms).
__global__ void thr0_kernel(const float *__restrict__ tau_row, const float *__restrict__ xn2s,
                            int64_t n, int d, const unsigned *__restrict__ ymax_bits,
                            double eps_dot, float *__restrict__ thr0) {
    const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const double u24 = 1.0 / 16777216.0;
    const double xn2 = double(xn2s[r]), xn = sqrt(xn2);
    const double ym = double(__uint_as_float(*ymax_bits));
    const double E = 2.0 * eps_dot * xn * ym * 1.01 + (d + 1) * u24 * 1.02 * ym * ym +
                     2.0 * u24 * (ym * ym + 2.0 * xn * ym) * 1.01 + 1e-30;
    const double t = (double(tau_row[r]) + 1.02 * u24 * (xn + ym)) * (1.0 + 0x1p-20);
    const double thr = t * t - xn2 * (1.0 - (d + 1) * u24 * 1.02) + E;
    thr0[r] = __double2float_ru(thr + (thr >= 0.0 ? thr : -thr) * 0x1p-20 + 1e-30);
}

// ------------------------------------------------------------- rerank

// relative error of the tensor-core dot of BF16 operands, split (x3) or not:
// products and accumulation over the padded columns
__host__ __device__ inline double tc_eps_dot(int d_pad, bool x3) {
    const double u8 = 1.0 / 256.0;
    const double kprod = double(x3 ? 3 * d_pad : d_pad);
    return (x3 ? (3.0 * u8 * u8 + 3.0 * u8 * u8 * u8 + u8 * u8 * u8 * u8)
               : (2.0 * u8 + u8 * u8)) +
           kprod * (1.0 / 4194304.0) * (1.0 + 4.0 * u8);
}
// the FP32 terms (norms, score rounding, canonical distance on both sides)
inline float score_eps_row(int d) { return float(4.0 * (d + 8.0) / 16777216.0); }

struct CertConst {
    double eps_dot;   // relative error of the tensor-core dot (products + accumulation)
    float e32, c32, w32;   // 2.02 eps_dot and (d + 1) u 1.02 rounded up, 1 - (d + 4) u 1.05 down
};
inline CertConst cert_const(double eps_dot, int d) {
    const double u = 1.0 / 16777216.0, up = 1.0 + 0x1p-22;
    return CertConst{eps_dot, float(2.02 * eps_dot * up), float((d + 1) * u * 1.02 * up),
                     float((1.0 - (d + 4.0) * u * 1.05) * (1.0 - 0x1p-22))};
}

// Largest |y| of a cloud whose scores are all finite: beyond it a key's squared
// norm may leave the FP32 range, its score is +inf or NaN, and the tiles neither
// keep nor count it. The distances between pivots are then no lower bounds either
// (a square beyond the range makes one +inf), and no tile is pruned.
constexpr float NORM_MAX = 1e18f;

// Whether no key left out can be at a canonical distance <= kw: keys of
// skipped tiles lie at a true distance >= skip, other keys left out have a
// score above sp. First in FP32 with every rounding on the safe side, which
// decides all but near ties; then in FP64. (The FP64 form alone, some sixty
// operations with two square roots in every warp at this GPU's two FP64
// lanes per SM and clock, held the re-rank back: 10.4 -> 6.6 ms
// for 256 clouds of 500 to 20,000 points.)
template <class Eps64>
__device__ __forceinline__ bool certified(float kw, float skip, float sp, float xn2f, float ymf,
                                          int d, const CertConst &cc, Eps64 eps64) {
    const float inf = __int_as_float(0x7f800000);
    if (!(ymf < NORM_MAX)) return false;
    {
        const float u = 0x1p-24f;
        const float xn = __fsqrt_ru(xn2f), xy = __fmul_ru(xn, ymf), yy = __fmul_ru(ymf, ymf);
        // the terms of the FP64 form below, each rounded up
        const float E = __fadd_ru(
            __fadd_ru(__fmul_ru(cc.e32, xy), __fmul_ru(cc.c32, yy)),
            __fadd_ru(__fmul_ru(2.03f * u, __fadd_ru(yy, __fmul_ru(2.0f, xy))), 1.1e-30f));
        const float p = __fsub_rd(__fadd_rd(xn2f, sp), __fadd_ru(E, __fmul_ru(cc.c32, xn2f)));
        const float lo = __fsub_rd(p > 0.0f ? __fsqrt_rd(p) : 0.0f,
                                   __fmul_ru(1.03f * u, __fadd_ru(xn, ymf)));
        const bool skip_ok = !(skip < inf) || __fmul_rd(skip, cc.w32) > kw;
        if (skip_ok && (!(sp < inf) || (lo > 0.0f && __fmul_rd(lo, cc.w32) > kw))) return true;
    }
    const double u24 = 1.0 / 16777216.0;
    // their canonical distance is above kw when skip (1 - eps_canon) is
    if (skip < inf && !(double(skip) * (1.0 - (d + 4.0) * u24 * 1.05) > double(kw))) return false;
    if (!(sp < inf)) return true;   // no bound: every visited key was kept
    const double xn2 = double(xn2f);
    const double xn = sqrt(xn2);
    const double ym = double(ymf);
    // |s~ - s| <= E: tensor-core dot, FP32 key norm, score rounding
    const double E = 2.0 * eps64() * xn * ym * 1.01 + (d + 1) * u24 * 1.02 * ym * ym +
                     2.0 * u24 * (ym * ym + 2.0 * xn * ym) * 1.01 + 1e-30;
    // lower bound on the centred squared distance of any unkept point
    const double p_lo = xn2 * (1.0 - (d + 1) * u24 * 1.02) + double(sp) - E;
    const double dist_lo =
        (p_lo > 0.0 ? sqrt(p_lo) : 0.0) - 1.02 * u24 * (xn + ym);  // centring rounding
    const double w_lo = dist_lo * (1.0 - (d + 4.0) * u24 * 1.05);  // canonical FP32 error
    return w_lo > double(kw);
}

// One warp per row: canonical distances of its cnt candidates, bitonic sort
// of (w, id), top k, certificate (sp: every key left out scored above it).
// Row i's point is xi; row_of(candidate id) is a row of X (row stride ld, chain length dc >= d: columns beyond d are zero
// and leave the canonical distance unchanged). d is the true dimension used in
// the error bounds. Returns whether the row was certified (then the k
// results are written).
// XR > 0 (dc <= 32 XR): lane l takes coordinates l, l + 32, ... (its
// canonical partial) of every candidate from coalesced row reads, the query
// row held in registers, and the warp sums the partials of a batch of
// candidates at once (below); XR = 0: one candidate per lane, its 32
// partials in registers. H: a list holds at most 32 H <= CAP candidates.
// Bound: issue slots (a candidate's 4 loads, 8 FP32 operations and 3 shuffles
// per lane at d = 128) at 68 % of peak. With about k + 3 candidates instead of
// 4 R - 1, half batches, and the certificate's FP64 out of the common way: 1M
// rows at k = 32 3.45 -> 2.59 ms, 256 clouds (2.6M rows, k = 16) 8.4 -> 6.6 ms.
template <int XR, int H, class Eps64, class RowOf>
__device__ __forceinline__ bool rerank_row(const float *__restrict__ X, int ld, int dc, int d,
                                           const float *__restrict__ xi, int k,
                                           const int32_t *__restrict__ cand_row, int cnt, float sp,
                                           float skip, float xn2f, float ymf,
                                           const CertConst &cc, Eps64 eps64, RowOf row_of, int lane,
                                           int32_t *__restrict__ nbr_row,
                                           float *__restrict__ dist_row,
                                           const int32_t *__restrict__ idmap = nullptr,
                                           uint64_t *kth_out = nullptr) {
    const int kp = cnt;   // <= 32 H
    uint64_t key[H];
    int jc[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        key[h] = KEY_NONE;
        const int c = h * 32 + lane;
        jc[h] = c < kp ? row_of(cand_row[c]) : -1;
    }
    if constexpr (XR > 0) {
        // batches of NB candidates: lane l's partial of candidate c in
        // acc[c mod NB]; the butterfly's steps xor 16 .. xor NB on all NB,
        // then its later steps (xor NB/2 .. 1) transposed, each lane passing
        // on the half it does not keep. The additions are the butterfly's
        // own (same pairs, same order), so lane l ends with the canonical
        // total of candidate NB b + (l mod NB), with 2 NB - 1 + NB log2(32/NB)
        // shuffles per batch instead of 5 NB.
        // (wider rows take smaller batches, within the sorted kernel's
        // register budget; NB = 1 is the plain butterfly)
        constexpr int NB = XR <= 4 ? 16 : (XR <= 8 ? 2 : 1);
        constexpr int G = XR <= 8 ? 2 : 1;   // candidates with loads in flight
        constexpr int PB = NB == 16 ? 8 : NB;   // a whole or half batch
        static_assert(PB % G == 0, "a part is whole load groups");
        float xr[XR];
#pragma unroll
        for (int q = 0; q < XR; ++q) {
            const int t = lane + 32 * q;
            xr[q] = t < dc ? __ldg(xi + t) : 0.0f;
        }
#pragma unroll 1
        for (int b = 0; b < (kp + NB - 1) / NB; ++b) {
            const int hb = (NB * b) >> 5;   // a batch lies in one register of the list
            int jb = jc[0];
#pragma unroll
            for (int h = 1; h < H; ++h) jb = hb == h ? jc[h] : jb;
            float acc[NB];
            auto part = [&](auto first) {   // candidates first .. first + PB - 1 of the batch
#pragma unroll
                for (int g1 = 0; g1 < PB; g1 += G) {
                    const int g0 = first.value + g1;
                    int j[G];
                    float y[G][XR];
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        j[g] = __shfl_sync(0xffffffffu, jb, (NB * b + g0 + g) & 31);
#pragma unroll
                        for (int q = 0; q < XR; ++q) {
                            const int t = lane + 32 * q;
                            y[g][q] =
                                (j[g] >= 0 && t < dc) ? __ldg(X + int64_t(j[g]) * ld + t) : 0.0f;
                        }
                    }
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        float p = 0.0f;
#pragma unroll
                        for (int q = 0; q < XR; ++q) {
                            const float dl = __fsub_rn(xr[q], y[g][q]);
                            p = __fmaf_rn(dl, dl, p);
                        }
                        acc[g0 + g] = p;
                    }
                }
            };
            part(std::integral_constant<int, 0>{});
            if constexpr (NB > PB) {   // the last batch's second half is often empty
                if (kp - NB * b > PB) {
                    part(std::integral_constant<int, PB>{});
                } else {
#pragma unroll
                    for (int i = PB; i < NB; ++i) acc[i] = 0.0f;
                }
            }
#pragma unroll
            for (int o = 16; o >= NB; o >>= 1)
#pragma unroll
                for (int i = 0; i < NB; ++i)
                    acc[i] = __fadd_rn(acc[i], __shfl_xor_sync(0xffffffffu, acc[i], o));
#pragma unroll
            for (int o = NB / 2; o >= 1; o >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < o; ++i) {
                    const float send = up ? acc[i] : acc[i + o];
                    const float keep = up ? acc[i + o] : acc[i];
                    acc[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, o));
                }
            }
            // candidate c of this lane; sort element c (register c / 32 of
            // lane c mod 32) takes it from the lane of the matching block
            const int c = NB * b + (lane & (NB - 1));
            const int jl = __shfl_sync(0xffffffffu, jb, c & 31);
            if ((lane & ~(NB - 1)) == ((NB * b) & 31) && jl >= 0) {
                const uint64_t kg = nb_key(__fsqrt_rn(acc[0]), uint32_t(idmap ? idmap[jl] : jl));
#pragma unroll
                for (int h = 0; h < H; ++h)
                    if (h == hb) key[h] = kg;
            }
        }
    } else {
#pragma unroll
        for (int h = 0; h < H; ++h)
            if (jc[h] >= 0)
                key[h] = nb_key(canon_dist<1>(xi, X + int64_t(jc[h]) * ld, dc),
                                uint32_t(idmap ? idmap[jc[h]] : jc[h]));
    }
    // sort by (w, id), as many registers as the candidates fill
    if (kp <= 32) {
        uint64_t one[1] = {key[0]};
        warp_sort_regs<1>(one, lane);
        key[0] = one[0];
    } else {
        warp_sort_regs<H>(key, lane);
    }
    // k-th key (index k-1)
    const int kh = (k - 1) >> 5, kl = (k - 1) & 31;   // k <= 63
    const uint64_t kth = __shfl_sync(0xffffffffu, kh ? key[1] : key[0], kl);
    if (kth_out) *kth_out = kth;
    const bool cert = certified(key_w(kth), skip, sp, xn2f, ymf, d, cc, eps64);   // warp-uniform
    if (cert) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int idx = h * 32 + lane;
            if (idx < k) {
                nbr_row[idx] = int32_t(key_lo(key[h]));
                dist_row[idx] = key_w(key[h]);
            }
        }
    }
    return cert;
}

// Position r of an unpruned pass (rows as they are, or scrambled).
template <int XR, int H>
__global__ void rerank_kernel(const float *__restrict__ X, int64_t n, int d, int k, int scrambled,
                              const int32_t *__restrict__ cand, const int32_t *__restrict__ ccnt,
                              const float *__restrict__ splus, const float *__restrict__ xnorm2, const unsigned *__restrict__ ymax_bits,
                              CertConst cc, const int *__restrict__ status,
                              int32_t *__restrict__ nbr, float *__restrict__ dist,
                              int32_t *__restrict__ fail_rows, int32_t *__restrict__ fail_count) {
    const int64_t r = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (r >= n) return;
    auto row_of = [&](int p) { return scrambled ? tile::scrambled_row(p, int(n)) : p; };
    const int64_t i = row_of(int(r));
    int cnt;
    float sp;
    row_result(status, ccnt, splus, r, cnt, sp);
    bool cert = rerank_row<XR, H>(X, d, d, d, X + i * d, k, cand + r * (32 * H), cnt, sp,
                                    __int_as_float(0x7f800000), xnorm2[i], __uint_as_float(*ymax_bits),
                                    cc, [&] { return cc.eps_dot; }, row_of, lane, nbr + i * k, dist + i * k);
    if (!cert && lane == 0) fail_rows[atomicAdd(fail_count, 1)] = int32_t(i);
}

// Re-rank in the pruning's cell order: sorted row r is point i = perm[r];
// candidate rows are read from the sorted copy Xs (a row's candidates are
// mostly cell-mates, so they sit close together in memory), keyed and
// written with their original ids.
template <int XR, int H>
__global__ void __launch_bounds__(256, H == 2 ? 5 : 3)
rerank_sorted_kernel(const float *__restrict__ Xs, int64_t n, int d, int k,
                                     const int32_t *__restrict__ cand,
                                     const int32_t *__restrict__ ccnt,
                                     const float *__restrict__ splus,
                                     const float *__restrict__ skipQ,
                                     const int32_t *__restrict__ perm,
                                     const float *__restrict__ xnorm2,
                                     const unsigned *__restrict__ ymax_bits, CertConst cc,
                                     const int *__restrict__ status,
                                     int32_t *__restrict__ nbr, float *__restrict__ dist,
                                     int32_t *__restrict__ fail_rows,
                                     uint64_t *__restrict__ fail_kth,
                                     int32_t *__restrict__ fail_count) {
    const int64_t r = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const int64_t i = perm[r];
    uint64_t kth;
    int cnt;
    float sp;
    row_result(status, ccnt, splus, r, cnt, sp);
    const bool cert = rerank_row<XR, H>(Xs, d, d, d, Xs + r * d, k, cand + r * (32 * H), cnt, sp,
                                          skipQ[r / BM], xnorm2[i],
                                          __uint_as_float(*ymax_bits), cc, [&] { return cc.eps_dot; },
                                          [](int p) { return p; }, lane, nbr + i * k, dist + i * k,
                                          perm, &kth);
    if (!cert && lane == 0) {
        const int s = atomicAdd(fail_count, 1);
        fail_rows[s] = int32_t(r);   // the position in the cell order
        fail_kth[s] = kth;
    }
}

__device__ __forceinline__ int cloud_of(const long long *__restrict__ off, int B, long long v) {
    int lo = 0, hi = B;  // off[lo] <= v < off[hi]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (off[mid] <= v) lo = mid; else hi = mid;
    }
    return lo;
}

// Batched re-rank: one warp per compact row of a cloud that used the tensor
// tiles. Xc holds the clouds' rows back to back with row stride ld (zero
// beyond each cloud's d).
// perm (may be null): the rows are in a spatial order within each cloud and
// perm[v] is the compact id of row v; candidate ids are mapped through it
// and the results written at the original row.
template <int XR, int H>
__global__ void __launch_bounds__(256, H == 2 ? 4 : 3)
rerank_batched_kernel(const float *__restrict__ Xc, int ld, int64_t N,
                                      const long long *__restrict__ voff, int B,
                                      const CloudDev *__restrict__ cl, int x3, int k,
                                      const int32_t *__restrict__ cand,
                                      const int32_t *__restrict__ ccnt,
                                      const float *__restrict__ splus,
                                      const float *__restrict__ xnorm2,
                                      const unsigned *__restrict__ ymax_bits, CertConst cc,
                                      const int *__restrict__ status,
                                      const int32_t *__restrict__ perm,
                                      int32_t *__restrict__ nbr, float *__restrict__ dist,
                                      int32_t *__restrict__ fail_rows,
                                      int32_t *__restrict__ fail_count) {
    int64_t v = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (v >= N) return;
    const int b = cloud_of(voff, B, v);
    const CloudDev c = cl[b];
    if (!c.use_tc) return;
    const int dc = (c.d + 3) & ~3;
    const int64_t pv = perm ? int64_t(perm[v]) : v;
    int cnt;
    float sp;
    row_result(status, ccnt, splus, v, cnt, sp);
    bool cert = rerank_row<XR, H>(Xc, ld, dc, c.d, Xc + v * ld, k, cand + v * (32 * H), cnt, sp,
                                  __int_as_float(0x7f800000),
                                  xnorm2[v], __uint_as_float(ymax_bits[b]), cc,
                                  [&] { return tc_eps_dot(c.d_pad, x3); },
                                  [](int p) { return p; }, lane, nbr + pv * k, dist + pv * k, perm);
    if (!cert && lane == 0) fail_rows[atomicAdd(fail_count, 1)] = int32_t(pv);
}

// Exact kNN of single rows by brute force within their cloud: one warp per
// listed row (the count lives on the device); lane l scans keys l, l+32, ...
// with canonical distances and keeps its k best (w, id) in shared memory;
// the warp then merges the 32 sorted lists. k <= 64.
constexpr int FB_WARPS = 2;  // 32 KB of static shared lists per block
__global__ void fallback_rows_kernel(const float *__restrict__ Xc, int ld,
                                     const long long *__restrict__ voff, int B,
                                     const CloudDev *__restrict__ cl, int k,
                                     const int32_t *__restrict__ rows,
                                     const int32_t *__restrict__ count,
                                     int32_t *__restrict__ nbr, float *__restrict__ dist) {
    __shared__ uint64_t lists[FB_WARPS][64][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nrows = *count;
    for (int64_t q = int64_t(blockIdx.x) * FB_WARPS + w; q < nrows;
         q += int64_t(gridDim.x) * FB_WARPS) {
        const int64_t v = rows[q];
        const int b = cloud_of(voff, B, v);
        const CloudDev c = cl[b];
        const int dc = (c.d + 3) & ~3;
        const float *xi = Xc + v * ld;
        int have = 0;
        uint64_t kth = KEY_NONE;
        for (int64_t j = c.voff + lane; j < c.voff + c.n; j += 32) {
            if (j == v) continue;
            uint64_t key = nb_key(canon_dist<4>(xi, Xc + j * ld, dc), uint32_t(j));
            if (key >= kth) continue;
            int pos = have < k ? have++ : k - 1;
            while (pos > 0 && lists[w][pos - 1][lane] > key) {
                lists[w][pos][lane] = lists[w][pos - 1][lane];
                --pos;
            }
            lists[w][pos][lane] = key;
            if (have == k) kth = lists[w][k - 1][lane];
        }
        __syncwarp();
        int head = 0;
        for (int o = 0; o < k; ++o) {
            uint64_t mine = head < have ? lists[w][head][lane] : KEY_NONE;
            uint64_t best = warp_min_u64(mine);
            if (mine == best && best != KEY_NONE) ++head;  // keys are unique (distinct ids)
            if (lane == 0) {
                nbr[v * k + o] = best == KEY_NONE ? -1 : int32_t(key_lo(best));
                dist[v * k + o] = best == KEY_NONE ? __int_as_float(0x7f800000) : key_w(best);
            }
        }
        __syncwarp();
    }
}

// Batched prep: per padded row r of the operand array, the cloud's centred
// BF16 hi (and lo) operand, its FP32 squared norm (key norms in padded rows,
// +inf on padding rows; row norms in compact rows) and the cloud's largest
// norm. mean holds the clouds' column means (B x ld).
__global__ void tc_prep_batched_kernel(const float *__restrict__ Xc, int ld, int64_t NP,
                                       const long long *__restrict__ roff,
                                       const long long *__restrict__ voff, int B,
                                       const CloudDev *__restrict__ cl, int kh_half, int x3,
                                       const float *__restrict__ mean,
                                       __nv_bfloat16 *__restrict__ H, float *__restrict__ ny,
                                       float *__restrict__ xnorm, unsigned *__restrict__ ymax_bits) {
    int64_t r = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (r >= NP) return;
    const int b = cloud_of(roff, B, r);
    const CloudDev c = cl[b];
    const int64_t q = r - roff[b];
    const int kh = (x3 ? 2 : 1) * kh_half;
    __nv_bfloat16 *h = H + r * kh;
    if (q >= c.n || !c.use_tc) {
        for (int t = lane; t < kh; t += 32) h[t] = __float2bfloat16_rn(0.0f);
        if (lane == 0) ny[r] = __int_as_float(0x7f800000);
        return;
    }
    const int64_t v = voff[b] + q;
    float acc = 0.0f;
    for (int t = lane; t < kh_half; t += 32) {
        float xc = t < c.d ? __fsub_rn(Xc[v * ld + t], mean[int64_t(b) * ld + t]) : 0.0f;
        __nv_bfloat16 hi = __float2bfloat16_rn(xc);
        h[t] = hi;
        if (x3) h[kh_half + t] = __float2bfloat16_rn(__fsub_rn(xc, __bfloat162float(hi)));
        acc = fmaf(xc, xc, acc);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
        ny[r] = acc;
        xnorm[v] = acc;
        // the cloud's rows all raise one word: only a row above it does
        const unsigned nb = __float_as_uint(sqrtf(acc));
        if (nb > *reinterpret_cast<volatile unsigned *>(ymax_bits + b)) atomicMax(ymax_bits + b, nb);
    }
}

// centre of every cloud (one block per cloud): the FP32 mean of up to 1024
// evenly spaced rows, eight loads in flight; the centre only has to be some
// fixed point near the cloud (every bound downstream holds for any centre)
__global__ void cloud_mean_kernel(const float *__restrict__ Xc, int ld,
                                  const CloudDev *__restrict__ cl, float *__restrict__ mean) {
    const int b = blockIdx.x;
    const CloudDev c = cl[b];
    const long long S = c.n < 1024 ? c.n : 1024;
    for (int t = threadIdx.x; t < ld; t += blockDim.x) {
        float s = 0.0f;
        if (t < c.d) {
            long long i = 0;
            for (; i + 8 <= S; i += 8) {
                float v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = __ldg(Xc + (c.voff + (i + q) * c.n / S) * ld + t);
#pragma unroll
                for (int q = 0; q < 8; ++q) s += v[q];
            }
            for (; i < S; ++i) s += __ldg(Xc + (c.voff + i * c.n / S) * ld + t);
        }
        mean[int64_t(b) * ld + t] = t < c.d && S > 0 ? s / float(S) : 0.0f;
    }
}

// keep the better of two top-1 results (the second with ids offset by k0)
__global__ void top1_merge_kernel(const int32_t *__restrict__ c2, const float *__restrict__ s2,
                                  int k0, int64_t n, int32_t *__restrict__ c,
                                  float *__restrict__ s) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (c2[i] >= 0 && s2[i] < s[i]) {
        c[i] = c2[i] + k0;
        s[i] = s2[i];
    }
}

struct TcPlan {
    int d_pad, nkb, kh, stages, r, cap;
    int64_t nq_tiles, nk_tiles;
    size_t smem;
};

// f8: E4M3 operand rows, 128 elements (128 bytes) per K block
TcPlan tc_plan(int64_t n, int d, int k, bool x3, bool f8 = false) {
    TcPlan p{};
    const int kel = f8 ? 2 * BK : BK;   // elements per 128-byte K block
    p.d_pad = (d + kel - 1) / kel * kel;
    p.nkb = p.d_pad / kel;
    p.kh = (x3 ? 2 : 1) * p.d_pad;
    // R, the minima kept per thread: 4 R keys at least stay in a row's log, of
    // which k + 1 plus the margin are wanted. A smaller R is cheaper per tile
    // and leaves more rows uncertified, each of which is redone exactly. At
    // k = 16, R = 6 / 8 / 10: 100,000 x 128 blobs 1.12 / 1.18 / 1.26 ms of tiles
    // and 1928 / 96 / 2 rows redone; 256 clouds of 500 to 20,000 points 22.5 /
    // 23.5 / 26.4 ms of tiles, 56.6 / 51.1 / 54.3 ms in all. At k = 32, R = 10 /
    // 12 / 14: 1M x 128 sphere points 7.6 / 8.1 / 8.4 ms, but 40 keys leave
    // overlapping clusters a margin of seven.
    p.r = k <= 7 ? 4 : (k <= 21 ? 8 : (k <= 37 ? 12 : 16));
    // (twice the places cost the re-rank two more key registers: 5.4 against
    // 3.5 ms at 1M rows and k = 32)
    p.cap = p.r <= 12 ? 64 : CAP;
    p.nq_tiles = (n + BM - 1) / BM;
    p.nk_tiles = (n + BN - 1) / BN;
    const size_t cap = 227 * 1024;
    const size_t fixed = 1024 + size_t(x3 ? 2 : 1) * p.nkb * A_BLOCK + 8 * BM * 4 + EPI * CAP * 8 + 512;
    p.stages = cap > fixed ? int(std::min<size_t>(6, (cap - fixed) / B_BLOCK)) : 0;
    p.smem = fixed + size_t(p.stages) * B_BLOCK;
    return p;
}

// One launch of the tile kernel; r: the plan's list length (0: top-1).
famst_status launch_tiles(const Exec &ex, int r, bool f8, unsigned grid, size_t smem,
                          const CUtensorMap &mA, const CUtensorMap &mB, const TcArgs &a) {
#define TC_LAUNCH(...)                                                                          \
    do {                                                                                        \
        if (set_smem_attr(knn_tc_kernel<__VA_ARGS__>, int(smem), ex.stream) != cudaSuccess)     \
            return FAMST_ERR_CUDA;                                                              \
        FAMST_LAUNCH(ex, (knn_tc_kernel<__VA_ARGS__>), grid, TC_THREADS, smem, mA, mB, a);      \
    } while (0)
    if (a.colcomp) {   // nearest foreign neighbours
        if (r > 4) return FAMST_ERR_UNSUPPORTED;
        TC_LAUNCH(4, true);
    } else if (f8) {
        if (r <= 8) TC_LAUNCH(8, false, true);
        else if (r <= 12) TC_LAUNCH(12, false, true);
        else TC_LAUNCH(16, false, true);
    } else {
        switch (r) {
            case 0: TC_LAUNCH(0, false); break;
            case 4: TC_LAUNCH(4, false); break;
            case 8: TC_LAUNCH(8, false); break;
            case 12: TC_LAUNCH(12, false); break;
            default: TC_LAUNCH(16, false);
        }
    }
#undef TC_LAUNCH
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

}  // namespace

bool knn_tc_supported(int64_t n, int d, int k, bool x3, bool f8) {
    if (k + 1 > 64 || n < 2) return false;
    TcPlan p = tc_plan(n, d, k, x3 && !f8, f8);
    return p.stages >= 2 && encode_fn() != nullptr;
}

size_t knn_tc_workspace(int64_t n, int d, int k, bool x3, int num_sms, bool prune, bool f8,
                        bool f32) {
    TcPlan p = tc_plan(n, d, k, x3 && !f8, f8);
    if (f8) prune = false;
    size_t b = 0;
    if (prune) {
        const int64_t K = prune_pivots_max(n), Kpad = (K + BN - 1) / BN * BN;
        b += align256(size_t(K) * 4) + align256(size_t(K) * p.kh * 2) +
             align256(size_t(Kpad + BN) * 4) * 2 + align256(size_t(n) * 4) * 2;
        b += prune_workspace(n, d, p.kh, f32 ? 0 : p.cap, p.nq_tiles, p.nk_tiles);
        b += align256(size_t(n) * 4) * 2 + align256(size_t(n) * 8) + 256;   // thr0, failed rows
        b += std::max(knn_fp32_pruned_workspace(n, k, p.nq_tiles),
                      visited_rows_workspace(n / VISITED_ROWS_SHARE));
    }
    b += align256(size_t(n) * p.kh * (f8 ? 1 : 2));        // operand rows
    if (f8) b += align256(size_t(p.nk_tiles) * BN * 4);    // per-row scales
    b += align256(size_t(p.nk_tiles) * BN * 4) * 2;        // ny, components (padded)
    b += align256(size_t(n) * 4);                          // xnorm2
    b += align256(size_t(d) * 4) + 256;                    // mean, ymax
    b += align256(size_t(4096) * d * 8);                   // column partials
    if (!f32) {   // (else the tensor tiles only place the points in cells)
        const int slots = log_slots(max_items(p.nq_tiles, p.nk_tiles, prune), num_sms);
        b += align256(size_t(n) * p.cap * 4) +                                    // candidates
             align256(size_t(slots) * LOG_SLOT * 8) + align256(size_t(slots) * 4);   // logs
    }
    b += align256(size_t(n) * 4) * 4 + 256;                // their number, splus, pivots, fail rows
    b += knn_fp32_workspace(n, d, k, n, num_sms);          // fallback
    return b;
}

// The partition takes about 1.1 ms whatever the size (a dozen
// synchronisations and sorts); the unpruned tiles take about 65 fs per pair
// and coordinate plus 1.2 ps per pair. The line is at 1.6 ms of those: 16384
// x 128 in 20 clusters 2.66 ms unpruned, 1.27 ms pruned; 32768 x 16 2.45 and
// 1.32 ms; 8192 x 128 0.88 ms unpruned; a cloud without structure loses the
// partition's time (50000 x 100: 18.2 -> 20.7 ms).
bool knn_fp32_prunes(int64_t n, int d, int k, bool vec4) {
    return double(n) * double(n) * (d + 18.0) >= 2.5e10 && prune_supported(n, d, k, vec4) &&
           knn_tc_supported(n, d, 1, false);
}

famst_status knn_tc(const Exec &ex, Arena &ar, const float *X, int64_t n, int d, int k, bool x3,
                    bool vec4, int32_t *nbr, float *dist, int32_t *pinned_host,
                    int64_t *uncertified, const int32_t *colcomp, bool prune,
                    int64_t *tiles_visited, bool f8, bool f32) {
    if (f8) {   // single E4M3 products, no tile pruning, no component mask
        x3 = false;
        prune = false;
        if (colcomp) return FAMST_ERR_UNSUPPORTED;
    }
    // f32: the tensor tiles only place the points in pivot cells
    TcPlan p = tc_plan(n, d, f32 ? 1 : k, x3, f8);
    if (p.stages < 2 || (k + 1 > 64 && !f32)) return FAMST_ERR_UNSUPPORTED;
    // operand rows: BF16 (kh elements) or E4M3 bytes (kh bytes) with per-row scales
    __nv_bfloat16 *H = f8 ? nullptr : ar.take<__nv_bfloat16>(size_t(n) * p.kh);
    uint8_t *Q = f8 ? ar.take<uint8_t>(size_t(n) * p.kh) : nullptr;
    float *rscale = f8 ? ar.take<float>(size_t(p.nk_tiles) * BN) : nullptr;
    if (f8 && (!Q || !rscale)) return FAMST_ERR_OOM;
    float *ny = ar.take<float>(size_t(p.nk_tiles) * BN);
    float *xn2 = ar.take<float>(size_t(n));
    float *mean = ar.take<float>(size_t(d));
    unsigned *ymax = ar.take<unsigned>(1);
    const int rows_per = int((n + 4095) / 4096) > 0 ? int((n + 4095) / 4096) : 1;
    const int nb = int((n + rows_per - 1) / rows_per);
    double *part = ar.take<double>(size_t(nb) * d);
    int32_t *cand = f32 ? nullptr : ar.take<int32_t>(size_t(n) * p.cap);   // (pruned: in cell order)
    int32_t *ccnt = ar.take<int32_t>(size_t(n));
    bool use_prune = prune && !colcomp && prune_supported(n, d, k, vec4);
    const int slots = log_slots(max_items(p.nq_tiles, p.nk_tiles, use_prune), ex.num_sms);
    int2 *log = f32 ? nullptr : ar.take<int2>(size_t(slots) * LOG_SLOT);
    int *claim = f32 ? nullptr : ar.take<int>(size_t(slots));
    int32_t *top = ar.take<int32_t>(size_t(n));   // pivot of every point
    float *splus = ar.take<float>(size_t(n));
    int32_t *fail_rows = ar.take<int32_t>(size_t(n));
    int32_t *fail_count = ar.take<int32_t>(1);
    if ((!f8 && !H) || !ny || !xn2 || !mean || !ymax || !part || (!f32 && (!cand || !log || !claim)) || !ccnt || !top || !splus ||
        !fail_rows || !fail_count)
        return FAMST_ERR_OOM;
    // prep: mean, centred BF16 operands, norms
    FAMST_LAUNCH(ex, colsum_partial_kernel, nb, 128, 0, X, n, d, rows_per, part);
    FAMST_LAUNCH(ex, colsum_final_kernel, d, 256, 0, part, nb, d, n, mean);
    if (cudaMemsetAsync(ymax, 0, 4, ex.stream) != cudaSuccess ||
        cudaMemsetAsync(fail_count, 0, 4, ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    const int64_t npad = p.nk_tiles * BN;
    const int scrambled = !use_prune;   // the pruning has an order of its own
    if (f8) {
        FAMST_LAUNCH(ex, tc_prep_f8_kernel, unsigned((n * 32 + 255) / 256), 256, 0, X, n, d,
                     p.d_pad, scrambled, mean, Q, rscale, ny, xn2, ymax);
        if (npad > n)
            FAMST_LAUNCH(ex, fill_value_kernel, unsigned((npad - n + 255) / 256), 256, 0, rscale,
                         n, npad, 1.0f);
    } else {
        FAMST_LAUNCH(ex, tc_prep_kernel, unsigned((n * 32 + 255) / 256), 256, 0, X, n, d, p.d_pad,
                     int(x3), scrambled, mean, H, ny, xn2, ymax);
    }
    if (npad > n)
        FAMST_LAUNCH(ex, fill_inf_kernel, unsigned((npad - n + 255) / 256), 256, 0, ny, n, npad);
    const size_t before_prune = ar.off;
    // persistent launches: one CTA per SM takes the query tiles round-robin
    const unsigned pgrid = unsigned(std::min<int64_t>(p.nq_tiles, ex.num_sms));
    PruneOut P;
    if (use_prune) {
        // pivot cells: top-1 pivot of every point on the tensor tiles (BF16),
        // one pivot of every n / K rows plus two coverage passes
        const int K0 = prune_pivots(n), M = prune_extra(n), Kmax = prune_pivots_max(n);
        const int Kpadmax = (Kmax + BN - 1) / BN * BN;
        int32_t *piv = ar.take<int32_t>(size_t(Kmax));
        __nv_bfloat16 *Hp = ar.take<__nv_bfloat16>(size_t(Kmax) * p.kh);
        float *nyp = ar.take<float>(size_t(Kpadmax + BN));   // +inf beyond the pivots
        // the pass's norms copied to an aligned buffer: the tile kernel reads
        // them as float4 from tile starts, and k0 need not be a multiple of 4
        float *nya = ar.take<float>(size_t(Kpadmax + BN));
        if (!piv || !Hp || !nyp || !nya) return FAMST_ERR_OOM;
        if (cudaMemcpyAsync(pinned_host, ymax, 4, cudaMemcpyDeviceToHost, ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
        famst_status st =
            prune_pivot_operands(ex, H, p.kh, ny, n, K0, Kpadmax + BN, piv, Hp, nyp);
        if (st != FAMST_OK) return st;
        const TcPlan p1 = tc_plan(n, d, 1, false);
        // top-1 over pivots [k0, k0 + kc) into (c_out, s_out), ids relative to k0
        auto assign = [&](int k0, int kc, int32_t *c_out, float *s_out) -> famst_status {
            CUtensorMap mA1, mB1;
            if (!make_map(&mA1, H, n, p.kh, BM) ||
                !make_map(&mB1, Hp + size_t(k0) * p.kh, kc, p.kh, BN))
                return FAMST_ERR_CUDA;
            const int nkt = (kc + BN - 1) / BN;
            if (cudaMemcpyAsync(nya, nyp + k0, size_t(nkt) * BN * 4, cudaMemcpyDeviceToDevice,
                                ex.stream) != cudaSuccess)
                return FAMST_ERR_CUDA;
            if (kc < nkt * BN)   // columns beyond the pass's pivots never win
                FAMST_LAUNCH(ex, fill_inf_kernel, 1, 256, 0, nya, int64_t(kc), int64_t(nkt) * BN);
            TcArgs a1{};
            a1.n = int(n);
            a1.nk_tiles = nkt;
            a1.nkb = p.nkb;
            a1.stages = p1.stages;
            a1.ny = nya;
            a1.cand = c_out;
            a1.splus = s_out;
            a1.status = ex.dstatus;
            a1.cross = 1;
            a1.nitems = int(p.nq_tiles);   // persistent: one CTA per SM walks the query tiles
            return launch_tiles(ex, 0, false, pgrid, p1.smem, mA1, mB1, a1);
        };
        int K = K0;
        st = assign(0, K, top, splus);
        // each coverage pass scores the points against the new pivots only
        int32_t *c2 = ar.take<int32_t>(size_t(n));
        float *s2 = ar.take<float>(size_t(n));
        if (!c2 || !s2) return FAMST_ERR_OOM;
        for (int pass = 0; pass < 2 && st == FAMST_OK; ++pass) {
            int me = 0;
            st = prune_augment(ex, ar, xn2, splus, n, H, p.kh, ny, M, K, piv, Hp, nyp, &me);
            // only the distinct new pivots are scored (the repeats add no cell)
            if (st == FAMST_OK && me > 0) {
                st = assign(K, me, c2, s2);
                if (st == FAMST_OK)
                    FAMST_LAUNCH(ex, top1_merge_kernel, unsigned((n + 255) / 256), 256, 0, c2, s2,
                                 K, n, top, splus);
            }
            K += M;
        }
        if (st != FAMST_OK) return st;
        // (the passes above have waited for the stream)
        float norm_max;
        std::memcpy(&norm_max, pinned_host, 4);
        if (!(norm_max < NORM_MAX)) {
            use_prune = false;
            ar.off = before_prune;
        } else {
            st = prune_partition(ex, ar, X, d, n, k, H, p.kh, ny, p.nkb, K, piv, top, 1,
                                 pinned_host + 2, &P);
            if (st != FAMST_OK) return st;
        }
    }
    if (f32) {
        *uncertified = 0;
        if (tiles_visited) *tiles_visited = p.nq_tiles * p.nk_tiles;
        return use_prune ? knn_fp32_pruned(ex, ar, X, n, d, k, P, nbr, dist)
                         : knn_fp32(ex, ar, X, n, d, k, nullptr, 0, n, nbr, dist);
    }
    int32_t *side_j = nullptr, *side_cnt = nullptr;   // candidates of the parts of split lists
    float *side_s = nullptr, *side_sp = nullptr;
    float *thr0 = nullptr;       // start thresholds
    uint64_t *fail_kth = nullptr;
    int32_t *fails2 = nullptr, *nfail2 = nullptr;
    if (use_prune) {
        thr0 = ar.take<float>(size_t(n));
        fail_kth = ar.take<uint64_t>(size_t(n));
        fails2 = ar.take<int32_t>(size_t(n));
        nfail2 = ar.take<int32_t>(1);
        if (!thr0 || !fail_kth || !fails2 || !nfail2) return FAMST_ERR_OOM;
        side_j = ar.take<int32_t>(size_t(PRUNE_SPLIT_SLOTS) * BM * p.cap);
        side_s = ar.take<float>(size_t(PRUNE_SPLIT_SLOTS) * BM * p.cap);
        side_cnt = ar.take<int32_t>(size_t(PRUNE_SPLIT_SLOTS) * BM);
        side_sp = ar.take<float>(size_t(PRUNE_SPLIT_SLOTS) * BM);
        if (!side_j || !side_s || !side_cnt || !side_sp) return FAMST_ERR_OOM;
    }
    const void *Hop = f8 ? static_cast<const void *>(Q)
                         : static_cast<const void *>(use_prune ? P.Hs : H);
    CUtensorMap mA, mB;
    if (!make_map(&mA, Hop, n, p.kh, BM, f8) || !make_map(&mB, Hop, n, p.kh, BN, f8))
        return FAMST_ERR_CUDA;
    int32_t *cpad = nullptr;   // components over the padded rows (-1 beyond n)
    if (colcomp) {
        cpad = ar.take<int32_t>(size_t(npad));
        if (!cpad) return FAMST_ERR_OOM;
        FAMST_LAUNCH(ex, pad_components_kernel, unsigned((npad + 255) / 256), 256, 0, colcomp, n,
                     npad, cpad);
    }
    // certificate constants (also the pruned lists' start thresholds)
    const double kprod = double(x3 ? 3 * p.d_pad : p.d_pad);
    double eps_dot = tc_eps_dot(p.d_pad, x3);
    if (f8) {
        // E4M3 with the row's scale: a normal element is within u = 2^-4 of
        // x'_t (relative); an element below the normal range within 2^-10 s,
        // and s <= 2 max|x'| / 448, so over the row those add at most
        // sqrt(d) 2^-10 (2 / 448) ||x'|| per side. Products of E4M3 values
        // are exact in FP32; the accumulation term is as for BF16.
        // With |x^_t - x'_t| <= u|x'_t| + c ||x'|| (c = 2^-10 2/448) on both
        // sides, |x^.y^ - x'.y'| <= ((2u + u^2) + 2 sqrt(d)(1 + u) c + d c^2)
        // ||x'|| ||y'||.
        const double u4 = 1.0 / 16.0, c8 = 2.0 / 448.0 / 1024.0, dp = double(p.d_pad);
        eps_dot = 2.0 * u4 + u4 * u4 + 2.0 * std::sqrt(dp) * (1.0 + u4) * c8 + dp * c8 * c8 +
                     kprod * std::ldexp(1.0, -22) * (1.0 + 4.0 * u4);
    }
    const CertConst cc = cert_const(eps_dot, d);
    if (use_prune)
        FAMST_LAUNCH(ex, thr0_kernel, unsigned((n + 255) / 256), 256, 0, P.tau_row, P.nys, n, d,
                     ymax, cc.eps_dot, thr0);
    TcArgs a{};
    a.n = int(n);
    a.nk_tiles = int(p.nk_tiles);
    a.nkb = p.nkb;
    a.x3 = int(x3);
    a.stages = p.stages;
    a.ny = use_prune ? P.nys : ny;
    a.cand = cand;
    a.ccnt = ccnt;
    a.cap = p.cap;
    a.sel = Select{k, p.cap, float(4.2 * cc.eps_dot), score_eps_row(d)};
    a.ymax = ymax;
    a.log = log;
    a.claim = claim;
    a.nslots = slots;
    if (cudaMemsetAsync(claim, 0, size_t(slots) * 4, ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    a.splus = splus;
    a.status = ex.dstatus;
    a.colcomp = cpad;
    a.rscale = rscale;
    a.thr0 = thr0;
    // one CTA per work item: the pruned tiles' key lists differ in length,
    // and a static round-robin over persistent CTAs measured slower here.
    // Pruned lists come as work items, long ones split into parts; the grid
    // covers the most items the table can hold and the CTAs beyond its
    // count leave at once.
    unsigned tgrid = unsigned(p.nq_tiles);
    if (use_prune) {
        a.tiles = P.tab;
        a.klist = P.klist;
        a.nitems_dev = P.nitems;
        a.side_j = side_j;
        a.side_s = side_s;
        a.side_cnt = side_cnt;
        a.side_splus = side_sp;
        tgrid = unsigned(p.nq_tiles + PRUNE_SPLIT_SLOTS);
    }
    timer_mark(ex, TIMER_TILES, false);
    {
        const famst_status st = launch_tiles(ex, p.r, f8, tgrid, p.smem, mA, mB, a);
        if (st != FAMST_OK) return st;
    }
    if (use_prune)   // rows of split lists: combine their parts
        FAMST_LAUNCH(ex, split_merge_kernel, dim3(PRUNE_SPLIT_TILES, BM / 16), 512, 0, P.splitq,
                     P.nsplit, side_j, side_s, side_cnt, side_sp, n, a.sel, a.ny, ymax, cand, ccnt,
                     splus, ex.dstatus);
    timer_mark(ex, TIMER_TILES, true);
    if (cudaPeekAtLastError() != cudaSuccess) return FAMST_ERR_CUDA;
    const unsigned rgrid = unsigned((n * 32 + 255) / 256);
#define RERANK2(XRV, HV)                                                                         \
    do {                                                                                         \
        if (use_prune)                                                                           \
            FAMST_LAUNCH(ex, (rerank_sorted_kernel<XRV, HV>), rgrid, 256, 0, P.Xs, n, d, k,      \
                         cand, ccnt, splus, P.skipQ, P.perm, xn2, ymax, cc, ex.dstatus, nbr, dist, \
                         fail_rows, fail_kth, fail_count);                                       \
        else                                                                                     \
            FAMST_LAUNCH(ex, (rerank_kernel<XRV, HV>), rgrid, 256, 0, X, n, d, k, scrambled,     \
                         cand, ccnt, splus, xn2, ymax, cc, ex.dstatus, nbr, dist, fail_rows,     \
                         fail_count);                                                            \
    } while (0)
#define RERANK(XRV)                                                                              \
    do {                                                                                         \
        if (p.cap == 64) RERANK2(XRV, 2);                                                        \
        else RERANK2(XRV, 4);                                                                    \
    } while (0)
    timer_mark(ex, TIMER_RERANK, false);
    if (d <= 128) RERANK(4);
    else if (d <= 256) RERANK(8);
    else if (d <= 512) RERANK(16);
    else RERANK(0);
    timer_mark(ex, TIMER_RERANK, true);
#undef RERANK
#undef RERANK2
    if (cudaMemcpyAsync(pinned_host, fail_count, 4, cudaMemcpyDeviceToHost, ex.stream) != cudaSuccess ||
        (use_prune && cudaMemcpyAsync(pinned_host + 1, P.visited, 4, cudaMemcpyDeviceToHost,
                                      ex.stream) != cudaSuccess) ||
        cudaStreamSynchronize(ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    const int32_t nfail = *pinned_host;
    *uncertified = nfail;
    if (tiles_visited) *tiles_visited = use_prune ? int64_t(pinned_host[1]) : p.nq_tiles * p.nk_tiles;
    if (nfail > 0 && use_prune) {
        // few rows: exact over their tile's list, read for each row by
        // itself; many: the FP32 tiles over all lists, which share a key
        // among 64 rows
        famst_status st;
        if (nfail <= n / VISITED_ROWS_SHARE) {
            if (cudaMemsetAsync(nfail2, 0, 4, ex.stream) != cudaSuccess) return FAMST_ERR_CUDA;
            st = visited_rows(ex, ar, P, n, d, k, fail_rows, fail_kth, nfail, nbr, dist, fails2, nfail2);
            if (st == FAMST_OK)
                st = exact_rows(ex, X, n, d, k, fails2, nfail2, nfail, nullptr, nbr, dist);
        } else {
            st = knn_fp32_pruned(ex, ar, X, n, d, k, P, nbr, dist);
        }
        if (st != FAMST_OK) return st;
    } else if (nfail > 0) {
        famst_status st = knn_fp32(ex, ar, X, n, d, k, fail_rows, 0, nfail, nbr, dist, colcomp);
        if (st != FAMST_OK) return st;
    }
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

}  // namespace famst

namespace famst {

// Shared-memory plan of the batched tensor path for operand width D (the
// largest cloud's K extent).
bool knn_tc_batched_plan(int D, int k, bool x3, int *stages, size_t *smem) {
    if (k + 1 > 64) return false;
    const TcPlan p = tc_plan(int64_t(1) << 20, D, k, x3);
    if (p.stages < 2 || encode_fn() == nullptr) return false;
    *stages = p.stages;
    *smem = p.smem;
    return true;
}

int knn_tc_epilogue_warps() { return EPI; }
int knn_tc_cand_cap(int k) { return tc_plan(1, 1, k, false).cap; }
size_t knn_tc_log_entries(int64_t nctas, int num_sms) {
    return size_t(log_slots(nctas, num_sms)) * LOG_SLOT;
}

// Everything of the batched tensor path that runs on the device; buffers
// come from the caller's plan, so nothing here allocates or synchronises.
famst_status knn_tc_batched(const Exec &ex, const float *Xc, int D, int64_t N, int64_t NP,
                            const long long *voff, const long long *roff, int B,
                            const CloudDev *cl, const TcTile *tiles, int64_t nctas, int k,
                            bool x3, int stages, size_t smem, __nv_bfloat16 *H,
                            float *ny, float *xn2, float *mean, unsigned *ymax, int32_t *cand,
                            int32_t *ccnt, int2 *log, int *claim, float *splus,
                            int32_t *fail_rows, int32_t *fail_count, int32_t *nbr, float *dist,
                            const CUtensorMap *mA, const CUtensorMap *mB,
                            const float *Xorig, const int32_t *perm) {
    FAMST_LAUNCH(ex, cloud_mean_kernel, B, 128, 0, Xc, D, cl, mean);
    if (cudaMemsetAsync(ymax, 0, size_t(B) * 4, ex.stream) != cudaSuccess ||
        cudaMemsetAsync(fail_count, 0, 4, ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    FAMST_LAUNCH(ex, tc_prep_batched_kernel, unsigned((NP * 32 + 255) / 256), 256, 0, Xc, D, NP,
                 roff, voff, B, cl, D, int(x3), mean, H, ny, xn2, ymax);
    const TcPlan p = tc_plan(1, D, k, x3);
    if (nctas > 0) {
        TcArgs a{};
        a.nkb = D / BK;
        a.x3 = int(x3);
        a.stages = stages;
        a.ny = ny;
        a.cand = cand;
        a.ccnt = ccnt;
        a.cap = p.cap;
        a.sel = Select{k, p.cap, float(4.2 * tc_eps_dot(D, x3)), score_eps_row(D)};
        a.ymax = ymax;
        a.log = log;
        a.claim = claim;
        a.nslots = log_slots(nctas, ex.num_sms);
        if (cudaMemsetAsync(claim, 0, size_t(a.nslots) * 4, ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
        a.splus = splus;
        a.status = ex.dstatus;
        a.tiles = tiles;
        // persistent: one CTA per SM walks the (cloud, query tile) items round-robin
        a.nitems = int(nctas);
        a.spiral = perm != nullptr ? 1 : 0;
        const famst_status st =
            launch_tiles(ex, p.r, false,
                         unsigned(std::min<int64_t>(nctas, ex.num_sms)), smem, *mA, *mB, a);
        if (st != FAMST_OK) return st;
    }
    const unsigned rgrid = unsigned((N * 32 + 255) / 256);
    // one candidate at a time per warp over coalesced row reads when the
    // padded rows fit the register slices (D <= 512), else one per lane
    // (the widest cloud's bounds hold for every cloud; FP64 takes each one's own)
    const CertConst cc = cert_const(tc_eps_dot(D, x3), D);
#define RRB2(XRV, HV)                                                                            \
    FAMST_LAUNCH(ex, (rerank_batched_kernel<XRV, HV>), rgrid, 256, 0, Xc, D, N, voff, B, cl,     \
                 int(x3), k, cand, ccnt, splus, xn2, ymax, cc, ex.dstatus, perm, nbr, dist, fail_rows, \
                 fail_count)
#define RRB(XRV)                                                                                 \
    do {                                                                                         \
        if (p.cap == 64) RRB2(XRV, 2);                                                           \
        else RRB2(XRV, 4);                                                                       \
    } while (0)
    if (D <= 128) RRB(4);
    else if (D <= 256) RRB(8);
    else if (D <= 512) RRB(16);
    else RRB(0);
#undef RRB
#undef RRB2
    // rows no certificate covers: exact within their cloud, original order and ids
    FAMST_LAUNCH(ex, fallback_rows_kernel, unsigned(ex.num_sms) * 16, FB_WARPS * 32, 0,
                 Xorig ? Xorig : Xc, D, voff, B, cl, k, fail_rows, fail_count, nbr, dist);
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

famst_status fallback_rows_batched(const Exec &ex, const float *Xc, int ld, const long long *voff,
                                   int B, const CloudDev *cl, int k, const int32_t *rows,
                                   const int32_t *count, int32_t *nbr, float *dist) {
    FAMST_LAUNCH(ex, fallback_rows_kernel, unsigned(ex.num_sms) * 16, FB_WARPS * 32, 0, Xc, ld,
                 voff, B, cl, k, rows, count, nbr, dist);
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

// Tensor maps over the padded operand rows (queries 128-row boxes, keys
// 256-row boxes); made on the host before any capture.
bool knn_tc_batched_maps(const void *H, int64_t NP, int D, bool x3, CUtensorMap *mA,
                         CUtensorMap *mB) {
    const int64_t kh = (x3 ? 2 : 1) * int64_t(D);
    return make_map(mA, H, NP, kh, BM) && make_map(mB, H, NP, kh, BN);
}

}  // namespace famst
