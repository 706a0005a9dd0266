// Phase 1 (Algorithm 1, GetANNs) as exact brute force on FP32 SIMT tiles.
//
// A block owns QM = 64 query rows and sweeps key tiles of KN = 128 points.
// For every (query, key) pair the block computes a fast squared distance:
// fmaf(x_t - y_t, x_t - y_t, .) over the even and over the odd coordinates,
// in order, in the two halves of packed FP32 pairs, then their sum (rows
// staged in shared memory as they are, in chunks of DC = 32 coordinates,
// double buffered by cp.async; a thread accumulates an 8 x 8 micro-tile). It
// keeps the k' = k + 8 best (sqrt p, id) of every row; the canonical re-rank
// below computes their canonical distances, sorts them, and certifies the
// row when the FP32 error bound proves no unkept point can reach the k-th
// canonical distance. Rows it cannot certify (ties at the boundary) are
// recomputed by an exact warp-per-row brute force on canonical distances.
//
// Bound: the FP32 pipe (two packed instructions per pair of coordinates and
// (query, key) pair). Rows stay in their own layout, so one 16-byte shared
// load feeds four coordinates: 16 loads per 256 packed instructions, and two
// blocks of four warps fit an SM, one computing while the other selects or
// waits at a barrier. 50021 x 100, k = 16: 59.5 ms with one block of eight
// warps per SM, scalar arithmetic and one selecting thread per list; 18.2 ms
// (1.37e13 coordinate pairs/s, 70% of the pipe's 1.95e13) with these tiles,
// and 1.6 ms where the cloud has 20 clusters and the pruned lists are used.
//
// Selection is fused: a thread compares its 64 values with their rows'
// thresholds (the k'-th kept, or a bound the caller knows in advance) in
// registers and appends the few survivors to the rows' queues in shared
// memory. A warp then takes each row whose queue is half full: the queue is
// sorted and merged into the row's sorted list by bitonic networks in
// registers (element 32 h + lane), two rows at a time. Values that found a
// queue full stay pending and are compared with the tightened threshold
// again. The n x n matrix never leaves the SM. When the key range is split
// over S blocks (small n) or a pruned tile's list is split, the re-rank
// merges the parts' lists.
#include <cuda_runtime.h>

#include <algorithm>

#include "famst_internal.cuh"

namespace famst {
namespace {

constexpr int QM = 64;
constexpr int KN = 128;
constexpr int DC = 32;
constexpr int NT = 128;
constexpr int RS = DC + 4;          // floats per staged row: 8 rows fall in 8 bank groups
constexpr int STAGE = (QM + KN) * RS;
constexpr int QCAP = 32;            // queued survivors per row
constexpr int FLUSH_AT = 16;        // a row is merged when its queue holds this many

// list registers per lane for kp candidates
inline int list_regs(int kp) { return kp <= 32 ? 1 : (kp <= 64 ? 2 : 4); }

struct KnnSmem {
    static size_t bytes(int kp) {
        return size_t(2 * STAGE) * sizeof(float) + size_t(kp + QCAP) * QM * sizeof(uint64_t) +
               size_t(QM) * 4 * 4;
    }
};

// ------------------------------------------- sorted lists held by a warp
// Element e = 32 h + lane of an ascending list sits in register h of its lane,
// KEY_NONE at the end.

// v bitonic -> ascending over the lanes
__device__ __forceinline__ uint64_t warp_bitonic32(uint64_t v, int lane) {
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const uint64_t o = shfl_xor_u64(v, s);
        const bool lower = (lane & s) == 0;
        v = (v < o) == lower ? v : o;
    }
    return v;
}
__device__ __forceinline__ uint64_t warp_sort32(uint64_t v, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int s = size >> 1; s >= 1; s >>= 1) {
            const uint64_t o = shfl_xor_u64(v, s);
            const bool lower = ((lane & s) == 0) == ((lane & size) == 0);
            v = (v < o) == lower ? v : o;
        }
    }
    return v;
}
// the list keeps its 32 H smallest of itself and the ascending batch B
template <int H>
__device__ __forceinline__ void warp_list_merge(uint64_t (&L)[H], uint64_t B, int lane) {
#pragma unroll
    for (int h = H - 1; h >= 0; --h) {
        const uint64_t rb = shfl_idx_u64(B, 31 - lane);
        const uint64_t lo = L[h] < rb ? L[h] : rb, hi = L[h] < rb ? rb : L[h];
        if (h + 1 < H) L[h + 1] = warp_bitonic32(hi, lane);
        B = warp_bitonic32(lo, lane);
    }
    L[0] = B;
}
// Insert key K; the last element drops out.
template <int H>
__device__ __forceinline__ void warp_list_insert(uint64_t (&L)[H], uint64_t K, int lane) {
    int pos = 0;
#pragma unroll
    for (int h = 0; h < H; ++h) pos += __popc(__ballot_sync(0xffffffffu, L[h] < K));
    uint64_t prev[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const uint64_t up = shfl_up_u64(L[h], 1);
        const uint64_t wrap = h > 0 ? shfl_idx_u64(L[h > 0 ? h - 1 : 0], 31) : KEY_NONE;
        prev[h] = lane == 0 ? wrap : up;
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int e = h * 32 + lane;
        L[h] = e < pos ? L[h] : (e == pos ? K : prev[h]);
    }
}
template <int H>
__device__ __forceinline__ uint64_t warp_list_at(const uint64_t (&L)[H], int e) {
    uint64_t v = L[0];
#pragma unroll
    for (int h = 1; h < H; ++h) v = (e >> 5) == h ? L[h] : v;
    return shfl_idx_u64(v, e & 31);
}

__device__ __forceinline__ void cp_async_f4(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_f1(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}

// p of every key at or below this is offered to the lists: the squared
// bound tau on a row's k-th neighbour distance, widened by the ratio of fast
// to canonical sums on both sides of the certificate's comparison
__device__ __forceinline__ float tau_p(float tau, float rho) {
    return __fmul_ru(__fmul_ru(tau, tau), __fmaf_ru(4.0f, rho, 1.0f + 0x1p-18f));
}

struct TileArgs {
    const float *X;
    int n, d, ld, kp;
    const int32_t *qrows;   // query rows (null: q0 + q)
    int64_t q0;
    int nq;
    int tiles_per_split;
    uint64_t *part;         // [split][query][kp] lists (null: nbr / dist)
    int32_t *nbr;
    float *dist;
    const F32Tile *btab;    // batched: one block per 64 query rows of one cloud
    const int32_t *colcomp; // keys of the query's own component are skipped
    // pruned lists: block b takes half b & 1 of work item b >> 1, 128 query rows with the 256-key
    // tiles klist[kt0 .. kt1); lists of a split item's part go to `side`
    const TcTile *items;
    const int32_t *nitems;
    const int32_t *klist;
    uint64_t *side;
    const float *tau;       // per query row: an upper bound on its k-th distance
    float rho;
    // split key ranges: the smallest threshold any of a query's parts has
    // reached (float bits, all ones at the start). A part's k'-th key is at
    // or above the query's, so every part may filter with it, and the parts
    // that run later insert little.
    unsigned *thr_g;
};

// VEC: rows are 16-byte aligned and a multiple of four floats apart, with
// zeros from column d to the next multiple of four.
template <int H, bool VEC>
__global__ void __launch_bounds__(NT, 2) knn_fp32_kernel(TileArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *stage = reinterpret_cast<float *>(smem_raw);
    uint64_t *Q = reinterpret_cast<uint64_t *>(stage + 2 * STAGE);   // [row][QCAP]
    uint64_t *L = Q + QCAP * QM;                                      // [row][kp]
    float *thr_s = reinterpret_cast<float *>(L + size_t(A.kp) * QM);
    int *qid_s = reinterpret_cast<int *>(thr_s + QM);
    int *comp_s = qid_s + QM;
    int *qcnt = comp_s + QM;   // survivors offered to the row's queue (may exceed QCAP)

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tx = tid & 15, ty = tid >> 4;
    const int kp = A.kp;
    const float inf = __int_as_float(0x7f800000);
    int n = A.n, d = A.d, nq = A.nq, shift = 0, key_base = 0, qbase = int(blockIdx.x) * QM;
    int64_t q0 = A.q0;
    int tile_begin, tile_end;   // 128-key tiles (of the list: two per entry)
    const int32_t *kl = nullptr;
    uint64_t *out = A.part;     // list of the block's first row
    if (A.btab) {
        const F32Tile T = A.btab[blockIdx.x];
        tile_begin = T.tile0;
        tile_end = T.tile1;
        key_base = T.key_base;
        n = T.key_end;
        d = T.d;
        shift = T.shift;
        nq = T.nq;
        q0 = T.qbase;
        qbase = 0;
    } else if (A.items) {
        if (int(blockIdx.x >> 1) >= __ldg(A.nitems)) return;
        const TcTile T = A.items[blockIdx.x >> 1];
        const int half = int(blockIdx.x & 1) * QM;
        kl = A.klist + T.kt0;
        tile_begin = 0;
        tile_end = 2 * (T.kt1 - T.kt0);
        qbase = T.q0 + half;
        q0 = 0;
        nq = T.row_end;
        out = T.part > 0 ? A.side + (size_t(T.part - 1) * 2 * QM + half) * kp
                         : A.part + size_t(qbase) * kp;
        if (qbase >= nq) return;
    } else {
        const int ntiles = (n + KN - 1) / KN;
        tile_begin = int(blockIdx.y) * A.tiles_per_split;
        tile_end = min(ntiles, tile_begin + A.tiles_per_split);
        if (out) out += (size_t(blockIdx.y) * nq + qbase) * kp;
    }
    if (tid < QM) {
        const int q = qbase + tid;
        const int id = q < nq ? (A.qrows ? A.qrows[q] : int(q0 + q)) : -1;
        qid_s[tid] = id;
        thr_s[tid] = id < 0 ? -1.0f : (A.tau ? tau_p(A.tau[id], A.rho) : inf);
        comp_s[tid] = A.colcomp && id >= 0 ? A.colcomp[id] : -1;
        qcnt[tid] = 0;
    }
    for (int x = tid; x < kp * QM; x += NT) L[x] = KEY_NONE;
    __syncthreads();

    const int nchunks = (d + DC - 1) / DC;
    const int nsteps = (tile_end - tile_begin) * nchunks;
    auto key0_of = [&](int tile) {
        return kl ? __ldg(kl + (tile >> 1)) * (2 * KN) + (tile & 1) * KN : key_base + tile * KN;
    };
    // stage step s (chunk s mod nchunks of a tile) into its buffer
    auto issue = [&](int s) {
        const int c0 = (s % nchunks) * DC;
        const int key0 = key0_of(tile_begin + s / nchunks);
        float *dst = stage + (s & 1) * STAGE;
        if constexpr (VEC) {
            const int c4 = (tid & 7) * 4, col = c0 + c4;
            if (col < d) {
#pragma unroll
                for (int r = 0; r < (QM + KN) / (NT / 8); ++r) {
                    const int row = (tid >> 3) + r * (NT / 8);
                    const int id = row < QM ? qid_s[row] : key0 + row - QM;
                    const bool ok = row < QM ? id >= 0 : id < n;
                    cp_async_f4(uint32_t(__cvta_generic_to_shared(dst + row * RS + c4)),
                                A.X + (ok ? int64_t(id) * A.ld + col : 0), ok ? 16 : 0);
                }
            }
        } else {
            const int d4 = min(DC, ((d - c0) + 3) & ~3);
            const int col = c0 + lane;
            if (lane < d4) {
                for (int row = warp; row < QM + KN; row += NT / 32) {
                    const int id = row < QM ? qid_s[row] : key0 + row - QM;
                    const bool ok = (row < QM ? id >= 0 : id < n) && col < d;
                    cp_async_f1(uint32_t(__cvta_generic_to_shared(dst + row * RS + lane)),
                                A.X + (ok ? int64_t(id) * A.ld + col : 0), ok ? 4 : 0);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    // merge the queues of this warp's rows that hold at least `least`, two
    // rows at a time (their shuffles overlap)
    auto flush = [&](int least) {
        const int mine = lane < QM / 4 ? min(qcnt[warp * (QM / 4) + lane], QCAP) : 0;
        unsigned full = __ballot_sync(0xffffffffu, mine >= least);
#pragma unroll 1
        while (full) {
            int row[2];
            uint64_t B[2], E[2][H];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = full ? __ffs(full) - 1 : -1;
                full &= full - 1;
                row[i] = r < 0 ? -1 : warp * (QM / 4) + r;
                const int c = r < 0 ? 0 : __shfl_sync(0xffffffffu, mine, r);
                B[i] = lane < c ? Q[row[i] * QCAP + lane] : KEY_NONE;
#pragma unroll
                for (int h = 0; h < H; ++h)
                    E[i][h] = r >= 0 && 32 * h + lane < kp ? L[row[i] * kp + 32 * h + lane]
                                                           : KEY_NONE;
            }
            B[0] = warp_sort32(B[0], lane);
            B[1] = warp_sort32(B[1], lane);
            warp_list_merge<H>(E[0], B[0], lane);
            warp_list_merge<H>(E[1], B[1], lane);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint64_t kth = warp_list_at<H>(E[i], kp - 1);
                if (row[i] < 0) continue;
#pragma unroll
                for (int h = 0; h < H; ++h)
                    if (32 * h + lane < kp) L[row[i] * kp + 32 * h + lane] = E[i][h];
                if (lane == 0) {
                    qcnt[row[i]] = 0;
                    if (kth != KEY_NONE) {
                        const float w = key_w(kth);
                        const float t = w * w * (1.0f + 0x1p-20f);
                        thr_s[row[i]] = fminf(thr_s[row[i]], t);
                        if (A.thr_g) atomicMin(A.thr_g + qbase + row[i], __float_as_uint(t));
                    }
                }
            }
        }
        __syncwarp();
    };

    if (nsteps > 0) issue(0);
    unsigned long long acc[8][8];
    for (int s = 0; s < nsteps; ++s) {
        const int c = s % nchunks;
        if (c == 0) {
            // (the row's own thread lowers it; read by others after a barrier)
            if (A.thr_g && tid < QM && qbase + tid < nq)
                thr_s[tid] = fminf(thr_s[tid], __uint_as_float(__ldcg(A.thr_g + qbase + tid)));
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // step s staged; every warp is done with step s - 1
        if (s + 1 < nsteps) issue(s + 1);
        const float *Qs = stage + (s & 1) * STAGE + ty * RS;
        const float *Ks = stage + (s & 1) * STAGE + (QM + tx) * RS;
        const int nt = min(DC, d - c * DC);
#pragma unroll 1
        for (int t = 0; t < nt; t += 4) {
            ulonglong2 b[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                b[j] = *reinterpret_cast<const ulonglong2 *>(Ks + 16 * j * RS + t);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(Qs + 8 * i * RS + t);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    acc[i][j] = f2_sqacc(f2_sub(a.x, b[j].x), acc[i][j]);
                    acc[i][j] = f2_sqacc(f2_sub(a.y, b[j].y), acc[i][j]);
                }
            }
        }
        if (c + 1 < nchunks) continue;
        // survivors: query ty + 8 i, key tx + 16 j; bit 8 i + j of `pend`
        // marks a value not yet queued
        const int key0 = key0_of(tile_begin + s / nchunks);
        float pv[64];
        unsigned long long pend = 0ull;
        auto compare = [&](unsigned long long among) {
            pend = 0ull;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float thr = thr_s[ty + 8 * i];
                float mn = pv[8 * i];
#pragma unroll
                for (int j = 1; j < 8; ++j) mn = fminf(mn, pv[8 * i + j]);
                if (mn <= thr) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (pv[8 * i + j] <= thr) pend |= 1ull << (8 * i + j);
                }
            }
            pend &= among;
        };
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) pv[8 * i + j] = f2_hsum(acc[i][j]);
        compare(~0ull);
        const bool last = s + 1 == nsteps;
        while (true) {
            const bool more = __syncthreads_or(pend != 0ull);
            if (!more && !last) break;
            // one survivor per thread and turn (one copy of the code: unrolled
            // over the 64 values it does not fit the instruction cache)
            unsigned long long left = 0ull;
#pragma unroll 1
            while (pend) {
                const int b = __ffsll(pend) - 1;
                pend &= pend - 1ull;
                float v[32];   // the value at b, by its bits
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = (b & 1) ? pv[2 * x + 1] : pv[2 * x];
#pragma unroll
                for (int w = 1; w < 6; ++w)
#pragma unroll
                    for (int x = 0; x < (32 >> w); ++x)
                        v[x] = (b >> w) & 1 ? v[2 * x + 1] : v[2 * x];
                const int row = ty + (b & ~7), jj = key0 + tx + 16 * (b & 7);
                bool in = jj < n && jj != qid_s[row];
                if (A.colcomp && in) in = A.colcomp[jj] != comp_s[row];
                if (!in) continue;
                const int slot = atomicAdd(&qcnt[row], 1);
                if (slot < QCAP) Q[row * QCAP + slot] = nb_key(__fsqrt_rn(v[0]), uint32_t(jj));
                else left |= 1ull << b;
            }
            __syncthreads();
            flush(more ? FLUSH_AT : 1);   // the last tile ends with every queue merged
            __syncthreads();
            if (!more) break;
            if (left) compare(left);
        }
    }
    const int rows = min(QM, nq - qbase);
    for (int x = tid; x < rows * kp; x += NT) {
        const uint64_t v = L[x];
        if (out) {
            out[x] = v;
        } else {
            const int64_t o = (A.btab ? q0 - shift : int64_t(qbase)) * kp + x;
            A.nbr[o] = v == KEY_NONE ? -1 : int32_t(key_lo(v)) - shift;
            A.dist[o] = v == KEY_NONE ? inf : key_w(v);
        }
    }
}

template <int H>
famst_status launch_tiles_h(const Exec &ex, dim3 grid, const TileArgs &A, bool vec) {
    const size_t smem = KnnSmem::bytes(A.kp);
    if (vec) {
        if (set_smem_attr(knn_fp32_kernel<H, true>, smem, ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
        FAMST_LAUNCH(ex, (knn_fp32_kernel<H, true>), grid, NT, smem, A);
    } else {
        if (set_smem_attr(knn_fp32_kernel<H, false>, smem, ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
        FAMST_LAUNCH(ex, (knn_fp32_kernel<H, false>), grid, NT, smem, A);
    }
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

famst_status launch_tiles(const Exec &ex, dim3 grid, const TileArgs &A) {
    const bool vec = (A.ld & 3) == 0 && (reinterpret_cast<uintptr_t>(A.X) & 15) == 0;
    switch (list_regs(A.kp)) {
        case 1: return launch_tiles_h<1>(ex, grid, A, vec);
        case 2: return launch_tiles_h<2>(ex, grid, A, vec);
        default: return launch_tiles_h<4>(ex, grid, A, vec);
    }
}

// ------------------------------------------------------------ exactness

constexpr int FP32_MARGIN = 8;   // candidates kept beyond k for the certificate

// Canonical squared distances of 32 keys (lane l's key `cand`, < 0: none)
// to one point whose coordinates t = l + 32 j lane l holds in xs[j]: lane l
// accumulates partial l of every key (coalesced loads), a butterfly
// transpose-sum then leaves key l's canonical value in lane l -- at every
// stage a lane adds the same pair of partial sums the canonical butterfly
// adds, for the key whose result it keeps.
template <int DJ>
__device__ __forceinline__ float warp_canon32(const float *__restrict__ X, int ld, int d,
                                              const float (&xs)[DJ], int self, int cand,
                                              int lane) {
    float acc[32];
#pragma unroll
    for (int s = 0; s < 32; ++s) {
        const int id = __shfl_sync(0xffffffffu, cand, s);
        const float *row = X + int64_t(id >= 0 ? id : self) * ld;
        float a = 0.0f;
#pragma unroll
        for (int j = 0; j < DJ; ++j) {
            const int t = lane + 32 * j;
            if (t < d) {
                const float x = __fsub_rn(__ldg(row + t), xs[j]);
                a = __fmaf_rn(x, x, a);
            }
        }
        acc[s] = a;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = up ? acc[i] : acc[i + o];
            const float keep = up ? acc[i + o] : acc[i];
            acc[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, o));
        }
    }
    return cand >= 0 ? acc[0] : 0.0f;
}

struct RerankArgs {
    const float *X;
    int d, ld, k, kp;
    int64_t nq;
    const int32_t *qrows;
    int64_t q0;
    const uint64_t *part;    // [part][query][kp] lists
    int S;
    float rho;
    int32_t *nbr;
    float *dist;
    int32_t *fail_rows, *fail_count;
    // pruned lists: X in cell order, perm[row] = point, split query tiles (128 rows)
    // tsplit[tile] = entry of splitq (q, first slot, parts) or -1
    const int32_t *perm;
    const int32_t *tsplit, *splitq;
    const uint64_t *side;
    const float *tau, *skipQ;
};

// Canonical re-rank of the FP32 tiles' kp candidates, one warp per query
// row q (point i = qrows[q] or q0 + q): the parts' lists merged, canonical
// distances (32 candidates at a time from coalesced row reads), sort by
// (w, id), certificate. Every unkept point has fast distance >= the kp-th
// kept one's, sp (and, where the lists started from a bound tau, p above
// tau_p(tau)); fast and canonical sums of the same rounded terms differ by a
// factor within 1 +- rho, so an unkept point's canonical distance is at least
// sp (1 - rho) and the row is certified when that, and the smallest distance
// of a key in a skipped tile, exceed the k-th.
template <int H, int DJ>
__global__ void __launch_bounds__(128) rerank_fp32_kernel(RerankArgs A) {
    const int64_t q = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= A.nq) return;
    const int d = A.d, k = A.k, kp = A.kp;
    const float inf = __int_as_float(0x7f800000);
    const int64_t r = A.qrows ? int64_t(A.qrows[q]) : A.q0 + q;   // row of X
    const int64_t i = A.perm ? int64_t(A.perm[r]) : r;            // point
    uint64_t E[H];
#pragma unroll
    for (int h = 0; h < H; ++h) E[h] = KEY_NONE;
    const uint64_t *lists = A.part + size_t(q) * kp;
    size_t step = size_t(A.nq) * kp;
    int S = A.S;
    if (A.perm) {
        const int ts = A.tsplit[q / (2 * QM)];
        S = 1;
        if (ts >= 0) {
            S = A.splitq[3 * ts + 2];
            step = size_t(2 * QM) * kp;
            lists = A.side + (size_t(A.splitq[3 * ts + 1]) * 2 * QM + q % (2 * QM)) * kp;
        }
    }
#pragma unroll
    for (int h = 0; h < H; ++h)
        if (32 * h + lane < kp) E[h] = lists[32 * h + lane];
    for (int s = 1; s < S; ++s) {
        lists += step;
        for (int b = 0; b < kp; b += 32) {
            const uint64_t B = b + lane < kp ? lists[b + lane] : KEY_NONE;
            if (!__any_sync(0xffffffffu, B < warp_list_at<H>(E, kp - 1))) break;
            warp_list_merge<H>(E, B, lane);
        }
    }
    const uint64_t last = warp_list_at<H>(E, kp - 1);
    float sp = last == KEY_NONE ? inf : key_w(last);
    if (A.tau) sp = fminf(sp, __fsqrt_rd(tau_p(A.tau[r], A.rho)));
    uint64_t key[H];
    if constexpr (DJ > 0) {
        float xs[DJ];
#pragma unroll
        for (int j = 0; j < DJ; ++j) {
            const int t = lane + 32 * j;
            xs[j] = t < d ? __ldg(A.X + r * A.ld + t) : 0.0f;
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int e = 32 * h + lane;
            const int cand = e < kp && E[h] != KEY_NONE ? int(key_lo(E[h])) : -1;
            const float p = warp_canon32<DJ>(A.X, A.ld, d, xs, int(r), cand, lane);
            key[h] = cand >= 0 ? nb_key(__fsqrt_rn(p), uint32_t(A.perm ? A.perm[cand] : cand))
                               : KEY_NONE;
        }
    } else {
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int e = 32 * h + lane;
            const int cand = e < kp && E[h] != KEY_NONE ? int(key_lo(E[h])) : -1;
            key[h] = KEY_NONE;
            if (cand >= 0)
                key[h] = nb_key(canon_dist<1>(A.X + r * A.ld, A.X + int64_t(cand) * A.ld, d),
                                uint32_t(A.perm ? A.perm[cand] : cand));
        }
    }
    warp_sort_regs<H>(key, lane);
    const uint64_t kth = warp_list_at<H>(key, k - 1);
    // (FP32, rounded down, decides all but near ties; FP64 the rest)
    bool cert = !(sp < inf) ||
                (kth != KEY_NONE && (__fmul_rd(sp, __fsub_rd(1.0f, A.rho)) > key_w(kth) ||
                                     double(sp) * (1.0 - double(A.rho)) > double(key_w(kth))));
    if (A.skipQ) {   // keys of skipped tiles lie at true distance >= skip
        const float skip = A.skipQ[q / (2 * QM)];
        cert &= !(skip < inf) || (kth != KEY_NONE &&
                                  double(skip) * (1.0 - (d + 4.0) * 0x1p-24 * 1.05) >
                                      double(key_w(kth)));
    }
    if (cert) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int e = h * 32 + lane;
            if (e < k) {
                A.nbr[i * k + e] = key[h] == KEY_NONE ? -1 : int32_t(key_lo(key[h]));
                A.dist[i * k + e] = key[h] == KEY_NONE ? inf : key_w(key[h]);
            }
        }
    } else if (lane == 0) {
        A.fail_rows[atomicAdd(A.fail_count, 1)] = int32_t(i);
    }
}

template <int H>
famst_status launch_rerank_h(const Exec &ex, const RerankArgs &A) {
    const unsigned grid = unsigned((A.nq * 32 + 127) / 128);
    const int dj = (A.d + 31) / 32;
    if (dj <= 1) FAMST_LAUNCH(ex, (rerank_fp32_kernel<H, 1>), grid, 128, 0, A);
    else if (dj <= 2) FAMST_LAUNCH(ex, (rerank_fp32_kernel<H, 2>), grid, 128, 0, A);
    else if (dj <= 4) FAMST_LAUNCH(ex, (rerank_fp32_kernel<H, 4>), grid, 128, 0, A);
    else if (dj <= 8) FAMST_LAUNCH(ex, (rerank_fp32_kernel<H, 8>), grid, 128, 0, A);
    else FAMST_LAUNCH(ex, (rerank_fp32_kernel<H, 0>), grid, 128, 0, A);
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

famst_status launch_rerank(const Exec &ex, const RerankArgs &A) {
    switch (list_regs(A.kp)) {
        case 1: return launch_rerank_h<1>(ex, A);
        case 2: return launch_rerank_h<2>(ex, A);
        default: return launch_rerank_h<4>(ex, A);
    }
}

__global__ void split_index_kernel(const int32_t *__restrict__ splitq,
                                   const int32_t *__restrict__ nsplit,
                                   int32_t *__restrict__ tsplit) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < *nsplit) tsplit[splitq[3 * s]] = s;
}

// Rows whose candidates from a pruned pass could not be certified, exact on
// canonical distances over the keys of their tile's list: VR_PARTS blocks
// per row (rows[] = positions in the cell order Xs), their warps taking 32
// keys at a time, each with its own sorted list; a block writes its k
// smallest, visited_merge_kernel takes the row's. The k-th distance of the
// uncertified candidates bounds the row's from above (kth0), so few keys are
// inserted. Bound: the L2 gathers of the listed rows; a tile that spans two
// clusters lists nearly every key, hence the parts.
constexpr int VR_WARPS = 4, VR_PARTS = 8;
template <int DJ>
__global__ void __launch_bounds__(VR_WARPS * 32)
visited_rows_kernel(const float *__restrict__ Xs, int64_t n, int d, int k,
                    const int32_t *__restrict__ rows, const uint64_t *__restrict__ kth0,
                    const int32_t *__restrict__ off, const int32_t *__restrict__ klist,
                    const int32_t *__restrict__ perm, uint64_t *__restrict__ lists_out) {
    __shared__ uint64_t lists[VR_WARPS][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r = rows[blockIdx.x];
    const int64_t tile = r / (2 * QM);
    const int t0 = off[tile], t1 = off[tile + 1];
    float xs[DJ];
#pragma unroll
    for (int j = 0; j < DJ; ++j) {
        const int t = lane + 32 * j;
        xs[j] = t < d ? __ldg(Xs + r * d + t) : 0.0f;
    }
    uint64_t E[2] = {KEY_NONE, KEY_NONE};
    const uint64_t bound = kth0[blockIdx.x];
    uint64_t kth = bound;
    // a list entry holds eight groups of 32 keys
    for (int g = int(blockIdx.y) * VR_WARPS + warp; g < 8 * (t1 - t0); g += VR_PARTS * VR_WARPS) {
        const int64_t j = int64_t(__ldg(klist + t0 + (g >> 3))) * 256 + 32 * (g & 7) + lane;
        const int cand = j < n && j != r ? int(j) : -1;
        const float p = warp_canon32<DJ>(Xs, d, d, xs, int(r), cand, lane);
        const uint64_t key =
            cand >= 0 ? nb_key(__fsqrt_rn(p), uint32_t(perm[cand])) : KEY_NONE;
        unsigned m = __ballot_sync(0xffffffffu, key <= kth);
        if (!m) continue;
        while (m) {
            warp_list_insert<2>(E, shfl_idx_u64(key, __ffs(m) - 1), lane);
            m &= m - 1;
        }
        const uint64_t mine = warp_list_at<2>(E, k - 1);
        kth = mine < bound ? mine : bound;
    }
    lists[warp][lane] = E[0];
    lists[warp][32 + lane] = E[1];
    __syncthreads();
    if (warp != 0) return;
    for (int w = 1; w < VR_WARPS; ++w) {
        warp_list_merge<2>(E, lists[w][lane], lane);
        warp_list_merge<2>(E, lists[w][32 + lane], lane);
    }
    uint64_t *o = lists_out + (size_t(blockIdx.x) * VR_PARTS + blockIdx.y) * 64;
    o[lane] = E[0];
    o[32 + lane] = E[1];
}

// One warp per row; a row that a skipped tile could still reach goes to
// `fails` (as a point).
__global__ void visited_merge_kernel(const uint64_t *__restrict__ lists, int64_t nrows, int d,
                                     int k, const int32_t *__restrict__ rows,
                                     const float *__restrict__ skipQ,
                                     const int32_t *__restrict__ perm, int32_t *__restrict__ nbr,
                                     float *__restrict__ dist, int32_t *__restrict__ fails,
                                     int32_t *__restrict__ nfails) {
    const int64_t q = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= nrows) return;
    const uint64_t *l = lists + size_t(q) * VR_PARTS * 64;
    uint64_t E[2] = {l[lane], l[32 + lane]};
    for (int b = 2; b < 2 * VR_PARTS; ++b) {
        const uint64_t B = l[32 * b + lane];
        if (__any_sync(0xffffffffu, B != KEY_NONE)) warp_list_merge<2>(E, B, lane);
    }
    const uint64_t kth = warp_list_at<2>(E, k - 1);
    const int64_t r = rows[q], i = perm[r];
    const float skip = skipQ[r / (2 * QM)];
    const bool cert = kth != KEY_NONE &&
                      (!(skip < __int_as_float(0x7f800000)) ||
                       double(skip) * (1.0 - (d + 4.0) * 0x1p-24 * 1.05) > double(key_w(kth)));
    if (!cert) {
        if (lane == 0) fails[atomicAdd(nfails, 1)] = int32_t(i);
        return;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int e = 32 * h + lane;
        if (e < k) {
            nbr[i * k + e] = int32_t(key_lo(E[h]));
            dist[i * k + e] = key_w(E[h]);
        }
    }
}

// Exact kNN of single rows on canonical distances, one warp per row of
// rows[0 .. *count): keys in rounds of 32 (warp_canon32), the k best (w, id)
// in a warp-wide sorted list. colcomp: keys of the row's own component are
// skipped. k <= 128; d <= 32 DJ, or DJ = 0 for any d.
template <int DJ>
__global__ void exact_rows_kernel(const float *__restrict__ X, int64_t n, int d, int k,
                                  const int32_t *__restrict__ rows,
                                  const int32_t *__restrict__ count,
                                  const int32_t *__restrict__ colcomp, int32_t *__restrict__ nbr,
                                  float *__restrict__ dist) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
    const int nrows = *count;
    for (int64_t q = w0; q < nrows; q += nw) {
        const int i = rows[q];
        float xs[DJ > 0 ? DJ : 1];
#pragma unroll
        for (int j = 0; j < DJ; ++j) {
            const int t = lane + 32 * j;
            xs[j] = t < d ? __ldg(X + int64_t(i) * d + t) : 0.0f;
        }
        const int my_comp = colcomp ? colcomp[i] : -1;
        uint64_t L[4] = {KEY_NONE, KEY_NONE, KEY_NONE, KEY_NONE};
        uint64_t kth = KEY_NONE;
        for (int64_t base = 0; base < n; base += 32) {
            const int64_t j = base + lane;
            int cand = (j < n && j != i) ? int(j) : -1;
            if (cand >= 0 && colcomp && colcomp[cand] == my_comp) cand = -1;
            if (__ballot_sync(0xffffffffu, cand >= 0) == 0u) continue;
            float p;
            if constexpr (DJ > 0) {
                p = warp_canon32<DJ>(X, d, d, xs, i, cand, lane);
            } else {   // any d: one key at a time, the whole warp per key
                p = 0.0f;
                for (int s = 0; s < 32; ++s) {
                    const int id = __shfl_sync(0xffffffffu, cand, s);
                    const float ps = canon_p_warp(X + int64_t(i) * d,
                                                  X + int64_t(id >= 0 ? id : i) * d, d, lane);
                    if (lane == s) p = ps;
                }
            }
            const uint64_t key = cand >= 0 ? nb_key(__fsqrt_rn(p), uint32_t(cand)) : KEY_NONE;
            unsigned pass = __ballot_sync(0xffffffffu, key < kth);
            while (pass) {
                const int s = __ffs(pass) - 1;
                pass &= pass - 1;
                const uint64_t K = shfl_idx_u64(key, s);
                if (K < kth) {
                    warp_list_insert<4>(L, K, lane);
                    kth = shfl_idx_u64(L[(k - 1) >> 5], (k - 1) & 31);
                }
            }
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int e = h * 32 + lane;
            if (e < k) {
                nbr[int64_t(i) * k + e] = L[h] == KEY_NONE ? -1 : int32_t(key_lo(L[h]));
                dist[int64_t(i) * k + e] = L[h] == KEY_NONE ? __int_as_float(0x7f800000) : key_w(L[h]);
            }
        }
    }
}

__device__ __forceinline__ int cloud_index(const long long *__restrict__ off, int B, long long v) {
    int lo = 0, hi = B;  // off[lo] <= v < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= v) lo = mid; else hi = mid;
    }
    return lo;
}

// Batched canonical re-rank: one block per FP32 tile, a warp per row; rows,
// ids and the distance rows live in the compact space Xc (row stride ld,
// zero beyond each cloud's d). The same certificate as rerank_fp32_kernel.
__global__ void rerank_fp32_batched_kernel(const float *__restrict__ Xc, int ld,
                                           const long long *__restrict__ voff, int B,
                                           const CloudDev *__restrict__ cl, int k, int kp,
                                           const F32Tile *__restrict__ tiles,
                                           const int32_t *__restrict__ cand,
                                           const float *__restrict__ wf, int32_t *__restrict__ nbr,
                                           float *__restrict__ dist, int32_t *__restrict__ fails,
                                           int32_t *__restrict__ nfail) {
    const F32Tile T = tiles[blockIdx.x];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int q = wib; q < T.nq; q += blockDim.x >> 5) {
        const int64_t v = int64_t(T.qbase) + q;
        const CloudDev c = cl[cloud_index(voff, B, v)];
        const int dc = (c.d + 3) & ~3;
        const double u = 1.0 / 16777216.0, nu = double(dc + 9) * u;
        const double rho = 2.01 * nu / (1.0 - nu) + 4.0 * u;
        const float *xi = Xc + v * ld;
        uint64_t key[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int p = h * 32 + lane;
            key[h] = KEY_NONE;
            if (p < kp) {
                const int j = cand[v * kp + p];
                if (j >= 0) key[h] = nb_key(canon_dist<4>(xi, Xc + int64_t(j) * ld, dc), uint32_t(j));
            }
        }
        warp_sort_regs<4>(key, lane);
        const uint64_t kth = shfl_idx_u64(key[(k - 1) >> 5], (k - 1) & 31);
        const int jl = cand[v * kp + kp - 1];
        const float sp = jl >= 0 ? wf[v * kp + kp - 1] : __int_as_float(0x7f800000);
        const bool cert = !(sp < __int_as_float(0x7f800000)) ||
                          (kth != KEY_NONE && double(sp) * (1.0 - rho) > double(key_w(kth)));
        if (cert) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int e = h * 32 + lane;
                if (e < k) {
                    nbr[v * k + e] = key[h] == KEY_NONE ? -1 : int32_t(key_lo(key[h]));
                    dist[v * k + e] = key[h] == KEY_NONE ? __int_as_float(0x7f800000) : key_w(key[h]);
                }
            }
        } else if (lane == 0) {
            fails[atomicAdd(nfail, 1)] = int32_t(v);
        }
    }
}

struct SplitPlan {
    int qblocks, S, tiles_per_split;
};

// Two blocks fit an SM. Few query blocks: the key range is split, down to two
// key tiles per block, until the grid is about eight rounds of the chip (a
// nearly empty last round then costs at most an eighth); every part fills its
// own lists, so large grids are not split.
constexpr int ROUNDS = 8;
SplitPlan plan(int64_t n, int64_t nq, int num_sms) {
    SplitPlan p;
    p.qblocks = int((nq + QM - 1) / QM);
    const int ntiles = int((n + KN - 1) / KN);
    const int slots = 2 * num_sms;
    int S = (ROUNDS * slots + p.qblocks - 1) / p.qblocks;
    S = std::min(S, std::max(1, ntiles / 2));
    // at most one round, when two tiles per block would make a little more
    if (p.qblocks * S > slots && p.qblocks * S < 2 * slots) S = std::max(1, slots / p.qblocks);
    p.tiles_per_split = (ntiles + S - 1) / S;
    p.S = (ntiles + p.tiles_per_split - 1) / p.tiles_per_split;
    return p;
}

}  // namespace

int fp32_kp(int64_t n, int k) {
    int64_t kp = k + FP32_MARGIN;
    if (kp > n - 1) kp = n - 1;
    if (kp > 128) kp = 128;
    return int(kp < k ? k : kp);
}

// for any number of query rows up to nq: S nq' <= ROUNDS slots QM + nq'
size_t knn_fp32_workspace(int64_t n, int d, int k, int64_t nq, int num_sms) {
    (void)d;
    const size_t lists = size_t(ROUNDS) * 2 * num_sms * QM + size_t(nq);
    return align256(size_t(nq) * 4) * 2 + 256 + align256(lists * fp32_kp(n, k) * sizeof(uint64_t));
}

size_t knn_fp32_pruned_workspace(int64_t n, int k, int64_t nq_tiles) {
    const size_t kp = size_t(fp32_kp(n, k));
    return align256(size_t(n) * kp * 8) + align256(size_t(PRUNE_SPLIT_SLOTS) * 2 * QM * kp * 8) +
           align256(size_t(nq_tiles) * 4) + align256(size_t(n) * 4) + 256;
}

famst_status exact_rows(const Exec &ex, const float *X, int64_t n, int d, int k,
                        const int32_t *rows, const int32_t *count, int64_t max_rows,
                        const int32_t *colcomp, int32_t *nbr, float *dist) {
    if (max_rows == 0) return FAMST_OK;
    if (k < 1 || k > 128) return FAMST_ERR_UNSUPPORTED;
    int64_t warps = max_rows < int64_t(ex.num_sms) * 16 ? max_rows : int64_t(ex.num_sms) * 16;
    const unsigned grid = unsigned((warps * 32 + 127) / 128);
    const int dj = (d + 31) / 32;
#define EXACT(DJV)                                                                              \
    FAMST_LAUNCH(ex, exact_rows_kernel<DJV>, grid, 128, 0, X, n, d, k, rows, count, colcomp, nbr, \
                 dist)
    if (dj <= 1) EXACT(1);
    else if (dj <= 2) EXACT(2);
    else if (dj <= 4) EXACT(4);
    else if (dj <= 8) EXACT(8);
    else if (dj <= 16) EXACT(16);
    else EXACT(0);
#undef EXACT
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

famst_status knn_fp32(const Exec &ex, Arena &ar, const float *X, int64_t n, int d, int k,
                      const int32_t *qrows, int64_t q0, int64_t nq, int32_t *nbr, float *dist,
                      const int32_t *colcomp) {
    if (nq == 0) return FAMST_OK;
    if (k < 1 || k > 128 || k > n - 1) return FAMST_ERR_UNSUPPORTED;
    const int kp = fp32_kp(n, k);
    const SplitPlan p = plan(n, nq, ex.num_sms);
    int32_t *fails = ar.take<int32_t>(size_t(nq));
    int32_t *nfail = ar.take<int32_t>(1);
    uint64_t *part = ar.take<uint64_t>(size_t(p.S) * nq * kp);
    if (!fails || !nfail || !part) return FAMST_ERR_OOM;
    TileArgs T{};
    T.X = X; T.n = int(n); T.d = d; T.ld = d; T.kp = kp;
    T.qrows = qrows; T.q0 = q0; T.nq = int(nq);
    T.tiles_per_split = p.tiles_per_split;
    T.part = part;
    T.colcomp = colcomp;
    if (p.S > 1) {
        T.thr_g = ar.take<unsigned>(size_t(nq));
        if (!T.thr_g) return FAMST_ERR_OOM;
        if (cudaMemsetAsync(T.thr_g, 0xff, size_t(nq) * 4, ex.stream) != cudaSuccess)
            return FAMST_ERR_CUDA;
    }
    famst_status st = launch_tiles(ex, dim3(p.qblocks, p.S), T);
    if (st != FAMST_OK) return st;
    if (cudaMemsetAsync(nfail, 0, 4, ex.stream) != cudaSuccess) return FAMST_ERR_CUDA;
    RerankArgs R{};
    R.X = X; R.d = d; R.ld = d; R.k = k; R.kp = kp; R.nq = nq; R.qrows = qrows; R.q0 = q0;
    R.part = part; R.S = p.S; R.rho = fast_rho(d, 1);
    R.nbr = nbr; R.dist = dist; R.fail_rows = fails; R.fail_count = nfail;
    st = launch_rerank(ex, R);
    if (st != FAMST_OK) return st;
    return exact_rows(ex, X, n, d, k, fails, nfail, nq, colcomp, nbr, dist);
}

// The FP32 tiles over the pruning's work items (points in cell order): every
// row of X, each starting from its bound tau on the k-th distance.
famst_status knn_fp32_pruned(const Exec &ex, Arena &ar, const float *X, int64_t n, int d, int k,
                             const PruneOut &P, int32_t *nbr, float *dist) {
    const int kp = fp32_kp(n, k);
    uint64_t *part = ar.take<uint64_t>(size_t(n) * kp);
    uint64_t *side = ar.take<uint64_t>(size_t(PRUNE_SPLIT_SLOTS) * 2 * QM * kp);
    int32_t *tsplit = ar.take<int32_t>(size_t(P.nq));
    int32_t *fails = ar.take<int32_t>(size_t(n));
    int32_t *nfail = ar.take<int32_t>(1);
    if (!part || !side || !tsplit || !fails || !nfail) return FAMST_ERR_OOM;
    if (cudaMemsetAsync(tsplit, 0xff, size_t(P.nq) * 4, ex.stream) != cudaSuccess ||
        cudaMemsetAsync(nfail, 0, 4, ex.stream) != cudaSuccess)
        return FAMST_ERR_CUDA;
    FAMST_LAUNCH(ex, split_index_kernel, (PRUNE_SPLIT_TILES + 255) / 256, 256, 0, P.splitq,
                 P.nsplit, tsplit);
    TileArgs T{};
    T.X = P.Xs; T.n = int(n); T.d = d; T.ld = d; T.kp = kp; T.nq = int(n);
    T.part = part; T.side = side;
    T.items = P.tab; T.nitems = P.nitems; T.klist = P.klist;
    T.tau = P.tau_row; T.rho = fast_rho(d, 1);
    famst_status st =
        launch_tiles(ex, dim3(unsigned(2 * (P.nq + PRUNE_SPLIT_SLOTS))), T);
    if (st != FAMST_OK) return st;
    RerankArgs R{};
    R.X = P.Xs; R.d = d; R.ld = d; R.k = k; R.kp = kp; R.nq = n;
    R.part = part; R.S = 1; R.rho = T.rho;
    R.nbr = nbr; R.dist = dist; R.fail_rows = fails; R.fail_count = nfail;
    R.perm = P.perm; R.tsplit = tsplit; R.splitq = P.splitq; R.side = side;
    R.tau = P.tau_row; R.skipQ = P.skipQ;
    st = launch_rerank(ex, R);
    if (st != FAMST_OK) return st;
    return exact_rows(ex, X, n, d, k, fails, nfail, n, nullptr, nbr, dist);
}

size_t visited_rows_workspace(int64_t nrows) {
    return align256(size_t(nrows) * VR_PARTS * 64 * sizeof(uint64_t));
}

famst_status visited_rows(const Exec &ex, Arena &ar, const PruneOut &P, int64_t n, int d, int k,
                          const int32_t *rows, const uint64_t *kth0, int64_t nrows, int32_t *nbr,
                          float *dist, int32_t *fails, int32_t *nfails) {
    if (nrows == 0) return FAMST_OK;
    const int dj = (d + 31) / 32;
    if (k > 64 || dj > 16) return FAMST_ERR_UNSUPPORTED;
    uint64_t *lists = ar.take<uint64_t>(size_t(nrows) * VR_PARTS * 64);
    if (!lists) return FAMST_ERR_OOM;
#define VISITED(DJV)                                                                             \
    FAMST_LAUNCH(ex, visited_rows_kernel<DJV>, dim3(unsigned(nrows), VR_PARTS), VR_WARPS * 32, 0, \
                 P.Xs, n, d, k, rows, kth0, P.off, P.klist, P.perm, lists)
    if (dj <= 1) VISITED(1);
    else if (dj <= 2) VISITED(2);
    else if (dj <= 4) VISITED(4);
    else if (dj <= 8) VISITED(8);
    else VISITED(16);
    FAMST_LAUNCH(ex, visited_merge_kernel, unsigned((nrows * 32 + 127) / 128), 128, 0, lists, nrows,
                 d, k, rows, P.skipQ, P.perm, nbr, dist, fails, nfails);
#undef VISITED
    return cudaPeekAtLastError() == cudaSuccess ? FAMST_OK : FAMST_ERR_CUDA;
}

}  // namespace famst

namespace famst {

// Batched exact kNN on FP32 tiles: one block per entry of `tiles` (64 query
// rows of one cloud against that cloud's keys) keeps kp candidates per row,
// then the batched canonical re-rank, then exact rows for the uncertified.
famst_status knn_fp32_batched(const Exec &ex, const float *Xc, int ld, const long long *voff,
                              int B, const CloudDev *cl, int k, int kp, const F32Tile *tiles,
                              int64_t nblocks, int32_t *c, float *w, int32_t *fails,
                              int32_t *nfail, int32_t *nbr, float *dist) {
    if (nblocks == 0) return FAMST_OK;
    if (k < 1 || k > 64 || kp < k || kp > 128) return FAMST_ERR_UNSUPPORTED;
    TileArgs T{};
    T.X = Xc; T.ld = ld; T.kp = kp; T.nbr = c; T.dist = w; T.btab = tiles;
    famst_status st = launch_tiles(ex, dim3(unsigned(nblocks)), T);
    if (st != FAMST_OK) return st;
    if (cudaMemsetAsync(nfail, 0, 4, ex.stream) != cudaSuccess) return FAMST_ERR_CUDA;
    FAMST_LAUNCH(ex, rerank_fp32_batched_kernel, unsigned(nblocks), 256, 0, Xc, ld, voff, B, cl, k,
                 kp, tiles, c, w, nbr, dist, fails, nfail);
    if (cudaPeekAtLastError() != cudaSuccess) return FAMST_ERR_CUDA;
    return fallback_rows_batched(ex, Xc, ld, voff, B, cl, k, fails, nfail, nbr, dist);
}

}  // namespace famst
