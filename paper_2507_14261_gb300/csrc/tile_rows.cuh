// Rows of the tensor tiles' work items (knn_tc.cu): which row stands at a place
// of a key tile, where a row's candidate count and bound go, and what stands
// there when its tiles were given up.
//
// Host and device: the CPU tests compile this header with a host compiler.
#pragma once

#include <cstddef>
#include <cstdint>
#include <limits>

#if defined(__CUDACC__)
#define TILE_HD __host__ __device__ __forceinline__
#else
#define TILE_HD inline
#endif

namespace famst {
namespace tile {

constexpr int ROWS = 128;   // query rows of a work item

// Row `row` (0 .. ROWS - 1) of an item that starts at padded row q0: its entry
// in the per-row arrays (compact id = padded row - shift), or, for part s + 1
// of a split key list, its entry in side slot s.
struct RowSlot {
    bool side;
    size_t at;
};
TILE_HD RowSlot row_slot(int q0, int row, int shift, int part) {
    RowSlot r;
    r.side = part > 0;
    r.at = part > 0 ? size_t(part - 1) * ROWS + size_t(row) : size_t(q0 + row - shift);
    return r;
}

// A row whose tiles were not finished (a bounded wait gave up, or no scratch
// area was free) has no candidates and is never certified: the kernels that
// follow in the stream use the counts as loop bounds before the host has read
// the status word, and recompute the row.
TILE_HD void give_up_row(RowSlot s, int32_t *cnt, float *splus, int32_t *side_cnt,
                         float *side_splus) {
    (s.side ? side_cnt : cnt)[s.at] = 0;
    (s.side ? side_splus : splus)[s.at] = -std::numeric_limits<float>::infinity();
}

constexpr int KEYS = 256;   // rows of a key tile

// A permutation of [0, n) without structure: which row stands at position
// `pos` (products with odd numbers, sums and xor-shifts modulo 2^b permute
// [0, 2^b); a value beyond n steps on until it is back inside, less than one
// step in the mean). Another `salt`, another permutation. (The odd numbers: 2^32
// over the golden ratio, as in Knuth's multiplicative hashing, and the two
// multipliers of A. Appleby's MurmurHash3 finaliser.)
//
// The tiles' threshold is the largest of four column groups' R-th scores
// (columns 16 g .. 16 g + 15 of every 64): tight when a row's near keys are
// spread over the groups, and soon when they do not come last. Rows as they
// come have neither. Where the index has a period (a pixel grid 64 wide, labels
// i mod 32, a signal of 64 samples a period) all near keys are in one or two
// groups, far ones set the threshold, hundreds of keys lie below it, and 40 to
// 100 % of the rows lose their certificate and are computed twice; where points
// come in spatial order every tile improves on the one before. In this order
// 22 to 64 keys end up below the threshold, whatever the rows. As they come /
// scrambled: a grid 64 wide, 3,968 x 3, k = 10 2.10 / 0.20 ms, its exact tree
// 11.4 / 1.35; 9,000 x 5 4.9 / 0.29 and 30 / 2.1; labels i mod 32, 8,000 x 5 1.14
// / 0.37 and 6.3 / 2.0; a random walk of 8,000 x 15 1.6 / 0.27 and 11.7 / 2.2.
// Rows already in random order: the same time.
TILE_HD int scrambled_row(int pos, int n, uint32_t salt = 0) {
#if defined(__CUDA_ARCH__)
    const int b = 32 - __clz(n - 1);
#else
    int b = 0;
    while ((int64_t(1) << b) < n) ++b;
#endif
    const uint32_t mask = (1u << b) - 1u;
    const int s = b < 2 ? 1 : (b + 1) / 2;
    uint32_t h = (salt + 1u) * 0x9E3779B1u;
    h = (h ^ (h >> 15)) * 0x85EBCA6Bu;
    h = (h ^ (h >> 13)) * 0xC2B2AE35u;
    h ^= h >> 16;
    uint32_t x = uint32_t(pos);
    do {
        x = (x * 0x9E3779B1u + h) & mask;
        x ^= x >> s;
        x = (x * 0x85EBCA6Bu + (h >> 8)) & mask;
        x ^= x >> s;
        x = (x * 0xC2B2AE35u + (h >> 16)) & mask;
        x ^= x >> s;
    } while (x >= uint32_t(n));
    return int(x);
}

}  // namespace tile
}  // namespace famst
