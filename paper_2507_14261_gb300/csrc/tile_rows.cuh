// Rows of the tensor tiles' work items (knn_tc.cu): where a row's candidate
// count and bound go, and what stands there when its tiles were given up.
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

}  // namespace tile
}  // namespace famst
