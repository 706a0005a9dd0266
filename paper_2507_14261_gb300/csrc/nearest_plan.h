// Sizes of the nearest-pair connect's buffers (connect_nearest.cu). Host only,
// so that they can be checked without a GPU over the whole range of calls:
// lambda t (t - 1) / 2 < 2^31 with 1 <= lambda <= 32.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace famst {

inline int64_t nearest_pairs(int64_t t) { return t * (t - 1) / 2; }

// The warp kernel's lists: sum over i of ceil(|C_i| / 32) (t - 1 - i)
// <= (n / 32 + t) t lists of lambda (u, v, w).
inline size_t nearest_warp_bytes(int64_t n, int64_t t, int lambda) {
    return size_t(n / 32 + t) * size_t(t) * size_t(lambda) * 12;
}

// Survivors of the tensor pass: two rows, a bound, an arrival number, a pair.
constexpr size_t NEAREST_SURVIVOR_BYTES = 24;

// bounds and slots, counts and offsets of the component pairs
inline size_t nearest_pair_bytes(int64_t t, int lambda) {
    return size_t(nearest_pairs(t)) * (size_t(lambda) * 4 + 12);
}

// Whether a call takes the tensor pass, and its room for survivors. No more
// memory than the warp kernel's lists would take and 1.6 GB, and always fewer
// than 2^31, so that 32-bit counts and offsets hold.
//
// Survivors per component pair, measured on sphere and blob clouds (100k to 1M
// points, 50 to 1000 components), in one search / in a search after a launch
// over the first 128 rows of every component that only lowers the bounds:
// lambda 1 133 / 42, lambda 5 510 / 140, lambda 10 893 / 402, lambda 32 1500 /
// 600 (most of them while only the sample's bound is known, so the second form
// needs a third of the room and 5 to 15 % more time). A pass whose survivors do
// not fit is thrown away, and the fewer points a component has, the less the
// pass gains (its tiles hold 128 rows of one component). Warp kernel / tensor
// pass: 100k x 128, lambda 5, 50 components 33.1 / 3.1 ms, 200 39.5 / 10.5, 800
// 56 / 47, 1600 73 / 130; 20k x 128, lambda 1, 600 components 10.1 / 7.2, 1200
// 11.7 / 15.3; 1M x 128, lambda 10, 1000 components 2514 / 690. So the pass runs
// where the room holds about half as much again as was measured and, in its
// second form, a component has 32 points or more on average; the warp kernel
// takes the rest.
struct NearestPlan {
    bool tensor = false;
    bool bounds_first = false;
    int64_t cap = 0;
};

inline NearestPlan nearest_plan(int64_t n, int64_t t, int lambda) {
    const int64_t pairs = nearest_pairs(t), all = n * (n - 1) / 2 + 1;
    const size_t warp = nearest_warp_bytes(n, t, lambda), pair = nearest_pair_bytes(t, lambda);
    const int64_t room = std::min(
        int64_t((warp > pair ? warp - pair : 0) / NEAREST_SURVIVOR_BYTES) + (int64_t(1) << 26),
        int64_t(1) << 30);
    const int64_t once = std::min(all, (int64_t(1) << 22) + (128 + 128 * lambda) * pairs);
    NearestPlan p;
    if (once <= room) {
        p.tensor = true;
        p.cap = once;
    } else if ((64 + 28 * lambda) * pairs <= room && n >= 32 * t) {
        p.tensor = p.bounds_first = true;
        p.cap = std::min(room, (int64_t(1) << 22) + 2 * (64 + 28 * lambda) * pairs);
    }
    return p;
}

}  // namespace famst
