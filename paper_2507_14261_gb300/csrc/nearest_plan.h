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

// Room for the survivors. A call whose survivors need more goes to the warp
// kernel, so this is a matter of speed: no more memory than the warp kernel
// itself would take, or 400 MB where that is little, and always fewer than
// 2^31, so that 32-bit counts and offsets hold.
inline int64_t nearest_cap(int64_t n, int64_t t, int lambda) {
    const int64_t wanted = (int64_t(1) << 22) + 64 * nearest_pairs(t);
    const size_t warp = nearest_warp_bytes(n, t, lambda), pair = nearest_pair_bytes(t, lambda);
    const int64_t room =
        int64_t((warp > pair ? warp - pair : 0) / NEAREST_SURVIVOR_BYTES) + (int64_t(1) << 24);
    return std::min({wanted, room, int64_t(1) << 30, n * (n - 1) / 2 + 1});
}

}  // namespace famst
