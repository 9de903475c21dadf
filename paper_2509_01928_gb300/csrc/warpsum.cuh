// Sum over a warp of 32-bit terms whose sum does not fit 32 bits.
#pragma once

namespace doch {

// the sum of v over the warp's 32 lanes, in every lane: two 32-bit reductions, of the upper and the lower
// 16 bits (|sums| < 2^21), instead of five 64-bit shuffles and additions
__device__ __forceinline__ long long warp_sum_wide(int v) {
    const int hi = __reduce_add_sync(0xffffffffu, v >> 16);
    const unsigned lo = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(v) & 0xffffu);
    return static_cast<long long>(hi) * 65536 + lo;
}

}  // namespace doch
