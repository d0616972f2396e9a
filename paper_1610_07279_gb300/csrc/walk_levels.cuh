// Forces whose block-step level the order of their sums may decide.
#pragma once

#include "keys_quant.cuh"

// Whether x = |a|^2 / c^2 is within 2^-17 of a power of 16, a threshold of the levels, on either side: 64 units in the last
// place above it, 128 of the smaller ones below.  The rounding errors of a sum of FP32 terms scale with the terms' sum of
// magnitudes: where that is up to some 30 |a| they are below the window, where the terms cancel further (the centre of a
// halo, the plane of a disk) a force outside of it may still cross a threshold with the order of its sums.
__host__ __device__ __forceinline__ bool near_level(float x) {
    const uint32_t b = gtq_bits(x), e = b >> 23, m = b & 0x7fffffu;
    if (e == 0u || e >= 255u) return false;
    return (m <= 64u && ((e - 127u) & 3u) == 0u) || (m >= 0x800000u - 128u && ((e - 126u) & 3u) == 0u);
}
