// A warp's interaction list in shared memory: four arrays (x, y, z, m) of `cap` entries from lx on.  The parts whose
// order between the lanes matters, apart from the kernels so that a host program can run them lane by lane.
#pragma once

#include <stdint.h>

// Entry e of a window whose first entry lies at slot `to` less the entries before it: `to` may have wrapped below
// zero, so the two are added as 32-bit numbers before they meet the pointer.
__host__ __device__ __forceinline__ float *list_at(float *lx, uint32_t to, uint32_t e) { return lx + (uint32_t)(to + e); }

// Every full chunk of the list is summed (sum(k0, k1): quads k0 to k1 by all lanes), then the rest, fewer than CHUNK
// entries from a later quad on, is moved to the front.  The list's number of entries becomes the rest's; returns the
// chunks summed.  A lane reads entries that other lanes wrote and writes ones that others read, so the warp meets
// before the sums, between the sums and the move, and after it.
template <uint32_t CHUNK, class Warp, class Sum>
__host__ __device__ __forceinline__ uint32_t flush_chunks(float *lx, uint32_t cap, uint32_t &list_n, const Warp &warp,
                                                          Sum sum) {
    warp.sync();
    const uint32_t full = list_n / CHUNK, lane = warp.lane();
    for (uint32_t c = 0; c < full; c++) sum(c * (CHUNK / 4), (c + 1) * (CHUNK / 4));
    list_n -= full * CHUNK;
    if (full) {
        warp.sync();
        if (4u * lane < list_n) {
            float4 *q = (float4 *)lx;
            const uint32_t from = full * (CHUNK / 4);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
            for (uint32_t c = 0; c < 4; c++) q[c * (cap / 4) + lane] = q[c * (cap / 4) + from + lane];
        }
    }
    warp.sync();
    return full;
}
