// Digit counts of the radix sort's passes, gathered by the kernel that reads or makes the keys (blocks of
// GT_SORT_DIGITS threads).
#pragma once

#include "gt_internal.cuh"

// One key per lane into the block's counts.  The keys of a tree rebuild arrive nearly sorted (the particles are
// still in the previous key order), so a warp's 32 neighbouring keys often share their high digits: such a digit
// is counted once for the whole warp, the others by one atomic per lane.
__device__ __forceinline__ void gt_count_digits(unsigned long long k, bool ok, uint32_t (*h)[GT_SORT_DIGITS]) {
    const uint32_t lo = (uint32_t)k, hi = (uint32_t)(k >> 32);
    // bits in which some lane's key differs from the first one's (a lane without a key: all)
    const uint32_t lo0 = __shfl_sync(0xffffffffu, lo, 0), hi0 = __shfl_sync(0xffffffffu, hi, 0);
    const uint32_t dlo = __reduce_or_sync(0xffffffffu, ok ? lo ^ lo0 : ~0u);
    const uint32_t dhi = __reduce_or_sync(0xffffffffu, ok ? hi ^ hi0 : ~0u);
    static_assert(GT_SORT_BITS == 8 && GT_SORT_PASSES == 8, "a byte per digit");
#pragma unroll
    for (int p = 0; p < GT_SORT_PASSES; p++) {
        const uint32_t word = p < 4 ? lo : hi, d = (word >> (8 * (p & 3))) & 0xffu;
        if ((((p < 4 ? dlo : dhi) >> (8 * (p & 3))) & 0xffu) == 0u) {
            if ((threadIdx.x & 31) == 0) atomicAdd(&h[p][d], 32u);
        } else if (ok) {
            atomicAdd(&h[p][d], 1u);
        }
    }
}

// The block's counts into the global ones; the last block to come turns them into every pass's digit starts (a
// launch of its own for that took 7 to 8 us) and resets the passes' tile tickets.
__device__ __forceinline__ void gt_finish_digits(const uint32_t (*h)[GT_SORT_DIGITS], uint32_t *hist, uint32_t *base,
                                                 DevCtl *ctl) {
    __shared__ bool last;
    __syncthreads();
    for (int p = 0; p < GT_SORT_PASSES; p++)
        if (h[p][threadIdx.x]) atomicAdd(&hist[p * GT_SORT_DIGITS + threadIdx.x], h[p][threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ctl->digits_done, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    static_assert(GT_SORT_DIGITS == 32 * GT_SORT_PASSES, "a warp per pass, eight digits per lane");
    const uint32_t p = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    uint32_t v[8], sum = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        v[j] = __ldcg(&hist[p * GT_SORT_DIGITS + 8 * lane + j]);
        sum += v[j];
    }
    uint32_t at = warp_incl_scan(sum) - sum;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        base[p * GT_SORT_DIGITS + 8 * lane + j] = at;
        at += v[j];
    }
    if (threadIdx.x < GT_SORT_PASSES) ctl->sort_ticket[threadIdx.x] = 0;
    if (threadIdx.x == 0) ctl->digits_done = 0;
}
