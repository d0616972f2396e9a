// Digit counts of the radix sort's passes, gathered by the kernel that reads or makes the keys (blocks of
// GT_SORT_DIGITS threads), and the ranking of keys by a digit.
#pragma once

#include "gt_internal.cuh"

// Where the digits of the tree's keys begin: two for the lowest 15 bits (the second reaches one bit into the next,
// which changes nothing), six for the 48 above (16 levels of the tree).
__host__ __device__ constexpr int gt_tree_digit_shift(int p) { return p < 2 ? 8 * p : 8 * p - 1; }

// One key per lane into the block's counts.  The keys of a tree rebuild arrive nearly sorted (the particles are
// still in the previous key order), so a warp's 32 neighbouring keys often share their high digits: such a digit
// is counted once for the whole warp, the others by one atomic per lane.  TREE: the digits of the tree's keys.
template <bool TREE>
__device__ __forceinline__ void gt_count_digits(unsigned long long k, bool ok, uint32_t (*h)[GT_SORT_DIGITS]) {
    static_assert(GT_SORT_BITS == 8 && GT_SORT_PASSES == 8, "a byte per digit");
    const unsigned long long high = TREE ? k << 1 : k;  // digits 2 to 7 (of the tree's keys) are bytes of this
    const uint32_t lo = (uint32_t)high, hi = (uint32_t)(high >> 32);
    // bits in which some lane's key differs from the first one's (a lane without a key: all)
    const uint32_t lo0 = __shfl_sync(0xffffffffu, lo, 0), hi0 = __shfl_sync(0xffffffffu, hi, 0);
    const uint32_t dlo = __reduce_or_sync(0xffffffffu, ok ? lo ^ lo0 : ~0u);
    const uint32_t dhi = __reduce_or_sync(0xffffffffu, ok ? hi ^ hi0 : ~0u);
#pragma unroll
    for (int p = 0; p < GT_SORT_PASSES; p++) {
        const uint32_t word = p < 4 ? lo : hi;
        const uint32_t d = TREE && p < 2 ? (uint32_t)(k >> (8 * p)) & 0xffu : (word >> (8 * (p & 3))) & 0xffu;
        // (a low digit of the tree's keys lies in the bits 1 to 16 of lo)
        const uint32_t differ = TREE && p < 2 ? (dlo >> (8 * p + 1)) & 0xffu
                                              : ((p < 4 ? dlo : dhi) >> (8 * (p & 3))) & 0xffu;
        if (differ == 0u) {
            if ((threadIdx.x & 31) == 0) atomicAdd(&h[p][d], 32u);
        } else if (ok) {
            atomicAdd(&h[p][d], 1u);
        }
    }
}

// Whether the tree's keys are sorted by all of their bits (eight passes) or by the highest 48 (six, and the runs of keys
// that agree there put in order), from the six digits' counts, each the largest and the sum of squared shares:
// - no run is longer than the smallest of the six largest counts.  From a hundredth of the keys on, the block that
//   sorts the longest run by itself may take longer than two passes over all keys (2^24: ~0.7 ms, 0.29 ms).  (Uniform
//   digits: 1/250 of 2^20 keys, 1/185 of 16384.)
// - a key's run has about n times the product of the squares' sums keys, if the digits are independent.  For Plummer
//   spheres of 2^17 to 2^22 with one particle so far off that the cells of level 16 hold several others, the estimate
//   is 1.3 to 1.4 where a sixth of the tiles hold a run of more than 16 keys, 2.5 to 4.5 where half or more do, and at most
//   0.2 where none do; below 10^-4 for the models.  From half of the tiles on, two passes are the faster way.
constexpr float GT_RUN_SHARE = 0.01f, GT_RUN_MEAN = 2.0f;

// The block's counts into the global ones; the last block to come turns them into every pass's digit starts (a
// launch of its own for that took 7 to 8 us), resets the passes' tile tickets, and makes the choice above (n: the number
// of keys).
__device__ __forceinline__ void gt_finish_digits(unsigned nb, const uint32_t (*h)[GT_SORT_DIGITS], long long n,
                                                 uint32_t *hist, uint32_t *base, DevCtl *ctl) {
    __shared__ bool last;
    __shared__ uint32_t most_sh[GT_SORT_PASSES];
    __shared__ float squares_sh[GT_SORT_PASSES];
    __syncthreads();
    for (int p = 0; p < GT_SORT_PASSES; p++)
        if (h[p][threadIdx.x]) atomicAdd(&hist[p * GT_SORT_DIGITS + threadIdx.x], h[p][threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ctl->digits_done, 1u) == nb - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    static_assert(GT_SORT_DIGITS == 32 * GT_SORT_PASSES, "a warp per pass, eight digits per lane");
    const uint32_t p = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const float share = 1.0f / (float)n;
    uint32_t v[8], sum = 0, most = 0;
    float squares = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        v[j] = __ldcg(&hist[p * GT_SORT_DIGITS + 8 * lane + j]);
        sum += v[j];
        most = max(most, v[j]);
        squares += (v[j] * share) * (v[j] * share);
    }
    most = __reduce_max_sync(0xffffffffu, most);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) squares += __shfl_xor_sync(0xffffffffu, squares, o);
    if (lane == 0) {
        most_sh[p] = most;
        squares_sh[p] = squares;
    }
    uint32_t at = warp_incl_scan(sum) - sum;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        base[p * GT_SORT_DIGITS + 8 * lane + j] = at;
        at += v[j];
    }
    __syncthreads();
    if (threadIdx.x < GT_SORT_PASSES) ctl->sort_ticket[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        uint32_t longest = 0xffffffffu;
        float run = (float)n;
        for (int k = 2; k < GT_SORT_PASSES; k++) {
            longest = min(longest, most_sh[k]);
            run *= squares_sh[k];
        }
        ctl->sort_whole = longest * share >= GT_RUN_SHARE || run >= GT_RUN_MEAN ? 1u : 0u;
        ctl->digits_done = ctl->run_count = 0;
    }
}

// Stable rank of a lane's digit among those that the warp has counted into cnt (a count per digit) and its lower
// lanes; the warp's digits are then counted too.  FULL: every lane has one; otherwise one without has GT_SORT_DIGITS.
template <bool FULL>
__device__ __forceinline__ uint32_t gt_rank_digit(uint32_t d, uint32_t *cnt) {
    const bool ok = FULL || d < GT_SORT_DIGITS;
    unsigned int peers = 0xffffffffu;  // lanes with the same digit (bit 8: none)
#pragma unroll
    for (int b = 0; b < (FULL ? GT_SORT_BITS : GT_SORT_BITS + 1); b++) {
        const unsigned int bal = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        peers &= ((d >> b) & 1u) ? bal : ~bal;
    }
    const unsigned int rank = __popc(peers & lanemask_lt());
    unsigned int prev = 0;
    if (ok) prev = cnt[d];
    __syncwarp();
    if (ok && rank == 0) cnt[d] = prev + __popc(peers);
    __syncwarp();
    return prev + rank;
}

// The same for a warp's keys, item j of lane l being key 32 j + l of m.  FULL: m == 32 IPT.
template <bool FULL, int IPT>
__device__ __forceinline__ void gt_rank_keys(const unsigned long long (&k)[IPT], int shift, int m, uint32_t *cnt,
                                             uint32_t (&loc)[IPT]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < IPT; j++) {
        const bool ok = FULL || 32 * j + lane < m;
        loc[j] = gt_rank_digit<FULL>(ok ? (uint32_t)(k[j] >> shift) & (GT_SORT_DIGITS - 1) : GT_SORT_DIGITS, cnt);
    }
}
