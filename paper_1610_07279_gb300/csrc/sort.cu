// Step A2: stable LSD radix sort of (63-bit key, 32-bit index) pairs (Sec. 2.1: the
// particles are sorted by their space-filling key with a library radix sort).
//
// Passes of 8-bit digits, one kernel per pass: eight for a caller's pairs, six over the highest 48 bits for
// the tree's keys, whose ties in those bits are then put in order (k_fix_runs); the digits of all passes are
// counted by the kernel that makes the keys (keys.cu), or for a caller's pairs by
//   k_hist_all     all eight digit counts in one read of the keys, and their starts   (reads 8 B/key)
//   k_onesweep     per 4096-key tile (256 threads) taken in ticket order: a stable rank of
//                  every key inside the tile (warp-striped; a key's peers with the same
//                  digit from nine ballots, its rank by popc), the tile's per-digit counts
//                  published and each digit's exclusive prefix over earlier tiles found
//                  by a decoupled look-back (256 digits in parallel, a window of
//                  GT_SORT_LB earlier tiles per step, every wait bounded), a local sort in
//                  shared memory, then coalesced writes of each digit run
//                  (reads and writes 12 B/key; 4 B of status per digit and tile: two flag
//                  bits, aggregate or inclusive prefix, and a 30-bit count; every pass has
//                  its own status rows, all cleared once per sort)
// Bound by the ranking (issue and shared memory), not by its ~25 B per key of HBM: 2^24 keys 146 us a pass, 63 at the
// copy rate.  Tiles of 256 threads with 16 keys each leave fewer warps' counts to scan than 512 with 8 (154 us); builds
// of 2^24 with tiles of 256 x 16, 256 x 14, 512 x 8, 384 x 12, 512 x 12 (two blocks per SM) and 512 x 10 (two): 2558,
// 2585, 2629, 2652, 2608 and 2557 us; sorts of 1000001 keys: 155, 151, 155, 161, 170 and 157.
#include <stddef.h>

#include <mutex>

#include "gt_internal.cuh"
#include "sort_digits.cuh"

namespace {

#ifndef GT_SORT_MINB
#define GT_SORT_MINB 3
#endif
#ifndef GT_SORT_LB
#define GT_SORT_LB 8               // earlier tiles read per look-back step
#endif
constexpr int RB = GT_SORT_BITS;   // digit bits
constexpr int R = 1 << RB;         // digits
constexpr int HT = R;              // threads of the histogram kernel
constexpr int ST = GT_SORT_ST;     // threads per tile (the first R of them also own one digit each)
constexpr int IPT = GT_SORT_IPT;   // keys per thread
constexpr int TILE = ST * IPT;     // keys per tile
constexpr int NW = ST / 32;
constexpr int PASSES = GT_SORT_PASSES;
constexpr uint32_t ST_AGG = 1u << 30;   // status word: the tile's own count of the digit
constexpr uint32_t ST_PRE = 2u << 30;   // status word: the inclusive count over tiles 0..t
constexpr uint32_t ST_VAL = ST_AGG - 1u;
constexpr size_t SCATTER_SMEM = TILE * sizeof(unsigned long long) + TILE * sizeof(uint32_t) +
                                (NW * R + 2 * R + NW + 1) * sizeof(uint32_t);
static_assert(ST >= R && ST % 32 == 0, "one thread per digit in the per-tile scans");

__global__ __launch_bounds__(HT) void k_hist_all(long long n, const unsigned long long *__restrict__ key,
                                                 uint32_t *__restrict__ hist /* PASSES x R */,
                                                 uint32_t *__restrict__ base, DevCtl *ctl) {
    gt_grid_ready();
    __shared__ uint32_t h[PASSES][R];
    for (int p = 0; p < PASSES; p++) h[p][threadIdx.x] = 0;
    __syncthreads();
    for (long long i0 = (long long)blockIdx.x * HT; i0 < n; i0 += (long long)gridDim.x * HT) {
        const long long i = i0 + threadIdx.x;
        gt_count_digits<false>(i < n ? key[i] : 0ull, i < n, h);
    }
    gt_finish_digits(gridDim.x, h, n, hist, base, ctl);
}

// Look-back of one digit: the count of digit d in all tiles before `tile`.  The status
// word of tile t, digit d sits at status[t * R + d], so the 256 threads of a tile read one
// contiguous row per predecessor; each step reads a window of LB rows at once and adds
// counts back to the first tile whose inclusive prefix is published.
__device__ __forceinline__ uint32_t lookback_digit(const uint32_t *status, int tile, int d, DevCtl *ctl) {
    constexpr int LB = GT_SORT_LB;
    uint32_t excl = 0;
    int t = tile - 1;
    unsigned int spins = 0;
    const unsigned int limit = gt_spin_limit(ctl);
    while (t >= 0) {
        uint32_t sv[LB];
#pragma unroll
        for (int j = 0; j < LB; j++)
            sv[j] = t - j >= 0 ? *((const volatile uint32_t *)&status[(size_t)(t - j) * R + d]) : ST_PRE;
        int used = 0;
        bool done = false, stalled = false;
#pragma unroll
        for (int j = 0; j < LB; j++) {
            if (done || stalled) continue;
            if (sv[j] & ST_PRE) {
                excl += sv[j] & ST_VAL;
                done = true;
            } else if (sv[j] & ST_AGG) {
                excl += sv[j] & ST_VAL;
                used = j + 1;
            } else {
                stalled = true;
            }
        }
        if (done) break;
        t -= used;
        if (stalled) {
            if (++spins > limit) {
                gt_set_error(ctl, GT_ETIMEOUT, GTK_SORT);
                break;
            }
            __nanosleep(32);
        }
    }
    return excl;
}

// What a pass over the tree's keys does that another doesn't: the first of the low passes makes the values (the keys'
// positions), both of them run only if the whole keys are sorted by passes (ctl->sort_whole), and the first of the
// others makes the values if not.
enum { PASS_PLAIN = 0, PASS_LOW_FIRST, PASS_LOW, PASS_HIGH_FIRST };

template <int MODE>
__device__ __forceinline__ void onesweep_body(const unsigned bid, const unsigned nb, long long n, int pass, int shift,
        const unsigned long long *__restrict__ kin, const uint32_t *__restrict__ vin,
        unsigned long long *__restrict__ kout, uint32_t *__restrict__ vout, const uint32_t *__restrict__ digit_base,
        uint32_t *status, int ntiles, DevCtl *ctl) {
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned long long *skey = (unsigned long long *)smraw;
    uint32_t *sval = (uint32_t *)(skey + TILE);
    uint32_t *wcnt = sval + TILE;     // NW x R: per-warp digit counts, then offsets
    uint32_t *dstart = wcnt + NW * R; // R: tile-local start of every digit
    uint32_t *gbase = dstart + R;     // R: global slot of every digit's first key in this tile
    uint32_t *scantmp = gbase + R;    // NW + 1
    __shared__ uint32_t tile_sh;
    if ((MODE == PASS_LOW_FIRST || MODE == PASS_LOW) && !ctl->sort_whole) return;
    const bool index = MODE == PASS_LOW_FIRST || (MODE == PASS_HIGH_FIRST && !ctl->sort_whole);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) tile_sh = atomicAdd(&ctl->sort_ticket[pass], 1u);
    for (int k = threadIdx.x; k < NW * R; k += ST) wcnt[k] = 0;
    __syncthreads();
    const int tile = (int)tile_sh;
    if (tile >= ntiles) return;

    // warp w owns keys [base, base + 32*IPT) of the tile, item j of lane l is base + 32 j + l:
    // visiting j in order and lanes in order visits the keys in index order (stability)
    const long long base = (long long)tile * TILE + w * (32 * IPT);
    unsigned long long k[IPT];
    uint32_t v[IPT], loc[IPT];
#pragma unroll
    for (int j = 0; j < IPT; j++) {
        const long long i = base + j * 32 + lane;
        k[j] = i < n ? kin[i] : 0ull;
        if (MODE == PASS_LOW_FIRST) v[j] = (uint32_t)i;
        else if (MODE != PASS_HIGH_FIRST) v[j] = i < n ? vin[i] : 0u;
    }
    if (MODE == PASS_HIGH_FIRST) {
#pragma unroll
        for (int j = 0; j < IPT; j++) {
            const long long i = base + j * 32 + lane;
            v[j] = (uint32_t)i;
            if (!index && i < n) v[j] = vin[i];
        }
    }
    if ((long long)(tile + 1) * TILE <= n) gt_rank_keys<true, IPT>(k, shift, 32 * IPT, wcnt + w * R, loc);
    else gt_rank_keys<false, IPT>(k, shift, (int)(n - base < 0 ? 0 : (n - base < 32 * IPT ? n - base : 32 * IPT)), wcnt + w * R, loc);
    __syncthreads();
    // thread d < R: exclusive offsets of the warps for digit d, the tile's count of digit d
    const int d = threadIdx.x;
    const bool dig = d < R;
    uint32_t cnt = 0;
    if (dig)
        for (int ww = 0; ww < NW; ww++) {
            const uint32_t t = wcnt[ww * R + d];
            wcnt[ww * R + d] = cnt;
            cnt += t;
        }
    // publish this tile's count of digit d as early as possible
    uint32_t *own = status + (size_t)tile * R + (dig ? d : 0);
    if (dig) *((volatile uint32_t *)own) = (tile == 0 ? ST_PRE : ST_AGG) | cnt;
    uint32_t total;
    const uint32_t ds0 = block_excl_scan<ST>(cnt, &total, scantmp);
    if (dig) dstart[d] = ds0;
    __syncthreads();
    // local sort by digit in shared memory (stable: warp offset + rank inside the warp)
#pragma unroll
    for (int j = 0; j < IPT; j++) {
        const bool ok = base + j * 32 + lane < n;
        if (ok) {
            const unsigned int dj = (unsigned int)((k[j] >> shift) & (R - 1));
            const uint32_t pos = dstart[dj] + wcnt[w * R + dj] + loc[j];
            skey[pos] = k[j];
            sval[pos] = v[j];
        }
    }
    // count of digit d in all earlier tiles, then this tile's inclusive prefix
    if (dig) {
        uint32_t excl = 0;
        if (tile > 0) {
            excl = lookback_digit(status, tile, d, ctl);
            *((volatile uint32_t *)own) = ST_PRE | (excl + cnt);
        }
        gbase[d] = digit_base[pass * R + d] + excl - dstart[d];
    }
    __syncthreads();
    const long long rem = n - (long long)tile * TILE;
    const int m = rem < TILE ? (int)rem : TILE;
    for (int p = threadIdx.x; p < m; p += ST) {
        const unsigned long long kk = skey[p];
        const unsigned int dk = (unsigned int)((kk >> shift) & (R - 1));
        const uint32_t g = gbase[dk] + (uint32_t)p;
        kout[g] = kk;
        vout[g] = sval[p];
    }
}

template <int MODE>
__global__ __launch_bounds__(ST, GT_SORT_MINB) void k_onesweep(long long n, int pass, int shift,
        const unsigned long long *__restrict__ kin, const uint32_t *__restrict__ vin,
        unsigned long long *__restrict__ kout, uint32_t *__restrict__ vout, const uint32_t *__restrict__ digit_base,
        uint32_t *status, int ntiles, DevCtl *ctl) {
    gt_grid_ready();
    onesweep_body<MODE>(blockIdx.x, gridDim.x, n, pass, shift, kin, vin, kout, vout, digit_base, status, ntiles, ctl);
}

// ---- keys that agree in the sorted bits --------------------------------------------
// The tree's keys are spread over the bounding cube by construction, so few of them agree in their highest 16 levels
// (48 bits): six passes over those bits leave short runs of keys that differ only below, and these are put in order
// here -- two passes fewer over all keys (2^24: 322 us of 1290) for one read of them (25 us).  The passes and all
// ways below are stable, so the result is that of a stable sort by the whole key.  Where long runs are to be expected the
// two low passes run as well (gt_finish_digits); what is left costs no more than they would, whatever the runs' lengths:
// short runs are put in order by a thread, the longer ones that begin in one tile of the keys together by a block in shared
// memory, and one that is too long for that by a block through the other buffers.  (A block for every run longer than 16
// keys, and the choice by one digit: a Plummer sphere of 2^22 with one particle at 2500 times its radius 3854 us the
// whole build, eight passes 1729.)
constexpr uint32_t RUN_SHORT = 16;  // keys that one thread puts in order by insertion
constexpr int FIX_ROUNDS = 8, FIX_TILE = 256 * FIX_ROUNDS;  // keys that a block of k_fix_runs looks at at a time

__device__ __forceinline__ bool same_run(unsigned long long a, unsigned long long b, int shift) {
    return ((a ^ b) >> shift) == 0ull;
}

// One thread per key: the first key of a short run of two or more has it put in order; of the longer ones that begin in a
// tile, the first and the last begin are listed.
__device__ __forceinline__ void fix_runs_body(const unsigned bid, const unsigned nb, long long n, int shift,
        unsigned long long *key, uint32_t *val, uint32_t *list, DevCtl *ctl) {
    if (ctl->sort_whole) return;
    __shared__ uint32_t first_sh, last_sh;
    if (threadIdx.x == 0) first_sh = ~0u, last_sh = 0u;
    __syncthreads();
    for (long long t = (long long)bid * FIX_TILE; t < n; t += (long long)nb * FIX_TILE) {
        uint32_t begins = 0;  // rounds in which this thread's key begins a run of two or more
#pragma unroll
        for (int r = 0; r < FIX_ROUNDS; r++) {
            const long long i = t + 256 * r + threadIdx.x;
            if (i + 1 >= n) continue;
            const unsigned long long k0 = key[i], k1 = key[i + 1], kb = i > 0 ? key[i - 1] : ~k0;
            if (same_run(k0, k1, shift) && !same_run(kb, k0, shift)) begins |= 1u << r;
        }
        for (; begins; begins &= begins - 1) {
            const long long i = t + 256 * (__ffs(begins) - 1) + threadIdx.x;
            const unsigned long long k0 = key[i];
            uint32_t len = 2;
            while (len <= RUN_SHORT && i + len < n && same_run(k0, key[i + len], shift)) len++;
            if (len > RUN_SHORT) {
                atomicMin(&first_sh, (uint32_t)i);
                atomicMax(&last_sh, (uint32_t)i);
                continue;
            }
            for (uint32_t j = 1; j < len; j++) {
                const unsigned long long k = key[i + j];
                const uint32_t v = val[i + j];
                uint32_t p = j;
                for (; p > 0 && key[i + p - 1] > k; p--) {
                    key[i + p] = key[i + p - 1];
                    val[i + p] = val[i + p - 1];
                }
                if (p != j) {
                    key[i + p] = k;
                    val[i + p] = v;
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && first_sh != ~0u) {
            const uint32_t at = atomicAdd(&ctl->run_count, 1u);
            list[2 * at] = first_sh;
            list[2 * at + 1] = last_sh;
            first_sh = ~0u;
            last_sh = 0u;
        }
        __syncthreads();
    }
}

__global__ __launch_bounds__(256) void k_fix_runs(long long n, int shift, unsigned long long *key, uint32_t *val,
        uint32_t *list, DevCtl *ctl) {
    gt_grid_ready();
    fix_runs_body(blockIdx.x, gridDim.x, n, shift, key, val, list, ctl);
}

// Shared memory of a block of k_fix_long_runs: three of them per SM.
struct FixShared {
    unsigned long long key[TILE];
    uint32_t val[TILE];
    uint16_t pos[TILE], run[TILE];  // an order of the keys, and the run of each (numbers from 0)
    uint32_t wcnt[NW * R];          // a count per warp and digit
    uint32_t dstart[R];             // where the next key of every digit goes
    uint32_t scantmp[NW + 1], wruns[NW];
};
constexpr size_t FIX_SMEM = sizeof(FixShared);

// The start of every digit's keys of the warp in its tile: the sums over the warps before, and (returned, for the
// thread's digit) the tile's count.
__device__ __forceinline__ uint32_t scan_warps(FixShared &sm) {
    uint32_t cnt = 0;
    if (threadIdx.x < R)
        for (int ww = 0; ww < NW; ww++) {
            const uint32_t t = sm.wcnt[ww * R + threadIdx.x];
            sm.wcnt[ww * R + threadIdx.x] = cnt;
            cnt += t;
        }
    return cnt;
}

// The first m keys in shared memory, whole runs, to global memory in the order of a stable sort by the whole key: by the
// bits below `shift`, then by run, on the keys' positions.  Left alone if in order already.
__device__ __forceinline__ void sort_region(FixShared &sm, int m, int shift, unsigned long long *key, uint32_t *val) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, base = w * 32 * IPT;
    bool out = false;
    for (int i = threadIdx.x; i + 1 < m; i += ST) out = out || sm.key[i] > sm.key[i + 1];
    if (!__syncthreads_or(out)) return;
    uint32_t id[IPT], runs = 0;
#pragma unroll
    for (int j = 0; j < IPT; j++) {
        const int i = base + 32 * j + lane;
        id[j] = (uint32_t)i;
        const unsigned begins = __ballot_sync(0xffffffffu, i > 0 && i < m && !same_run(sm.key[i - 1], sm.key[i], shift));
        if (i < m) sm.run[i] = (uint16_t)(runs + (uint32_t)__popc(begins & (lanemask_lt() | (1u << lane))));
        runs += (uint32_t)__popc(begins);
    }
    if (lane == 0) sm.wruns[w] = runs;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int ww = 0; ww < NW; ww++) {
        before += ww < w ? sm.wruns[ww] : 0u;
        all += sm.wruns[ww];
    }
    for (int i = base + lane; i < base + 32 * IPT && i < m; i += 32) sm.run[i] = (uint16_t)(sm.run[i] + before);
    __syncthreads();
    // digits: the low bits (the last digit reaches into the run's own bits, which the runs' digits outweigh), the run
    const int low = (shift + RB - 1) / RB, passes = low + (all == 0u ? 0 : (all < R ? 1 : 2));
    for (int p = 0; p < passes; p++) {
        for (int i = threadIdx.x; i < NW * R; i += ST) sm.wcnt[i] = 0;
        __syncthreads();
        uint32_t dig[IPT], loc[IPT];
#pragma unroll
        for (int j = 0; j < IPT; j++) {
            dig[j] = R;
            if (base + 32 * j + lane < m)
                dig[j] = (p < low ? (uint32_t)(sm.key[id[j]] >> (RB * p)) : (uint32_t)sm.run[id[j]] >> (RB * (p - low))) & (R - 1);
        }
        if (base < m) {
#pragma unroll
            for (int j = 0; j < IPT; j++) loc[j] = gt_rank_digit<false>(dig[j], sm.wcnt + w * R);
        }
        __syncthreads();
        const uint32_t cnt = scan_warps(sm);
        uint32_t total;
        const uint32_t e = block_excl_scan<ST>(cnt, &total, sm.scantmp);
        if (threadIdx.x < R) sm.dstart[threadIdx.x] = e;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < IPT; j++)
            if (dig[j] < R) sm.pos[sm.dstart[dig[j]] + sm.wcnt[w * R + dig[j]] + loc[j]] = (uint16_t)id[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < IPT; j++)
            if (dig[j] < R) id[j] = sm.pos[base + 32 * j + lane];
    }
#pragma unroll
    for (int j = 0; j < IPT; j++) {
        const int i = base + 32 * j + lane;
        if (i < m) {
            key[i] = sm.key[id[j]];
            val[i] = sm.val[id[j]];
        }
    }
}

// A run that is longer than a tile, from key0[first] on, by one block, tile after tile through the other buffers.  Left
// alone if in order already (equal keys, most of all).
__device__ __forceinline__ void sort_long_run(FixShared &sm, long long first, long long n, int shift,
        unsigned long long *key0, uint32_t *val0, unsigned long long *key1, uint32_t *val1) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long k0 = key0[first];
    // its end: every round cuts what is left to a part in 256
    long long a = first, b = n;  // key0[a] belongs to it, key0[b] (if b < n) doesn't
    while (b - a > 1) {
        const long long step = (b - a + ST - 1) / ST, i = a + step * threadIdx.x;
        const int in = __syncthreads_count(i < b && same_run(k0, key0[i], shift));  // the first `in` threads
        a += step * (in - 1);
        b = a + step < b ? a + step : b;
    }
    const long long len = a + 1 - first;
    bool out = false;
    for (long long i = first + 1 + threadIdx.x; i < first + len && !out; i += 8 * ST) {
        unsigned long long k[8], kb[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const long long at = i + (long long)j * ST < first + len ? i + (long long)j * ST : i;
            k[j] = key0[at];
            kb[j] = key0[at - 1];
        }
#pragma unroll
        for (int j = 0; j < 8; j++) out = out || kb[j] > k[j];
    }
    if (!__syncthreads_or(out)) return;
    unsigned long long *ka = key0 + first, *kb = key1 + first;
    uint32_t *va = val0 + first, *vb = val1 + first;
    for (int s0 = 0; s0 < shift; s0 += RB) {  // (digits above the run's own bits agree: the last one may hold some)
        if (threadIdx.x < R) sm.wcnt[threadIdx.x] = 0;  // where every digit starts
        __syncthreads();
        for (long long i = threadIdx.x; i < len; i += ST) atomicAdd(&sm.wcnt[(ka[i] >> s0) & (R - 1)], 1u);
        __syncthreads();
        uint32_t total;
        const uint32_t e = block_excl_scan<ST>(threadIdx.x < R ? sm.wcnt[threadIdx.x] : 0u, &total, sm.scantmp);
        if (threadIdx.x < R) sm.dstart[threadIdx.x] = e;
        __syncthreads();
        for (long long t0 = 0; t0 < len; t0 += TILE) {
            for (int i = threadIdx.x; i < NW * R; i += ST) sm.wcnt[i] = 0;
            __syncthreads();
            const long long base = t0 + w * (32 * IPT);
            const int m = (int)(len - base < 0 ? 0 : (len - base < 32 * IPT ? len - base : 32 * IPT));
            unsigned long long k[IPT];
            uint32_t v[IPT], loc[IPT];
#pragma unroll
            for (int j = 0; j < IPT; j++) {
                const int i = 32 * j + lane;
                k[j] = i < m ? ka[base + i] : 0ull;
                v[j] = i < m ? va[base + i] : 0u;
            }
            gt_rank_keys<false, IPT>(k, s0, m, sm.wcnt + w * R, loc);
            __syncthreads();
            const uint32_t cnt = scan_warps(sm);
            __syncthreads();
#pragma unroll
            for (int j = 0; j < IPT; j++) {
                if (32 * j + lane >= m) continue;
                const uint32_t d = (uint32_t)(k[j] >> s0) & (R - 1);
                const uint32_t pos = sm.dstart[d] + sm.wcnt[w * R + d] + loc[j];
                kb[pos] = k[j];
                vb[pos] = v[j];
            }
            __syncthreads();
            if (threadIdx.x < R) sm.dstart[threadIdx.x] += cnt;
            __syncthreads();
        }
        unsigned long long *kt = ka;
        ka = kb;
        kb = kt;
        uint32_t *vt = va;
        va = vb;
        vb = vt;
    }
    if (ka != key0 + first)
        for (long long i = threadIdx.x; i < len; i += ST) {
            key0[first + i] = ka[i];
            val0[first + i] = va[i];
        }
}

// The listed tiles, a block each: from the first long run's first key to the last one's last, if it is at most TILE keys
// on, in shared memory (runs that begin in a tile of FIX_TILE keys); a longer last run by itself.
__device__ __forceinline__ void fix_long_runs_body(const unsigned bid, const unsigned nb, long long n, int shift,
        unsigned long long *key0, uint32_t *val0, unsigned long long *key1, uint32_t *val1,
        const uint32_t *__restrict__ list, DevCtl *ctl) {
    extern __shared__ __align__(16) unsigned char smraw[];
    static_assert(FIX_TILE <= TILE && TILE <= 65536, "the last run begins in the tile; 16-bit positions");
    FixShared &sm = *(FixShared *)smraw;
    const uint32_t tiles = ctl->run_count;  // 0 if the whole keys were sorted
    for (uint32_t t = bid; t < tiles; t += nb) {
        const long long first = list[2 * t];
        const int last = (int)(list[2 * t + 1] - list[2 * t]);
        const int room = n - first < TILE ? (int)(n - first) : TILE;
        for (int i = threadIdx.x; i < room; i += ST) {
            sm.key[i] = key0[first + i];
            sm.val[i] = val0[first + i];
        }
        __syncthreads();
        const unsigned long long kl = sm.key[last];
        int end = last + 1, no = room;  // the last run's end, by bisection: keys before `end` are before it
        while (end < no) {
            const int mid = (end + no) / 2;
            if (same_run(kl, sm.key[mid], shift)) end = mid + 1;
            else no = mid;
        }
        const bool open = end == room && first + room < n && same_run(kl, key0[first + room], shift);
        sort_region(sm, open ? last : end, shift, key0 + first, val0 + first);
        __syncthreads();
        if (open) sort_long_run(sm, first + last, n, shift, key0, val0, key1, val1);
        __syncthreads();
    }
}

__global__ __launch_bounds__(ST, 3) void k_fix_long_runs(long long n, int shift, unsigned long long *key0,
        uint32_t *val0, unsigned long long *key1, uint32_t *val1, const uint32_t *__restrict__ list, DevCtl *ctl) {
    gt_grid_ready();
    fix_long_runs_body(blockIdx.x, gridDim.x, n, shift, key0, val0, key1, val1, list, ctl);
}

// ---- a table of systems ----
template <int MODE>
__global__ __launch_bounds__(ST, GT_SORT_MINB) void kg_onesweep(const GroupedSys *__restrict__ t, int pass, int shift) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const int ntiles = gt_sort_tiles(s.n), src = pass & 1;
    if (!(s.flags & GT_SYS_BUILD) || (int)blockIdx.y >= ntiles) return;
    onesweep_body<MODE>(blockIdx.y, (unsigned)ntiles, s.n, pass, shift, (const unsigned long long *)s.sb.key[src],
                        s.sb.val[src], (unsigned long long *)s.sb.key[src ^ 1], s.sb.val[src ^ 1], s.sb.digit_base,
                        s.sb.status + (size_t)pass * R * ntiles, ntiles, s.ctl);
}

__host__ __device__ inline unsigned fix_blocks(long long n, int nsm) { return gt_grid(n, FIX_TILE, nsm * 8); }
__host__ __device__ inline unsigned fix_long_blocks(long long n, int nsm) { return gt_grid(n, TILE, nsm * 3); }

__global__ __launch_bounds__(256) void kg_fix_runs(const GroupedSys *__restrict__ t, int shift, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = fix_blocks(s.n, nsm);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb)
        fix_runs_body(blockIdx.y, nb, s.n, shift, (unsigned long long *)s.sb.key[0], s.sb.val[0], s.sb.status, s.ctl);
}

__global__ __launch_bounds__(ST, 3) void kg_fix_long_runs(const GroupedSys *__restrict__ t, int shift, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = fix_long_blocks(s.n, nsm);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb)
        fix_long_runs_body(blockIdx.y, nb, s.n, shift, (unsigned long long *)s.sb.key[0], s.sb.val[0],
                           (unsigned long long *)s.sb.key[1], s.sb.val[1], s.sb.status, s.ctl);
}

}  // namespace

void gt_sort_init() {
    gt_keys_init();
    for (auto kernel : {k_onesweep<PASS_PLAIN>, k_onesweep<PASS_LOW_FIRST>, k_onesweep<PASS_LOW>,
                        k_onesweep<PASS_HIGH_FIRST>})
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SCATTER_SMEM);
    for (auto kernel : {kg_onesweep<PASS_PLAIN>, kg_onesweep<PASS_LOW_FIRST>, kg_onesweep<PASS_LOW>,
                        kg_onesweep<PASS_HIGH_FIRST>})
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SCATTER_SMEM);
    cudaFuncSetAttribute(kg_fix_long_runs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FIX_SMEM);
    cudaFuncSetAttribute(k_fix_long_runs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FIX_SMEM);
}

namespace {

// pass p reads buffers p & 1 and writes the others
template <int MODE>
void onesweep(SortBufs &b, int64_t n, DevCtl *ctl, int pass, int shift, cudaStream_t st) {
    const int ntiles = gt_sort_tiles(n), src = pass & 1;
    gt_launch(k_onesweep<MODE>, ntiles, ST, SCATTER_SMEM, st, n, pass, shift, (const unsigned long long *)b.key[src],
              b.val[src], (unsigned long long *)b.key[src ^ 1], b.val[src ^ 1], b.digit_base,
              b.status + (size_t)pass * R * ntiles, ntiles, ctl);
    gt_note_launches(1);
}

}  // namespace

void gt_launch_sort_tree(SortBufs &b, int64_t n, DevCtl *ctl, int nsm, cudaStream_t st) {
    if (n <= 0) return;
    onesweep<PASS_LOW_FIRST>(b, n, ctl, 0, gt_tree_digit_shift(0), st);
    onesweep<PASS_LOW>(b, n, ctl, 1, gt_tree_digit_shift(1), st);
    onesweep<PASS_HIGH_FIRST>(b, n, ctl, 2, gt_tree_digit_shift(2), st);
    for (int p = 3; p < PASSES; p++) onesweep<PASS_PLAIN>(b, n, ctl, p, gt_tree_digit_shift(p), st);
    const int shift = gt_tree_digit_shift(2);
    uint32_t *list = b.status;  // the look-backs are over
    gt_launch(k_fix_runs, fix_blocks(n, nsm), 256, 0, st, n, shift, (unsigned long long *)b.key[0], b.val[0], list,
              ctl);
    gt_launch(k_fix_long_runs, fix_long_blocks(n, nsm), ST, FIX_SMEM, st, n, shift,
              (unsigned long long *)b.key[0], b.val[0], (unsigned long long *)b.key[1], b.val[1], list, ctl);
    gt_note_launches(2);
}

// ---- sort without allocation (gt_sort_pairs_noalloc) -----------------------------
// All scratch of one sort of up to GT_NOALLOC_SORT_MAX pairs lives in this array:
// [alternate keys | alternate values | digit bases | control block | digit counts |
// look-back status].  Host code must not use the symbol as an address: the device
// address is looked up once per device below.
namespace {

constexpr size_t NA_ALIGN = 256;
constexpr size_t na_up(size_t b) { return (b + NA_ALIGN - 1) / NA_ALIGN * NA_ALIGN; }
constexpr size_t NA_TILES = (GT_NOALLOC_SORT_MAX + TILE - 1) / TILE;
constexpr size_t NA_OFF_VAL = na_up((size_t)GT_NOALLOC_SORT_MAX * sizeof(unsigned long long));
constexpr size_t NA_OFF_BASE = NA_OFF_VAL + na_up((size_t)GT_NOALLOC_SORT_MAX * sizeof(uint32_t));
constexpr size_t NA_OFF_CTL = NA_OFF_BASE + na_up(PASSES * R * sizeof(uint32_t));
constexpr size_t NA_OFF_HIST = NA_OFF_CTL + na_up(sizeof(DevCtl));
constexpr size_t NA_OFF_STATUS = NA_OFF_HIST + PASSES * R * sizeof(uint32_t);
constexpr size_t NA_BYTES = NA_OFF_STATUS + na_up(PASSES * R * NA_TILES * sizeof(uint32_t));
static_assert(offsetof(DevCtl, err) < offsetof(DevCtl, digits_done), "a latched error is kept until it is read");

__device__ __align__(256) unsigned char g_noalloc_sort_scratch[NA_BYTES];

constexpr int NA_MAX_DEVICES = 256;
std::mutex g_na_mu;
char *g_na_addr[NA_MAX_DEVICES] = {};

// Device address of the scratch array on the current device (looked up once per device).
int noalloc_scratch(char **out, bool *first_use) {
    *first_use = false;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return GT_ECUDA;
    if (dev < 0 || dev >= NA_MAX_DEVICES) return GT_EINVAL;
    std::lock_guard<std::mutex> lock(g_na_mu);
    if (!g_na_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_sort_scratch) != cudaSuccess || !p) return GT_ECUDA;
        gt_sort_init();  // the sort kernel's shared-memory limit, on this device
        g_na_addr[dev] = (char *)p;
        *first_use = true;
    }
    *out = g_na_addr[dev];
    return GT_OK;
}

// The control block lies right before the digit counts (b.hist): from its counter of finished blocks on, all is cleared
// together, so that a sort doesn't depend on how an earlier one ended (one that another overlapped may leave the counter
// off, and the digits' starts and the tiles' tickets would never be set again).
void launch_sort(SortBufs &b, int64_t n, DevCtl *ctl, cudaStream_t st) {
    if (n <= 1) return;
    char *from = (char *)&ctl->digits_done;
    cudaMemsetAsync(from, 0, (size_t)((char *)b.hist - from) + gt_sort_scratch_bytes(n), st);
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long blocks = (n + HT - 1) / HT;
    k_hist_all<<<(unsigned)(blocks < nsm * 8 ? blocks : nsm * 8), HT, 0, st>>>(n, (const unsigned long long *)b.key[0],
                                                                               b.hist, b.digit_base, ctl);
    gt_note_launches(1);
    for (int p = 0; p < PASSES; p++) onesweep<PASS_PLAIN>(b, n, ctl, p, RB * p, st);
}

}  // namespace

extern "C" int gt_sort_pairs_noalloc(uint64_t *d_keys, uint32_t *d_vals, int64_t n, gt_stream stream) {
    if (n < 0 || (n > 0 && (!d_keys || !d_vals))) return GT_EINVAL;
    if (n > GT_NOALLOC_SORT_MAX) return GT_EINVAL;  // larger than the static scratch
    char *base = nullptr;
    bool first_use = false;
    const int rc = noalloc_scratch(&base, &first_use);
    if (rc != GT_OK) return rc;
    if (n <= 1) return GT_OK;
    cudaStream_t st = (cudaStream_t)stream;
    DevCtl *ctl = (DevCtl *)(base + NA_OFF_CTL);
    // the histograms, the look-back status words and the counters are cleared by the sort itself; the
    // control block (tickets, error word) starts at zero once, on the first call on a
    // device, after which every call leaves it consistent for the next
    if (first_use) {
        if (cudaMemsetAsync(ctl, 0, sizeof(DevCtl), st) != cudaSuccess) return GT_ECUDA;
    }
    SortBufs b;
    b.key[0] = d_keys;
    b.val[0] = d_vals;
    b.key[1] = (uint64_t *)base;
    b.val[1] = (uint32_t *)(base + NA_OFF_VAL);
    b.status = (uint32_t *)(base + NA_OFF_STATUS);
    b.hist = (uint32_t *)(base + NA_OFF_HIST);
    b.digit_base = (uint32_t *)(base + NA_OFF_BASE);
    launch_sort(b, n, ctl, st);  // an even number of passes leaves the result in d_keys/d_vals
    return cudaGetLastError() == cudaSuccess ? GT_OK : GT_ECUDA;
}

extern "C" int gt_sort_noalloc_status(gt_stream stream) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return GT_ECUDA;
    if (dev < 0 || dev >= NA_MAX_DEVICES) return GT_EINVAL;
    char *base;
    {
        std::lock_guard<std::mutex> lock(g_na_mu);
        base = g_na_addr[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaStreamSynchronize(st) != cudaSuccess) return GT_ECUDA;
    if (!base) return GT_OK;  // no sort has run on this device
    DevCtl *ctl = (DevCtl *)(base + NA_OFF_CTL);
    int err = 0;
    if (cudaMemcpyAsync(&err, &ctl->err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return GT_ECUDA;
    if (err && (cudaMemsetAsync(&ctl->err, 0, 2 * sizeof(int), st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess))
        return GT_ECUDA;
    return err;
}

void gt_grouped_sort(const GroupedSys *t, const GroupedPlan &p, int nsm, cudaStream_t st) {
    if (p.n_build <= 0) return;
    if (p.n_build <= GT_SMALL_SORT) {  // (a small system among larger ones costs their launches nothing)
        gt_grouped_small_sort(t, p, st);
        return;
    }
    gt_grouped_keys(t, p, nsm, st);
    const dim3 grid(p.count, gt_sort_tiles(p.n_build));
    gt_launch(kg_onesweep<PASS_LOW_FIRST>, grid, ST, SCATTER_SMEM, st, t, 0, gt_tree_digit_shift(0));
    gt_launch(kg_onesweep<PASS_LOW>, grid, ST, SCATTER_SMEM, st, t, 1, gt_tree_digit_shift(1));
    gt_launch(kg_onesweep<PASS_HIGH_FIRST>, grid, ST, SCATTER_SMEM, st, t, 2, gt_tree_digit_shift(2));
    for (int q = 3; q < PASSES; q++)
        gt_launch(kg_onesweep<PASS_PLAIN>, grid, ST, SCATTER_SMEM, st, t, q, gt_tree_digit_shift(q));
    const int shift = gt_tree_digit_shift(2);
    gt_launch(kg_fix_runs, dim3(p.count, fix_blocks(p.n_build, nsm)), 256, 0, st, t, shift, nsm);
    gt_launch(kg_fix_long_runs, dim3(p.count, fix_long_blocks(p.n_build, nsm)), ST, FIX_SMEM, st, t, shift, nsm);
    gt_note_launches(PASSES + 2);
}
