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
// here -- two passes fewer over all keys (2^24: 322 us of 1290) for one read of them (25 us).  The passes and all three
// ways below are stable, so the result is that of a stable sort by the whole key.  Where the particles fill only a
// small part of the cube (one far particle is enough), the digit of levels 11 to 13 takes few values: once one of them
// holds a sixteenth of the keys (smooth models: a few hundredths of that share) the two low passes run as well.
constexpr uint32_t RUN_SHORT = 16;  // keys that one thread puts in order by insertion
constexpr int RUN_SMEM = TILE;      // keys that a block puts in order in shared memory

__device__ __forceinline__ bool same_run(unsigned long long a, unsigned long long b, int shift) {
    return ((a ^ b) >> shift) == 0ull;
}

// One thread per key: the first key of a run of two or more has it put in order, or listed if it is longer and not in
// order already as far as looked.
__device__ __forceinline__ void fix_runs_body(const unsigned bid, const unsigned nb, long long n, int shift,
        unsigned long long *key, uint32_t *val, uint32_t *list, DevCtl *ctl) {
    if (ctl->sort_whole) return;
    for (long long i = bid * 256ll + threadIdx.x; i < n; i += (long long)nb * 256) {
        const unsigned long long k0 = key[i];
        if (i + 1 >= n || !same_run(k0, key[i + 1], shift)) continue;
        if (i > 0 && same_run(key[i - 1], k0, shift)) continue;
        uint32_t len = 2;
        while (len <= RUN_SHORT && i + len < n && same_run(k0, key[i + len], shift)) len++;
        if (len > RUN_SHORT) {
            list[atomicAdd(&ctl->run_count, 1u)] = (uint32_t)i;
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
}

__global__ __launch_bounds__(256) void k_fix_runs(long long n, int shift, unsigned long long *key, uint32_t *val,
        uint32_t *list, DevCtl *ctl) {
    gt_grid_ready();
    fix_runs_body(blockIdx.x, gridDim.x, n, shift, key, val, list, ctl);
}

// The listed runs, a block each: by digits in shared memory, or, beyond RUN_SMEM keys, tile by tile through the
// other buffers.  Runs that are in order (equal keys, most of all) are left alone.
__device__ __forceinline__ void fix_long_runs_body(const unsigned bid, const unsigned nb, long long n, int shift,
        unsigned long long *key0, uint32_t *val0, unsigned long long *key1, uint32_t *val1,
        const uint32_t *__restrict__ list, DevCtl *ctl) {
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned long long *skey = (unsigned long long *)smraw;
    uint32_t *sval = (uint32_t *)(skey + TILE);
    uint32_t *wcnt = sval + TILE;      // NW x R
    uint32_t *dstart = wcnt + NW * R;  // R: where the next key of every digit goes
    uint32_t *scantmp = dstart + 2 * R;
    __shared__ int sorted_sh;
    __shared__ unsigned long long len_sh;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t runs = ctl->run_count;  // 0 if the whole keys were sorted
    for (uint32_t r = bid; r < runs; r += nb) {
        const long long first = list[r];
        const unsigned long long k0 = key0[first];
        if (threadIdx.x == 0) {
            sorted_sh = 1;
            len_sh = ~0ull;
        }
        __syncthreads();
        for (long long at = first;; at += ST) {  // the run's end, and whether its keys are in order
            const long long i = at + threadIdx.x;
            const bool in = i < n && same_run(k0, key0[i], shift);
            if (!in) atomicMin(&len_sh, (unsigned long long)(i - first));
            else if (i > first && key0[i - 1] > key0[i]) sorted_sh = 0;
            __syncthreads();
            const bool end = len_sh != ~0ull;
            __syncthreads();
            if (end) break;
        }
        const long long len = (long long)len_sh;
        const bool sorted = sorted_sh != 0;
        __syncthreads();
        if (sorted) continue;
        unsigned long long *ka = key0 + first, *kb = key1 + first;
        uint32_t *va = val0 + first, *vb = val1 + first;
        const bool once = len <= RUN_SMEM;
        for (int s0 = 0; s0 < shift; s0 += RB) {  // (digits above the run's own bits agree: the last one may hold some)
            if (!once) {  // where every digit starts
                if (threadIdx.x < R) wcnt[threadIdx.x] = 0;
                __syncthreads();
                for (long long i = threadIdx.x; i < len; i += ST) atomicAdd(&wcnt[(ka[i] >> s0) & (R - 1)], 1u);
                __syncthreads();
                uint32_t total;
                const uint32_t c = threadIdx.x < R ? wcnt[threadIdx.x] : 0u;
                const uint32_t e = block_excl_scan<ST>(c, &total, scantmp);
                if (threadIdx.x < R) dstart[threadIdx.x] = e;
                __syncthreads();
            }
            for (long long t0 = 0; t0 < len; t0 += TILE) {
                for (int i = threadIdx.x; i < NW * R; i += ST) wcnt[i] = 0;
                __syncthreads();
                const long long base = t0 + w * (32 * IPT);
                const int m = (int)(len - base < 0 ? 0 : (len - base < 32 * IPT ? len - base : 32 * IPT));
                unsigned long long k[IPT];
                uint32_t v[IPT], loc[IPT];
#pragma unroll
                for (int j = 0; j < IPT; j++) {
                    const int i = 32 * j + lane;
                    k[j] = 0ull;
                    v[j] = 0u;
                    if (i < m) {
                        if (once && s0 > 0) {
                            k[j] = skey[base + i];
                            v[j] = sval[base + i];
                        } else {
                            k[j] = ka[base + i];
                            v[j] = va[base + i];
                        }
                    }
                }
                gt_rank_keys<false, IPT>(k, s0, m, wcnt + w * R, loc);
                __syncthreads();
                uint32_t cnt = 0;
                if (threadIdx.x < R)
                    for (int ww = 0; ww < NW; ww++) {
                        const uint32_t t = wcnt[ww * R + threadIdx.x];
                        wcnt[ww * R + threadIdx.x] = cnt;
                        cnt += t;
                    }
                if (once) {
                    uint32_t total;
                    const uint32_t e = block_excl_scan<ST>(cnt, &total, scantmp);
                    if (threadIdx.x < R) dstart[threadIdx.x] = e;
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < IPT; j++) {
                    if (32 * j + lane >= m) continue;
                    const uint32_t d = (uint32_t)(k[j] >> s0) & (R - 1);
                    const uint32_t pos = dstart[d] + wcnt[w * R + d] + loc[j];
                    if (once) {
                        skey[pos] = k[j];
                        sval[pos] = v[j];
                    } else {
                        kb[pos] = k[j];
                        vb[pos] = v[j];
                    }
                }
                __syncthreads();
                if (!once && threadIdx.x < R) dstart[threadIdx.x] += cnt;
                __syncthreads();
            }
            if (!once) {
                unsigned long long *kt = ka;
                ka = kb;
                kb = kt;
                uint32_t *vt = va;
                va = vb;
                vb = vt;
            }
        }
        if (once) {
            for (long long i = threadIdx.x; i < len; i += ST) {
                key0[first + i] = skey[i];
                val0[first + i] = sval[i];
            }
        } else if (ka != key0 + first) {
            for (long long i = threadIdx.x; i < len; i += ST) {
                key0[first + i] = ka[i];
                val0[first + i] = va[i];
            }
        }
        __syncthreads();
    }
}

__global__ __launch_bounds__(ST) void k_fix_long_runs(long long n, int shift, unsigned long long *key0,
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

__host__ __device__ inline unsigned fix_blocks(long long n, int nsm) { return gt_grid(n, 256, nsm * 16); }
__host__ __device__ inline unsigned fix_long_blocks(long long n, int nsm) { return gt_grid(n, 4 * TILE, nsm); }

__global__ __launch_bounds__(256) void kg_fix_runs(const GroupedSys *__restrict__ t, int shift, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = fix_blocks(s.n, nsm);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb)
        fix_runs_body(blockIdx.y, nb, s.n, shift, (unsigned long long *)s.sb.key[0], s.sb.val[0], s.sb.status, s.ctl);
}

__global__ __launch_bounds__(ST) void kg_fix_long_runs(const GroupedSys *__restrict__ t, int shift, int nsm) {
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
    cudaFuncSetAttribute(kg_fix_long_runs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SCATTER_SMEM);
    cudaFuncSetAttribute(k_fix_long_runs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SCATTER_SMEM);
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
    gt_launch(k_fix_long_runs, fix_long_blocks(n, nsm), ST, SCATTER_SMEM, st, n, shift,
              (unsigned long long *)b.key[0], b.val[0], (unsigned long long *)b.key[1], b.val[1], list, ctl);
    gt_note_launches(2);
}

void gt_launch_sort(SortBufs &b, int64_t n, DevCtl *ctl, cudaStream_t st) {
    if (n <= 1) return;
    cudaMemsetAsync(b.hist, 0, gt_sort_scratch_bytes(n), st);
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long blocks = (n + HT - 1) / HT;
    k_hist_all<<<(unsigned)(blocks < nsm * 8 ? blocks : nsm * 8), HT, 0, st>>>(n, (const unsigned long long *)b.key[0],
                                                                               b.hist, b.digit_base, ctl);
    gt_note_launches(1);
    for (int p = 0; p < PASSES; p++) onesweep<PASS_PLAIN>(b, n, ctl, p, RB * p, st);
}

// ---- sort without allocation (gt_sort_pairs_noalloc) -----------------------------
// All scratch of one sort of up to GT_NOALLOC_SORT_MAX pairs lives in this array:
// [control block | alternate keys | alternate values | digit counts | look-back status |
// digit bases].  Host code must not use the symbol as an address: the device
// address is looked up once per device below.
namespace {

constexpr size_t NA_ALIGN = 256;
constexpr size_t na_up(size_t b) { return (b + NA_ALIGN - 1) / NA_ALIGN * NA_ALIGN; }
constexpr size_t NA_TILES = (GT_NOALLOC_SORT_MAX + TILE - 1) / TILE;
constexpr size_t NA_OFF_KEY = na_up(sizeof(DevCtl));
constexpr size_t NA_OFF_VAL = NA_OFF_KEY + na_up((size_t)GT_NOALLOC_SORT_MAX * sizeof(unsigned long long));
constexpr size_t NA_OFF_HIST = NA_OFF_VAL + na_up((size_t)GT_NOALLOC_SORT_MAX * sizeof(uint32_t));
constexpr size_t NA_OFF_STATUS = NA_OFF_HIST + PASSES * R * sizeof(uint32_t);
constexpr size_t NA_OFF_BASE = NA_OFF_STATUS + na_up(PASSES * R * NA_TILES * sizeof(uint32_t));
constexpr size_t NA_BYTES = NA_OFF_BASE + na_up(PASSES * R * sizeof(uint32_t));

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
    DevCtl *ctl = (DevCtl *)base;
    // the histograms and the look-back status words are cleared by the sort itself; the
    // control block (tickets, error word) starts at zero once, on the first call on a
    // device, after which every call leaves it consistent for the next
    if (first_use) {
        if (cudaMemsetAsync(ctl, 0, sizeof(DevCtl), st) != cudaSuccess) return GT_ECUDA;
    }
    SortBufs b;
    b.key[0] = d_keys;
    b.val[0] = d_vals;
    b.key[1] = (uint64_t *)(base + NA_OFF_KEY);
    b.val[1] = (uint32_t *)(base + NA_OFF_VAL);
    b.status = (uint32_t *)(base + NA_OFF_STATUS);
    b.hist = (uint32_t *)(base + NA_OFF_HIST);
    b.digit_base = (uint32_t *)(base + NA_OFF_BASE);
    gt_launch_sort(b, n, ctl, st);  // an even number of passes leaves the result in d_keys/d_vals
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
    DevCtl *ctl = (DevCtl *)base;
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
    gt_launch(kg_fix_long_runs, dim3(p.count, fix_long_blocks(p.n_build, nsm)), ST, SCATTER_SMEM, st, t, shift, nsm);
    gt_note_launches(PASSES + 2);
}
