// Step A1: bounding cube and 63-bit Morton keys (Sec. 2.1; Morton key layout of
// Appendix A: every 3-bit digit is (x, y, z) with x the most significant bit).
//
// The bounding box reads 16 B per particle and folds every block's extrema into the control
// block; the key pass reads 16 B and writes 8 B (the index of the first sort pass's input is its
// position), counts the digits of the sort's eight passes on the way, and its last block turns the
// counts into the digits' starts.
#include <float.h>

#include "gt_internal.cuh"
#include "keys_quant.cuh"
#include "sort_digits.cuh"

namespace {

constexpr int BBOX_THREADS = 256;
// Blocks per SM of the key pass: every block adds up to 2048 counts to the global ones, which below ~2^22 keys costs
// more than the warps hide (whole builds with 4 and with 8: 2^19 203 and 208 us, 2^20 291 and 302, 2^21 442 and 442, 2^22
// 761 and 761; an earlier 2^24 3009 and 3001).
constexpr int64_t KEYS_MANY = 1 << 22;

__device__ __forceinline__ void bbox_body(const unsigned bid, const unsigned nb, const float4 *__restrict__ posm,
        long long n, DevCtl *ctl, uint4 *__restrict__ clear, long long nclear) {
    // the sort's counts and look-back words, which the next launch wants at zero
    for (long long i = bid * (long long)BBOX_THREADS + threadIdx.x; i < nclear;
         i += (long long)nb * BBOX_THREADS)
        clear[i] = make_uint4(0u, 0u, 0u, 0u);
    float mn0 = FLT_MAX, mn1 = FLT_MAX, mn2 = FLT_MAX;
    float mx0 = -FLT_MAX, mx1 = -FLT_MAX, mx2 = -FLT_MAX;
    for (long long i = bid * (long long)BBOX_THREADS + threadIdx.x; i < n;
         i += (long long)nb * BBOX_THREADS) {
        const float4 p = posm[i];
        mn0 = fminf(mn0, p.x); mx0 = fmaxf(mx0, p.x);
        mn1 = fminf(mn1, p.y); mx1 = fmaxf(mx1, p.y);
        mn2 = fminf(mn2, p.z); mx2 = fmaxf(mx2, p.z);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn0 = fminf(mn0, __shfl_xor_sync(0xffffffffu, mn0, o));
        mn1 = fminf(mn1, __shfl_xor_sync(0xffffffffu, mn1, o));
        mn2 = fminf(mn2, __shfl_xor_sync(0xffffffffu, mn2, o));
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
        mx2 = fmaxf(mx2, __shfl_xor_sync(0xffffffffu, mx2, o));
    }
    __shared__ float s[BBOX_THREADS / 32][6];
    const int w = threadIdx.x >> 5;
    if (lane_id() == 0) {
        s[w][0] = mn0; s[w][1] = mn1; s[w][2] = mn2;
        s[w][3] = mx0; s[w][4] = mx1; s[w][5] = mx2;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        float v = s[0][threadIdx.x];
        for (int k = 1; k < BBOX_THREADS / 32; k++)
            v = threadIdx.x < 3 ? fminf(v, s[k][threadIdx.x]) : fmaxf(v, s[k][threadIdx.x]);
        if (threadIdx.x < 3) atomicMin(&ctl->bbox[threadIdx.x], gt_ordered(v));
        else atomicMax(&ctl->bbox[threadIdx.x], gt_ordered(v));
    }
}

__global__ __launch_bounds__(BBOX_THREADS) void k_bbox(const float4 *__restrict__ posm, long long n, DevCtl *ctl,
        uint4 *__restrict__ clear, long long nclear) {
    gt_grid_ready();
    bbox_body(blockIdx.x, gridDim.x, posm, n, ctl, clear, nclear);
}

// Spread the low 11 bits of v so that bit b lands on bit 3b.
__device__ __forceinline__ uint32_t spread3(uint32_t v) {
    v = (v | (v << 16)) & 0x070000ffu;
    v = (v | (v << 8)) & 0x0700f00fu;
    v = (v | (v << 4)) & 0x430c30c3u;
    return (v | (v << 2)) & 0x49249249u;
}

// The bits of three 21-bit integers interleaved, x the most significant of every triplet.
__device__ __forceinline__ unsigned long long interleave(uint32_t x, uint32_t y, uint32_t z) {
    const uint32_t xl = spread3(x & 0x7ffu);
    const uint32_t lo = (xl << 2) | (spread3(y & 0x7ffu) << 1) | spread3(z & 0x7ffu);
    const uint32_t hi = (spread3(x >> 11) << 2) | (spread3(y >> 11) << 1) | spread3(z >> 11);
    return ((unsigned long long)((hi << 1) | (xl >> 30)) << 32) | lo;
}

constexpr unsigned long long QMAX = (1ull << GT_KEY_LEVELS) - 1ull;

// floor((x - xmin) * 2^21/side) with FP64 roundings (RN difference, RN product, then the floor), clamped to
// 2^21 - 1: in integer arithmetic (keys_quant.cuh), or for the operands it does not take, on the FP64 pipe -- x
// widened exactly on the integer pipe, the floor the round-down conversion (the product is >= 0).
__device__ __noinline__ uint32_t quantise_slow(float x, float xmin, double scale) {
    unsigned long long q;
    if (quantise_exact(x, xmin, (unsigned long long)__double_as_longlong(scale), QMAX, &q)) return (uint32_t)q;
    q = __double2ull_rd(__dmul_rn(__dsub_rn(f2d(x), f2d(xmin)), scale));
    return (uint32_t)(q < QMAX ? q : QMAX);
}

// Peano-Hilbert order (Sec. 2.1, App. A), Skilling's transpose method on the three
// 21-bit integers: the rotations and reflections are undone from the top bit down, a
// Gray code runs across the axes, and the transposed bits are interleaved like a Morton
// key (axis 0 the most significant of every triplet).
__device__ __forceinline__ void hilbert_transpose(uint32_t &x0, uint32_t &x1, uint32_t &x2) {
#pragma unroll 4
    for (uint32_t q = 1u << (GT_KEY_LEVELS - 1); q > 1u; q >>= 1) {
        const uint32_t p = q - 1u;
        if (x0 & q) x0 ^= p;  // axis 0 against itself: a reflection or nothing
        if (x1 & q) { x0 ^= p; } else { const uint32_t t = (x0 ^ x1) & p; x0 ^= t; x1 ^= t; }
        if (x2 & q) { x0 ^= p; } else { const uint32_t t = (x0 ^ x2) & p; x0 ^= t; x2 ^= t; }
    }
    x1 ^= x0;
    x2 ^= x1;
    uint32_t t = 0u;
#pragma unroll 4
    for (uint32_t q = 1u << (GT_KEY_LEVELS - 1); q > 1u; q >>= 1)
        if (x2 & q) t ^= q - 1u;
    x0 ^= t;
    x1 ^= t;
    x2 ^= t;
}

// The grid of a set of positions: the cube's lower corner and scale, and the scale on the FP32 pipe.
struct KeyGrid {
    float x0, y0, z0, sh, sl;
    double scale;
    bool fp32;
    __device__ __forceinline__ unsigned long long key(const float4 &p, int curve) const {
        uint32_t x = 0, y = 0, z = 0;
        if (!fp32 || !quantise_fp32(p.x, x0, sh, sl, &x)) x = quantise_slow(p.x, x0, scale);
        if (!fp32 || !quantise_fp32(p.y, y0, sh, sl, &y)) y = quantise_slow(p.y, y0, scale);
        if (!fp32 || !quantise_fp32(p.z, z0, sh, sl, &z)) z = quantise_slow(p.z, z0, scale);
        if (curve == GT_KEY_HILBERT) hilbert_transpose(x, y, z);
        return interleave(x, y, z);
    }
};

// 2^21 / the cube's side, 0 for a side of 0, from the extrema (minima, then maxima).
__device__ __forceinline__ double cube_scale(const float *ext) {
    double side = 0.0;
    for (int a = 0; a < 3; a++) {
        const double e = __dsub_rn((double)ext[a + 3], (double)ext[a]);
        if (e > side) side = e;
    }
    return side > 0.0 ? __ddiv_rn((double)(1u << GT_KEY_LEVELS), side) : 0.0;
}

// Bound by issue: ~100 instructions per key of quantisation and interleaving on the FP32 and integer pipes and
// ~50 of digit counting, against 24 B of HBM.
__device__ __forceinline__ void keys_body(const unsigned bid, const unsigned nb, const float4 *__restrict__ posm,
        long long n, int curve, DevCtl *ctl, unsigned long long *__restrict__ key, uint32_t *__restrict__ hist,
        uint32_t *__restrict__ base) {
    __shared__ uint32_t h[GT_SORT_PASSES][GT_SORT_DIGITS];
    __shared__ double scale_sh;
    __shared__ float ext[6];
    for (int p = 0; p < GT_SORT_PASSES; p++) h[p][threadIdx.x] = 0;
    if (threadIdx.x < 6) ext[threadIdx.x] = gt_unordered(ctl->bbox[threadIdx.x]);
    __syncthreads();
    if (threadIdx.x == 0) scale_sh = cube_scale(ext);
    __syncthreads();
    KeyGrid grid{ext[0], ext[1], ext[2], 0.f, 0.f, scale_sh, false};
    grid.fp32 = gtq_fp32_scale(grid.scale, &grid.sh, &grid.sl);
    const bool sized = grid.scale > 0.0;
    for (long long i0 = (long long)bid * 256; i0 < n; i0 += (long long)nb * 256) {
        const long long i = i0 + threadIdx.x;
        const bool ok = i < n;
        unsigned long long k = 0;
        if (ok && sized) k = grid.key(posm[i], curve);
        if (ok) key[i] = k;
        gt_count_digits<true>(k, ok, h);
    }
    gt_finish_digits(nb, h, n, hist, base, ctl);
}

__global__ __launch_bounds__(256) void k_keys(const float4 *__restrict__ posm, long long n, int curve, DevCtl *ctl,
        unsigned long long *__restrict__ key, uint32_t *__restrict__ hist, uint32_t *__restrict__ base) {
    gt_grid_ready();
    keys_body(blockIdx.x, gridDim.x, posm, n, curve, ctl, key, hist, base);
}

// Small systems: the bounding box, the keys and the whole sort in one block, in shared memory (through the kernels
// above: thirteen launches, of which every sort pass takes 10 us for the latency of its chain; 8192 particles ~90 us).
// The passes move 16-bit positions only and look the digits up in the keys, which stay: the wavefronts of one SM's
// shared memory and its ballots bound it (7 us a pass; 48 us in all, 70 with keys that move too and eight passes).  Five
// passes over the highest 40 bits, then the short runs that agree there; a longer run that is out of order takes all
// eight passes.
constexpr int SMALL_THREADS = 1024, SMALL_WARPS = SMALL_THREADS / 32, SMALL_IPT = 8;
static_assert(SMALL_THREADS * SMALL_IPT == GT_SMALL_SORT && SMALL_THREADS == 4 * GT_SORT_DIGITS, "one block's keys");
constexpr size_t SMALL_SMEM = GT_SMALL_SORT * (sizeof(unsigned long long) + sizeof(uint16_t)) +
                              SMALL_WARPS * GT_SORT_DIGITS * sizeof(uint32_t);
constexpr int SMALL_SHIFT = 23, SMALL_RUN = 32;  // bits left to the runs; the longest one that a thread puts in order

__device__ __forceinline__ void small_sort_body(const unsigned bid, const unsigned nb,
        const float4 *__restrict__ posm, int n, int curve, unsigned long long *__restrict__ key,
        uint32_t *__restrict__ val) {
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned long long *skey = (unsigned long long *)smraw;
    uint32_t *wcnt = (uint32_t *)(skey + GT_SMALL_SORT);  // a count per warp and digit
    uint16_t *sid = (uint16_t *)(wcnt + SMALL_WARPS * GT_SORT_DIGITS);
    __shared__ float part_ext[SMALL_WARPS][6], ext[6];
    __shared__ uint32_t part[4][GT_SORT_DIGITS], tmp[SMALL_THREADS / 32 + 1];
    __shared__ double scale_sh;
    __shared__ int redo_sh;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, base = w * 32 * SMALL_IPT;
    const int m = n - base < 0 ? 0 : (n - base < 32 * SMALL_IPT ? n - base : 32 * SMALL_IPT);  // this warp's keys
    float v[6];
    for (int a = 0; a < 6; a++) v[a] = a < 3 ? FLT_MAX : -FLT_MAX;
    for (int i = lane; i < m; i += 32) {
        const float4 p = posm[base + i];
        v[0] = fminf(v[0], p.x); v[1] = fminf(v[1], p.y); v[2] = fminf(v[2], p.z);
        v[3] = fmaxf(v[3], p.x); v[4] = fmaxf(v[4], p.y); v[5] = fmaxf(v[5], p.z);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        for (int a = 0; a < 6; a++) {
            const float t = __shfl_xor_sync(0xffffffffu, v[a], o);
            v[a] = a < 3 ? fminf(v[a], t) : fmaxf(v[a], t);
        }
    if (lane == 0)
        for (int a = 0; a < 6; a++) part_ext[w][a] = v[a];
    __syncthreads();
    if (threadIdx.x < 6) {
        float t = part_ext[0][threadIdx.x];
        for (int k = 1; k < SMALL_WARPS; k++)
            t = threadIdx.x < 3 ? fminf(t, part_ext[k][threadIdx.x]) : fmaxf(t, part_ext[k][threadIdx.x]);
        ext[threadIdx.x] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        scale_sh = cube_scale(ext);
        redo_sh = 0;
    }
    __syncthreads();
    KeyGrid grid{ext[0], ext[1], ext[2], 0.f, 0.f, scale_sh, false};
    grid.fp32 = gtq_fp32_scale(grid.scale, &grid.sh, &grid.sl);
    const bool sized = grid.scale > 0.0;
    uint32_t id[SMALL_IPT];
#pragma unroll
    for (int j = 0; j < SMALL_IPT; j++) {
        const int i = 32 * j + lane;
        id[j] = (uint32_t)(base + i);
        if (i < m) skey[base + i] = sized ? grid.key(posm[base + i], curve) : 0ull;
    }
    const unsigned char *bytes = (const unsigned char *)skey;
    const int d = threadIdx.x & (GT_SORT_DIGITS - 1), q = threadIdx.x / GT_SORT_DIGITS;  // a digit, and eight warps
    // one pass over the digit at `shift`: the positions in sid, and in the order's items again in id
    auto pass = [&](int shift) {
        for (int i = threadIdx.x; i < SMALL_WARPS * GT_SORT_DIGITS; i += SMALL_THREADS) wcnt[i] = 0;
        __syncthreads();
        uint32_t dig[SMALL_IPT], loc[SMALL_IPT];
#pragma unroll
        for (int j = 0; j < SMALL_IPT; j++) {
            dig[j] = GT_SORT_DIGITS;
            if (32 * j + lane < m) {
                if ((shift & 7) == 0) dig[j] = bytes[8 * id[j] + shift / 8];
                else dig[j] = (uint32_t)(skey[id[j]] >> shift) & (GT_SORT_DIGITS - 1);
            }
        }
        uint32_t *own = wcnt + w * GT_SORT_DIGITS;
#pragma unroll
        for (int j = 0; j < SMALL_IPT; j++)
            loc[j] = m == 32 * SMALL_IPT ? gt_rank_digit<true>(dig[j], own) : gt_rank_digit<false>(dig[j], own);
        __syncthreads();
        uint32_t cnt = 0;
#pragma unroll
        for (int ww = 0; ww < SMALL_WARPS / 4; ww++) {
            uint32_t *c = &wcnt[(q * (SMALL_WARPS / 4) + ww) * GT_SORT_DIGITS + d];
            const uint32_t t = *c;
            *c = cnt;
            cnt += t;
        }
        part[q][d] = cnt;
        __syncthreads();
        uint32_t sum = 0, total;
        if (q == 0)
            for (int r = 0; r < 4; r++) sum += part[r][d];
        uint32_t at = block_excl_scan<SMALL_THREADS>(sum, &total, tmp);
        if (q == 0)
            for (int r = 0; r < 4; r++) {
                const uint32_t c = part[r][d];
                part[r][d] = at;
                at += c;
            }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < SMALL_IPT; j++)
            if (32 * j + lane < m) sid[part[w / (SMALL_WARPS / 4)][dig[j]] + own[dig[j]] + loc[j]] = (uint16_t)id[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < SMALL_IPT; j++)
            if (32 * j + lane < m) id[j] = sid[base + 32 * j + lane];
    };
    for (int shift = SMALL_SHIFT; shift < 63; shift += GT_SORT_BITS) pass(shift);
    auto same = [&](int i, int j) { return ((skey[sid[i]] ^ skey[sid[j]]) >> SMALL_SHIFT) == 0ull; };
    // Pairs out of order within a run.  The first one of a run of at most SMALL_RUN keys has its thread put the run in
    // order, after every thread has looked; one in a longer run (a thread looks no further than SMALL_RUN keys either way)
    // has everything sorted again.
    auto run_start = [&](int i) {
        while (i > 0 && same(i - 1, i)) i--;
        return i;
    };
    uint32_t mine = 0;
    for (int j = 0, i = threadIdx.x; i + 1 < n; j++, i += SMALL_THREADS) {
        if (!same(i, i + 1) || skey[sid[i]] <= skey[sid[i + 1]]) continue;
        int a = i, b = i + 2;
        bool first = true;
        while (first && a > 0 && i - a < SMALL_RUN && same(a - 1, a)) {
            first = skey[sid[a - 1]] <= skey[sid[a]];
            a--;
        }
        if (!first) continue;
        while (b < n && b - a <= SMALL_RUN && same(i, b)) b++;
        if (b - a > SMALL_RUN) redo_sh = 1;
        else mine |= 1u << j;
    }
    __syncthreads();
    for (uint32_t m = mine; m; m &= m - 1) {
        const int i = (__ffs(m) - 1) * SMALL_THREADS + (int)threadIdx.x, a = run_start(i);
        for (int j = i + 1 - a; a + j < n && same(a, a + j); j++) {
            const uint16_t v = sid[a + j];
            const unsigned long long kv = skey[v];
            int p = j;
            for (; p > 0 && skey[sid[a + p - 1]] > kv; p--) sid[a + p] = sid[a + p - 1];
            sid[a + p] = v;
        }
    }
    __syncthreads();
    const bool redo = redo_sh != 0;
#pragma unroll
    for (int j = 0; j < SMALL_IPT; j++)
        if (32 * j + lane < m) id[j] = sid[base + 32 * j + lane];
    __syncthreads();
    if (redo)  // (the order so far is stable, so sorting it by the whole key is too)
        for (int shift = 0; shift < 63; shift += GT_SORT_BITS) pass(shift);
#pragma unroll
    for (int j = 0; j < SMALL_IPT; j++) {
        const int i = 32 * j + lane;
        if (i < m) {
            key[base + i] = skey[id[j]];
            val[base + i] = id[j];
        }
    }
}

__global__ __launch_bounds__(SMALL_THREADS) void k_small_sort(const float4 *__restrict__ posm, int n, int curve,
        unsigned long long *__restrict__ key, uint32_t *__restrict__ val) {
    gt_grid_ready();
    small_sort_body(blockIdx.x, gridDim.x, posm, n, curve, key, val);
}

// ---- a table of systems ----
__device__ __forceinline__ const float4 *keyed(const GroupedSys &s) {
    return (s.flags & GT_SYS_PREDICTED) ? s.posm_tmp : s.posm;
}

__host__ __device__ inline unsigned keys_blocks(long long n, int nsm) {
    return gt_grid(n, 256, (long long)nsm * (n < KEYS_MANY ? 4 : 8));
}

__global__ __launch_bounds__(BBOX_THREADS) void kg_bbox(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, BBOX_THREADS, nsm * 4);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb)
        bbox_body(blockIdx.y, nb, keyed(s), s.n, s.ctl, (uint4 *)s.sb.hist, (long long)(gt_sort_scratch_bytes(s.n) / 16));
}

__global__ __launch_bounds__(256) void kg_keys(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = keys_blocks(s.n, nsm);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb)
        keys_body(blockIdx.y, nb, keyed(s), s.n, s.curve, s.ctl, (unsigned long long *)s.sb.key[0], s.sb.hist,
                  s.sb.digit_base);
}

__global__ __launch_bounds__(SMALL_THREADS) void kg_small_sort(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    if (s.flags & GT_SYS_BUILD)
        small_sort_body(0, 1, keyed(s), (int)s.n, s.curve, (unsigned long long *)s.sb.key[0], s.sb.val[0]);
}

}  // namespace

void gt_launch_bbox(const float4 *posm, int64_t n, int nblk, DevCtl *ctl, SortBufs &b, cudaStream_t st) {
    if (n <= 0) return;
    static_assert(GT_SORT_DIGITS * 4 % 16 == 0, "cleared 16 bytes at a time");
    gt_launch(k_bbox, gt_grid(n, BBOX_THREADS, nblk), BBOX_THREADS, 0, st, posm, n, ctl, (uint4 *)b.hist,
              (long long)(gt_sort_scratch_bytes(n) / 16));
    gt_note_launches(1);
}

void gt_launch_keys(const float4 *posm, int64_t n, int curve, DevCtl *ctl, SortBufs &b, int nsm, cudaStream_t st) {
    if (n <= 0) return;
    gt_launch(k_keys, keys_blocks(n, nsm), 256, 0, st, posm, n, curve, ctl, (unsigned long long *)b.key[0], b.hist,
              b.digit_base);
    gt_note_launches(1);
}

void gt_keys_init() {
    cudaFuncSetAttribute(k_small_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM);
    cudaFuncSetAttribute(kg_small_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM);
}

void gt_launch_small_sort(const float4 *posm, int64_t n, int curve, SortBufs &b, cudaStream_t st) {
    if (n <= 0) return;
    gt_launch(k_small_sort, 1, SMALL_THREADS, SMALL_SMEM, st, posm, (int)n, curve, (unsigned long long *)b.key[0],
              b.val[0]);
    gt_note_launches(1);
}

void gt_grouped_small_sort(const GroupedSys *t, const GroupedPlan &p, cudaStream_t st) {
    gt_launch(kg_small_sort, p.count, SMALL_THREADS, SMALL_SMEM, st, t);
    gt_note_launches(1);
}

void gt_grouped_keys(const GroupedSys *t, const GroupedPlan &p, int nsm, cudaStream_t st) {
    gt_launch(kg_bbox, dim3(p.count, gt_grid(p.n_build, BBOX_THREADS, nsm * 4)), BBOX_THREADS, 0, st, t, nsm);
    gt_launch(kg_keys, dim3(p.count, keys_blocks(p.n_build, nsm)), 256, 0, st, t, nsm);
    gt_note_launches(2);
}
