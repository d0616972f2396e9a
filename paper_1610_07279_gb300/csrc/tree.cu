// Steps A4-A5: breadth-first octree over the sorted keys and the pseudo
// j-particles (Sec. 2.1, Fig. 1).
//
// A4.  A cell at level l with more than leaf_max particles (and l < 21) splits into the
// non-empty ranges of its particles' level-(l + 1) digit; children are numbered after
// their level, level by level and, inside a level, by first particle.  With leaf_max up
// to 64 the whole tree comes from one sweep over the sorted keys (k_flat_*: every
// particle's leaf level from the digits in which its neighbours' keys differ, then the
// nodes' starts and ends counted, scanned and scattered by level); larger leaves take
// one kernel per level (k_build_level: the "seven partitions" of a cell's key range by a
// lock-step 7-way binary search, children numbered by a block scan plus a decoupled
// look-back over tiles taken in ticket order).  Both give the same numbering.
//
// A5, one launch over a cell list bucketed by level and size: a leaf's lane sums its
// particles in FP64 (mass, m x, m y, m z); a cell with children sums its children's FP64
// sums in child order once the level below is done -- every FP64 instruction runs with
// full warps, which matters on this GPU's narrow FP64 pipe.  m_J = (float)M and
// r_J = (float)S / (float)M (a cell of one particle is that particle); b_J is the
// largest FP32 |r - r_J| of a leaf's particles, or the largest |r_c - r_J| + b_c
// over a cell's children, widened by (1 + 2^-20) so that FP32 rounding cannot
// shrink it below the true enclosing radius.  FP64 is kept to the four sums (FP64
// throughput is low on this GPU).  Every operation carries an explicit rounding,
// so the result is the same bit for bit on every run.
#include "gt_internal.cuh"

namespace {

constexpr int BT = 256;         // threads per build block
constexpr int NPT = 1;          // cells per thread
constexpr int BTILE = BT * NPT; // cells per tile

__global__ void k_build_init(long long n, Nodes nd, DevCtl *ctl) {
    gt_grid_ready();
    for (int b = threadIdx.x; b < GT_CELL_BUCKETS; b += blockDim.x) ctl->cell_bucket[b] = 0;
    if (threadIdx.x != 0) return;
    // root = level 0, all particles; level_start[0..1]
    ctl->level_start[0] = 0;
    ctl->level_start[1] = n > 0 ? 1u : 0u;
    if (n > 0) {
        nd.first[0] = 0;
        nd.count[0] = (uint32_t)n;
        nd.parent[0] = -1;
    }
}

__global__ __launch_bounds__(BT) void k_build_level(int lvl, const unsigned long long *__restrict__ skey,
                                                    int leaf_max, Nodes nd, long long cap,
                                                    unsigned long long *status, DevCtl *ctl) {
    gt_grid_ready();
    __shared__ uint32_t tmp[BT / 32 + 1];
    __shared__ uint32_t tile_sh, excl_sh;
    const uint32_t lo = ctl->level_start[lvl], hi = ctl->level_start[lvl + 1];
    const uint32_t cnt = hi - lo;
    if (cnt == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->level_start[lvl + 2] = hi;
        return;
    }
    const uint32_t ntiles = (cnt + BTILE - 1) / BTILE;
    const uint32_t tag = ctl->epoch * 32u + (uint32_t)lvl;
    const bool can_split = lvl < GT_KEY_LEVELS;
    const int shift = 3 * (GT_KEY_LEVELS - 1 - lvl);
    for (;;) {
        if (threadIdx.x == 0) tile_sh = atomicAdd(&ctl->tile_ticket[lvl], 1u);
        __syncthreads();
        const uint32_t tile = tile_sh;
        __syncthreads();
        if (tile >= ntiles) break;
        uint32_t bnd[NPT][9];
        uint32_t nc[NPT];
        uint32_t tsum = 0;
#pragma unroll
        for (int q = 0; q < NPT; q++) {
            const uint32_t c = lo + tile * BTILE + threadIdx.x * NPT + q;
            nc[q] = 0;
            if (c < hi) {
                const uint32_t f = nd.first[c], k = nd.count[c];
                if (can_split && k > (uint32_t)leaf_max) {
                    // smallest p in [f, f+k) with digit(p) >= d, for d = 1..7, in lock step
                    uint32_t l7[7], h7[7];
#pragma unroll
                    for (int d = 0; d < 7; d++) { l7[d] = f; h7[d] = f + k; }
                    const int iters = 32 - __clz(k);
                    for (int it = 0; it < iters; it++) {
#pragma unroll
                        for (int d = 0; d < 7; d++) {
                            if (l7[d] < h7[d]) {
                                const uint32_t mid = (l7[d] + h7[d]) >> 1;
                                const uint32_t dig = (uint32_t)((__ldg(&skey[mid]) >> shift) & 7ull);
                                if (dig < (uint32_t)(d + 1)) l7[d] = mid + 1; else h7[d] = mid;
                            }
                        }
                    }
                    bnd[q][0] = f;
#pragma unroll
                    for (int d = 0; d < 7; d++) bnd[q][d + 1] = l7[d];
                    bnd[q][8] = f + k;
#pragma unroll
                    for (int d = 0; d < 8; d++) nc[q] += bnd[q][d + 1] > bnd[q][d] ? 1u : 0u;
                }
            }
            tsum += nc[q];
        }
        uint32_t total;
        uint32_t excl = block_excl_scan<BT>(tsum, &total, tmp);
        if (threadIdx.x < 32) {
            const uint32_t e = lookback_warp(status, tile, total, tag, ctl, GTK_BUILD);
            if (threadIdx.x == 0) excl_sh = e;
        }
        __syncthreads();
        uint32_t next = hi + excl_sh + excl;  // node id of this thread's first child
#pragma unroll
        for (int q = 0; q < NPT; q++) {
            const uint32_t c = lo + tile * BTILE + threadIdx.x * NPT + q;
            if (c >= hi) continue;
            if (nc[q] == 0) {  // a leaf
                nd.child[c] = -1;
                nd.nchild[c] = 0;
                continue;
            }
            if ((long long)next + nc[q] > cap) {
                gt_set_error(ctl, GT_EOVERFLOW, GTK_BUILD);
                nd.child[c] = -1;
                nd.nchild[c] = 0;
                next += nc[q];
                continue;
            }
            nd.child[c] = (int32_t)next;
            nd.nchild[c] = nc[q];
#pragma unroll
            for (int d = 0; d < 8; d++) {
                if (bnd[q][d + 1] > bnd[q][d]) {
                    nd.first[next] = bnd[q][d];
                    nd.count[next] = bnd[q][d + 1] - bnd[q][d];
                    nd.parent[next] = (int32_t)c;
                    nd.child[next] = -1;
                    nd.nchild[next] = 0;
                    next++;
                }
            }
        }
        if (tile == ntiles - 1 && threadIdx.x == BT - 1) {
            unsigned long long end = (unsigned long long)hi + excl_sh + total;
            if (end > (unsigned long long)cap) {
                gt_set_error(ctl, GT_EOVERFLOW, GTK_BUILD);
                end = (unsigned long long)cap;
            }
            ctl->level_start[lvl + 2] = (uint32_t)end;
        }
    }
}

// ---- A4 in one sweep over the sorted keys (leaf_max <= FLAT_LWIN) ------------------
// d(p), the index of the first 3-bit digit in which keys p - 1 and p differ (21 for equal
// keys; -1 at p = 0 and p = n), says at which levels a new cell begins at particle p: a
// run of particles between two positions with d < l shares its first l digits, so it is
// one level-l cell of the full octree.  The tree keeps a level-l run iff its parent run
// holds more than leaf_max particles, so particle i's leaf is at the first level whose
// run around i holds at most leaf_max -- found from the d values within leaf_max of i.
// Particle i then starts a node at every level l with d(i) < l <= leaf level(i), and ends
// one (as its last particle) at every l with d(i + 1) < l <= leaf level(i).  Counting
// those starts and ends per level and tile, scanning, and scattering them by rank gives
// the same numbering as the level-by-level split: level by level, and inside a level by
// first particle.  A node's first child starts at its own first particle; the others
// are the next nodes of the child level that start before its end.
constexpr int FLAT_LWIN = GT_FLAT_LEAF_MAX;              // the largest leaf_max of this build
constexpr int FB = 256;                    // threads per block
// Particles per tile: a block takes its tile's rounds of FB particles one after another, so that small systems,
// which fill few blocks, get short tiles (8192 particles: k_flat_scatter 15.6 us with 8 rounds).  Whole builds with two
// and with eight: 2^20 291 and 296 us, 2^20.5 355 and 352, 2^21 443 and 444, 2^21.5 562 and 562, 2^22 769 and 761, 2^23
// 1423 and 1409.
#ifndef GT_FLAT_SMALL
#define GT_FLAT_SMALL (1 << 21)            // systems up to this size take tiles of two rounds, larger ones of eight
#endif
int flat_rounds(int64_t n) { return n <= GT_FLAT_SMALL ? 2 : 8; }
constexpr int NREC = 2 * GT_TREE_LEVELS;   // start and end counters per level

__device__ __forceinline__ int key_diff_digit(unsigned long long a, unsigned long long b) {
    const unsigned long long x = a ^ b;  // keys use bits 0..62, so clz >= 1
    return x ? (__clzll((long long)x) - 1) / 3 : GT_KEY_LEVELS;
}

// Leaf level of the particle at ds[j]: the run around it at level l holds at most M
// particles iff, for some a in [0, M), positions i - a .. i and i + 1 .. i + M - a both
// hold a d below l; so the leaf level is 1 + min over a of max(the smallest d of the
// first window, the smallest d of the second).  MT > 0: M = MT, unrolled in registers.
template <int MT>
__device__ __forceinline__ int leaf_level_of(const int8_t *ds, int j) {
    int mr[MT + 1];  // mr[b]: smallest d over i + 1 .. i + b
    int m = 127;
#pragma unroll
    for (int b = 1; b <= MT; b++) {
        m = min(m, (int)ds[j + b]);
        mr[b] = m;
    }
    int ml = 127, best = 127;
#pragma unroll
    for (int a = 0; a < MT; a++) {
        ml = min(ml, (int)ds[j - a]);
        best = min(best, max(ml, mr[MT - a]));
    }
    return min(best + 1, GT_KEY_LEVELS);
}

// d and the leaf level of every particle (packed (d + 1) | leaf << 8), and every tile's
// start and end counts per level (column-major: counter k of tile t at cnt[k * ntiles + t]).
// MT > 0: leaf_max == MT; MT == 0: any leaf_max up to FLAT_LWIN (running minima in shared memory).
template <int MT, int ROUNDS>
__device__ __forceinline__ void flat_marks_body(const unsigned bid, const unsigned nb,
        const unsigned long long *__restrict__ skey, long long n, int M, uint16_t *__restrict__ dl,
        uint32_t *__restrict__ cnt, int ntiles) {
    constexpr int W = FLAT_LWIN, FT = ROUNDS * FB;
    constexpr int MW = MT > 0 ? 1 : W;
    __shared__ int8_t ds[FT + 2 * W + 1];      // d of positions base - W .. base + FT + W
    __shared__ uint8_t mr[MW][FB];             // generic: 1 + smallest d over (i, i + b]
    __shared__ unsigned int c[NREC];
    const long long base = (long long)bid * FT;
    for (int j = threadIdx.x; j < FT + 2 * W + 1; j += FB) {
        const long long p = base - W + j;
        ds[j] = (int8_t)((p > 0 && p < n) ? key_diff_digit(skey[p - 1], skey[p]) : -1);
    }
    for (int j = threadIdx.x; j < NREC; j += FB) c[j] = 0;
    __syncthreads();
    for (int r = 0; r < ROUNDS; r++) {
        const int t = r * FB + threadIdx.x;
        const long long i = base + t;
        if (i >= n) break;
        const int j = t + W;  // position i in ds
        int leaf;
        if constexpr (MT > 0) {
            leaf = leaf_level_of<MT>(ds, j);
        } else {
            int m = 127;
            for (int b = 1; b <= M; b++) {
                m = min(m, (int)ds[j + b]);
                mr[b - 1][threadIdx.x] = (uint8_t)(m + 1);
            }
            int ml = 127, best = 127;
            for (int a = 0; a < M; a++) {
                ml = min(ml, (int)ds[j - a]);
                best = min(best, max(ml, (int)mr[M - a - 1][threadIdx.x] - 1));
            }
            leaf = min(best + 1, GT_KEY_LEVELS);
        }
        const int d0 = ds[j], d1 = ds[j + 1];
        dl[i] = (uint16_t)((d0 + 1) | (leaf << 8));
        for (int l = d0 + 1; l <= leaf; l++) atomicAdd(&c[l], 1u);
        for (int l = d1 + 1; l <= leaf; l++) atomicAdd(&c[GT_TREE_LEVELS + l], 1u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < NREC; k += FB) cnt[(size_t)k * ntiles + bid] = c[k];
}

template <int MT, int ROUNDS>
__global__ __launch_bounds__(FB) void k_flat_marks(const unsigned long long *__restrict__ skey, long long n, int M,
        uint16_t *__restrict__ dl, uint32_t *__restrict__ cnt, int ntiles) {
    gt_grid_ready();
    flat_marks_body<MT, ROUNDS>(blockIdx.x, gridDim.x, skey, n, M, dl, cnt, ntiles);
}

// The last block of a kernel to come here gets true (its threads see what the others wrote before); *done starts at
// zero and is left at zero.
__device__ __forceinline__ bool last_block(unsigned nb, unsigned int *done) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(done, 1u) == nb - 1u;
        if (last) *done = 0u;
    }
    __syncthreads();
    __threadfence();
    return last;
}

// one block per counter: exclusive scan over the tiles, the column total into tot[k]; the last block then sets the
// level starts from the per-level node counts (clamped to the node capacity) and clears the cell list's counters
__device__ __forceinline__ void flat_scan_body(const unsigned bid, const unsigned nb, uint32_t *__restrict__ cnt,
        int ntiles, uint32_t *__restrict__ tot, long long cap, DevCtl *ctl) {
    __shared__ unsigned int tmp[1024 / 32 + 1];
    uint32_t *col = cnt + (size_t)bid * ntiles;
    unsigned int carry = 0;
    for (int b0 = 0; b0 < ntiles; b0 += 1024) {
        const int t = b0 + (int)threadIdx.x;
        const unsigned int v = t < ntiles ? col[t] : 0u;
        unsigned int total;
        const unsigned int e = block_excl_scan<1024>(v, &total, tmp);
        if (t < ntiles) col[t] = carry + e;
        carry += total;
    }
    if (threadIdx.x == 0) tot[bid] = carry;
    if (!last_block(nb, &ctl->scan_done)) return;
    for (int b = threadIdx.x; b < GT_CELL_BUCKETS; b += 1024) ctl->cell_bucket[b] = 0;
    if (threadIdx.x >= 32) return;
    const int l = threadIdx.x;
    unsigned long long sum = l < GT_TREE_LEVELS ? __ldcg(&tot[l]) : 0ull;
    const unsigned long long own = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, sum, o);
        if (l >= o) sum += t;
    }
    const unsigned long long most = (unsigned long long)cap, before = l < GT_TREE_LEVELS ? sum - own : sum;
    if (l < GT_TREE_LEVELS + 2) ctl->level_start[l] = (uint32_t)(before < most ? before : most);
    if (l == GT_TREE_LEVELS && sum > most) gt_set_error(ctl, GT_EOVERFLOW, GTK_BUILD);
}

__global__ __launch_bounds__(1024) void k_flat_scan(uint32_t *__restrict__ cnt, int ntiles,
        uint32_t *__restrict__ tot, long long cap, DevCtl *ctl) {
    gt_grid_ready();
    flat_scan_body(blockIdx.x, gridDim.x, cnt, ntiles, tot, cap, ctl);
}

// every start and end to its node: first, the first child and the parent along a
// particle's own chain of starts, leaves; an end goes to count (as the end position)
template <int ROUNDS>
__device__ __forceinline__ void flat_scatter_body(const unsigned bid, const unsigned nb,
        const uint16_t *__restrict__ dl, long long n, const uint32_t *__restrict__ cnt, int ntiles, long long cap,
        Nodes nd, const DevCtl *__restrict__ ctl) {
    constexpr int FT = ROUNDS * FB;
    __shared__ uint32_t lb[GT_TREE_LEVELS];
    __shared__ uint32_t run[NREC];
    __shared__ uint32_t wc[FB / 32][NREC];
    __shared__ uint16_t dls[FT + 1];
    const long long base = (long long)bid * FT;
    for (int k = threadIdx.x; k < GT_TREE_LEVELS; k += FB) lb[k] = ctl->level_start[k];
    for (int k = threadIdx.x; k < NREC; k += FB) run[k] = cnt[(size_t)k * ntiles + bid];
    for (int j = threadIdx.x; j <= FT; j += FB) dls[j] = base + j < n ? dl[base + j] : (uint16_t)0;  // d(n) = -1
    __syncthreads();
    const int w = threadIdx.x >> 5;
    const unsigned int lt = lanemask_lt();
    for (int r = 0; r < ROUNDS; r++) {
        const int t = r * FB + threadIdx.x;
        const long long i = base + t;
        const bool valid = i < n;
        const int v = dls[t];
        const int slo = valid ? (v & 0xff) : GT_TREE_LEVELS, leaf = v >> 8;
        const int elo = valid ? (dls[t + 1] & 0xff) : GT_TREE_LEVELS;
        // ranks inside the round: per-warp counts, then warps in order after the tile's
        // offset; a warp visits only the levels at which one of its lanes has a record
        const int has = slo <= leaf || elo <= leaf;
        const int lmin = __reduce_min_sync(0xffffffffu, has ? min(slo, elo) : GT_TREE_LEVELS);
        const int lmax = __reduce_max_sync(0xffffffffu, has ? leaf : -1);
        if ((threadIdx.x & 31) < GT_TREE_LEVELS) {
            wc[w][threadIdx.x & 31] = 0;
            wc[w][GT_TREE_LEVELS + (threadIdx.x & 31)] = 0;
        }
        __syncwarp();
        for (int l = lmin; l <= lmax; l++) {
            const unsigned int bs = __ballot_sync(0xffffffffu, slo <= l && l <= leaf);
            const unsigned int be = __ballot_sync(0xffffffffu, elo <= l && l <= leaf);
            if ((threadIdx.x & 31) == 0) {
                wc[w][l] = __popc(bs);
                wc[w][GT_TREE_LEVELS + l] = __popc(be);
            }
        }
        __syncthreads();
        if (threadIdx.x < NREC) {
            uint32_t s = run[threadIdx.x];
            for (int q = 0; q < FB / 32; q++) {
                const uint32_t x = wc[q][threadIdx.x];
                wc[q][threadIdx.x] = s;
                s += x;
            }
            run[threadIdx.x] = s;
        }
        __syncthreads();
        long long prev = -1;  // this particle's node one level up, when it starts one there
        for (int l = lmin; l <= lmax; l++) {
            const bool hs = slo <= l && l <= leaf, he = elo <= l && l <= leaf;
            const unsigned int bs = __ballot_sync(0xffffffffu, hs);
            const unsigned int be = __ballot_sync(0xffffffffu, he);
            if (hs) {
                const long long id = (long long)lb[l] + wc[w][l] + __popc(bs & lt);
                if (prev >= 0) nd.child[prev] = id < cap ? (int32_t)id : -1;
                if (id < cap) {
                    nd.first[id] = (uint32_t)i;
                    if (l == 0 || prev >= 0) nd.parent[id] = (int32_t)prev;  // else: the link pass
                    if (l == leaf) {
                        nd.child[id] = -1;
                        nd.nchild[id] = 0;
                    }
                }
                prev = id < cap ? id : -1;
            }
            if (he) {
                const long long id = (long long)lb[l] + wc[w][GT_TREE_LEVELS + l] + __popc(be & lt);
                if (id < cap) nd.count[id] = (uint32_t)(i + 1);
            }
        }
        __syncthreads();  // wc is rewritten by the next round
    }
}

template <int ROUNDS>
__global__ __launch_bounds__(FB) void k_flat_scatter(const uint16_t *__restrict__ dl, long long n,
        const uint32_t *__restrict__ cnt, int ntiles, long long cap, Nodes nd, const DevCtl *__restrict__ ctl) {
    gt_grid_ready();
    flat_scatter_body<ROUNDS>(blockIdx.x, gridDim.x, dl, n, cnt, ntiles, cap, nd, ctl);
}

// per node: count = end - first; a node with children counts them (the nodes of the
// next level from its first child on that start before its end) and is their parent
__device__ __forceinline__ void flat_link_body(const unsigned bid, const unsigned nb, Nodes nd, long long cap,
        const DevCtl *__restrict__ ctl) {
    __shared__ uint32_t ls[GT_TREE_LEVELS + 2];
    for (int i = threadIdx.x; i < GT_TREE_LEVELS + 2; i += 256) ls[i] = ctl->level_start[i];
    __syncthreads();
    const long long nn = ls[GT_TREE_LEVELS];
    for (long long p = bid * 256ll + threadIdx.x; p < nn; p += (long long)nb * 256) {
        const uint32_t f = nd.first[p], e = nd.count[p];
        nd.count[p] = e - f;
        const int32_t c0 = nd.child[p];
        if (c0 < 0) continue;
        int lvl = 0;  // the last level starting at or before p
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (lvl + step < GT_TREE_LEVELS && ls[lvl + step] <= (uint32_t)p) lvl += step;
        long long hi = ls[lvl + 2];
        if (hi > cap) hi = cap;
        uint32_t nch = 1;
        for (int q = 1; q < 8; q++) {
            const long long c = (long long)c0 + q;
            if (c >= hi || nd.first[c] >= e) break;
            nd.parent[c] = (int32_t)p;
            nch++;
        }
        nd.nchild[p] = nch;
    }
}

__global__ __launch_bounds__(256) void k_flat_link(Nodes nd, long long cap, const DevCtl *__restrict__ ctl) {
    gt_grid_ready();
    flat_link_body(blockIdx.x, gridDim.x, nd, cap, ctl);
}

__device__ __forceinline__ float sq3f(float dx, float dy, float dz) {
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// ---- cell lists for the per-step pseudo j-particle pass ---------------------------
// Every node goes once into nd.cells, level by level; inside a level the leaves come
// first, bucketed by particle count (1..16, then all larger), then the cells with
// children, bucketed by number of children.  A warp of the pseudo-j pass then takes
// cells of one size, so the FP64 sums run with all lanes busy.  The order inside a
// bucket is free: every cell's result depends on its own particles or children only.

// bucket of node p, given the level ranges ls[0..GT_TREE_LEVELS]
__device__ __forceinline__ int cell_bucket_of(const Nodes &nd, uint32_t p, const uint32_t *ls) {
    int lvl = 0;  // the last level starting at or before p
#pragma unroll
    for (int step = 16; step > 0; step >>= 1)
        if (lvl + step < GT_TREE_LEVELS && ls[lvl + step] <= p) lvl += step;
    if (nd.child[p] < 0) {
        const uint32_t k = nd.count[p];
        return lvl * GT_LEVEL_BUCKETS + (k >= GT_LEAF_BUCKETS ? GT_LEAF_BUCKETS : (int)k) - 1;
    }
    return lvl * GT_LEVEL_BUCKETS + GT_LEAF_BUCKETS + (int)nd.nchild[p] - 1;
}

__device__ __forceinline__ void cell_count_body(const unsigned bid, const unsigned nb, Nodes nd, long long cap,
        DevCtl *ctl) {
    __shared__ uint32_t ls[GT_TREE_LEVELS + 1];
    __shared__ uint32_t h[GT_CELL_BUCKETS];
    for (int i = threadIdx.x; i <= GT_TREE_LEVELS; i += 256) ls[i] = ctl->level_start[i];
    for (int i = threadIdx.x; i < GT_CELL_BUCKETS; i += 256) h[i] = 0;
    __syncthreads();
    long long nn = ls[GT_TREE_LEVELS];
    if (nn > cap) nn = cap;
    for (long long p = bid * 256ll + threadIdx.x; p < nn; p += (long long)nb * 256)
        atomicAdd(&h[cell_bucket_of(nd, (uint32_t)p, ls)], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < GT_CELL_BUCKETS; i += 256)
        if (h[i]) atomicAdd(&ctl->cell_bucket[i], h[i]);
    if (!last_block(nb, &ctl->cells_done)) return;
    // bucket sizes -> fill cursors, and where every level's leaves and cells with children start
    constexpr int PER = (GT_CELL_BUCKETS + 255) / 256;  // neighbouring buckets of a thread
    __shared__ unsigned int tmp[256 / 32 + 1];
    uint32_t v[PER], sum = 0, total;
#pragma unroll
    for (int j = 0; j < PER; j++) {
        const int b = PER * (int)threadIdx.x + j;
        v[j] = b < GT_CELL_BUCKETS ? __ldcg(&ctl->cell_bucket[b]) : 0u;
        sum += v[j];
    }
    __shared__ uint32_t seg[2 * GT_TREE_LEVELS + 1];
    uint32_t start = block_excl_scan<256>(sum, &total, tmp);
#pragma unroll
    for (int j = 0; j < PER; j++) {
        const int b = PER * (int)threadIdx.x + j;
        if (b < GT_CELL_BUCKETS) {
            ctl->cell_bucket[b] = start;
            const int q = b % GT_LEVEL_BUCKETS;
            if (q == 0) seg[2 * (b / GT_LEVEL_BUCKETS)] = start;
            if (q == GT_LEAF_BUCKETS) seg[2 * (b / GT_LEVEL_BUCKETS) + 1] = start;
        }
        start += v[j];
    }
    if (threadIdx.x == 0) seg[2 * GT_TREE_LEVELS] = total;
    __syncthreads();
    if (threadIdx.x <= 2 * GT_TREE_LEVELS) ctl->seg[threadIdx.x] = seg[threadIdx.x];
    if (threadIdx.x >= 32) return;
    // flat (a walk of it packs its batches): fewer than five children per cell, and fewer than 4.5 averaged over the levels
    const int l = threadIdx.x;
    const uint32_t parents = l < GT_KEY_LEVELS ? seg[2 * l + 2] - seg[2 * l + 1] : 0u;
    const uint32_t children = parents ? seg[2 * l + 4] - seg[2 * l + 2] : 0u;
    const uint32_t sixteenths = parents ? (uint32_t)(16ull * children / parents) : 0u;
    const unsigned levels = __ballot_sync(0xffffffffu, parents != 0u);
    const uint32_t by_level = __reduce_add_sync(0xffffffffu, sixteenths);
    const uint32_t all_parents = __reduce_add_sync(0xffffffffu, parents);
    const uint32_t all_children = __reduce_add_sync(0xffffffffu, children);
    if (l == 0) ctl->flat = all_children < 5ull * all_parents && by_level < 72u * __popc(levels) ? 1u : 0u;
}

__global__ __launch_bounds__(256) void k_cell_count(Nodes nd, long long cap, DevCtl *ctl) {
    gt_grid_ready();
    cell_count_body(blockIdx.x, gridDim.x, nd, cap, ctl);
}

// A block takes a contiguous range of nodes, counts them per bucket in shared memory,
// reserves its room in every bucket with one global atomic each, and fills it.
constexpr int CF_NODES = 4096;  // most nodes of such a range; small trees take shorter ones, so that every block has one

__device__ __forceinline__ void cell_fill_body(const unsigned bid, const unsigned nb, Nodes nd, long long cap,
        DevCtl *ctl) {
    __shared__ uint32_t ls[GT_TREE_LEVELS + 1];
    __shared__ uint32_t h[GT_CELL_BUCKETS];
    for (int i = threadIdx.x; i <= GT_TREE_LEVELS; i += 256) ls[i] = ctl->level_start[i];
    long long nn = ctl->level_start[GT_TREE_LEVELS];
    if (nn > cap) nn = cap;
    const long long share = ((nn + nb - 1) / nb + 255) / 256 * 256;
    const long long chunk = share < CF_NODES ? share : CF_NODES;
    for (long long b0 = (long long)bid * chunk; b0 < nn; b0 += (long long)nb * chunk) {
        __syncthreads();
        for (int i = threadIdx.x; i < GT_CELL_BUCKETS; i += 256) h[i] = 0;
        __syncthreads();
        const long long b1 = b0 + chunk < nn ? b0 + chunk : nn;
        for (long long p = b0 + threadIdx.x; p < b1; p += 256)
            atomicAdd(&h[cell_bucket_of(nd, (uint32_t)p, ls)], 1u);
        __syncthreads();
        for (int i = threadIdx.x; i < GT_CELL_BUCKETS; i += 256)
            if (h[i]) h[i] = atomicAdd(&ctl->cell_bucket[i], h[i]);
        __syncthreads();
        for (long long p = b0 + threadIdx.x; p < b1; p += 256)
            nd.cells[atomicAdd(&h[cell_bucket_of(nd, (uint32_t)p, ls)], 1u)] = (uint32_t)p;
    }
}

__global__ __launch_bounds__(256) void k_cell_fill(Nodes nd, long long cap, DevCtl *ctl) {
    gt_grid_ready();
    cell_fill_body(blockIdx.x, gridDim.x, nd, cap, ctl);
}

// ---- A5: pseudo j-particles, every node in one launch ------------------------------
// The cell list's segments (a level's leaves, a level's cells with children) are cut
// into chunks of PL nodes, handed out by a ticket counter in this order: the leaves of
// level 21; then, for l = 20 .. 0, the leaves of level l and the cells with children of
// level l + 1; the cells of level 0 last.  A chunk of cells of level l waits until every
// chunk of level l + 1 is finished: those hold smaller tickets, so the blocks holding
// them are running and the wait ends (it is bounded all the same).  Leaves wait for
// nothing, so their FP64 sums fill the time a level's cells wait for the one below.
#ifndef GT_PSEUDO_PU
#define GT_PSEUDO_PU 2  // a leaf's particles loaded per round
#endif
#ifndef GT_PSEUDO_CU
#define GT_PSEUDO_CU 2  // a cell's children loaded per round
#endif
#ifndef GT_PSEUDO_COOP
#define GT_PSEUDO_COOP 16384  // a level's cells with children taken eight lanes each when at most this many
#endif
#ifndef GT_PSEUDO_MINB
#define GT_PSEUDO_MINB 6  // resident blocks per SM (the grid) the register budget is sized for
#endif
constexpr int PL = 128;  // nodes per chunk, one per thread
constexpr uint32_t PU = GT_PSEUDO_PU, CU = GT_PSEUDO_CU;
constexpr int NSEG = 2 * GT_TREE_LEVELS;

// Leaf c: one lane sums its particles in FP64 (mass, m x, m y, m z) in particle order.
// The masses and the cells' members do not change between tree builds, so the mass
// sums are formed at a build (WITH_MASS) and read back at the other block steps: the
// same values, one FP64 addition per particle fewer.
template <bool WITH_MASS>
__device__ __forceinline__ void pseudo_leaf(const Nodes &nd, const float4 *__restrict__ posm, uint32_t c) {
    const uint32_t f = nd.first[c];
    const uint32_t k = nd.count[c];
    double m = WITH_MASS ? 0.0 : nd.sum[c].m, sx = 0.0, sy = 0.0, sz = 0.0;
    // in particle order; the loads of PU particles go out before their sums
    // (m x is exact in FP64, so the fused form rounds once like + does)
    for (uint32_t i0 = f; i0 < f + k; i0 += PU) {
        float4 p[PU];
#pragma unroll
        for (uint32_t q = 0; q < PU; q++)
            if (i0 + q < f + k) p[q] = posm[i0 + q];
#pragma unroll
        for (uint32_t q = 0; q < PU; q++)
            if (i0 + q < f + k) {
                const double mi = f2d(p[q].w);
                if (WITH_MASS) m = __dadd_rn(m, mi);
                sx = __fma_rn(mi, f2d(p[q].x), sx);
                sy = __fma_rn(mi, f2d(p[q].y), sy);
                sz = __fma_rn(mi, f2d(p[q].z), sz);
            }
    }
    float jx, jy, jz;
    if (k == 1) {  // a cell of one particle is that particle
        const float4 p = posm[f];
        jx = p.x; jy = p.y; jz = p.z;
    } else {
        const float mf = d2f(m);
        jx = __fdiv_rn(d2f(sx), mf);
        jy = __fdiv_rn(d2f(sy), mf);
        jz = __fdiv_rn(d2f(sz), mf);
    }
    float d2max = 0.0f, b2 = 0.0f;  // b2: B_2 of the multipole MAC
    for (uint32_t i0 = f; i0 < f + k; i0 += PU) {
        float4 p[PU];
#pragma unroll
        for (uint32_t q = 0; q < PU; q++)
            if (i0 + q < f + k) p[q] = posm[i0 + q];
#pragma unroll
        for (uint32_t q = 0; q < PU; q++)
            if (i0 + q < f + k) {
                const float d2 = sq3f(__fsub_rn(p[q].x, jx), __fsub_rn(p[q].y, jy), __fsub_rn(p[q].z, jz));
                if (d2 > d2max) d2max = d2;
                b2 = __fadd_rn(b2, __fmul_rn(p[q].w, d2));
            }
    }
    nd.sum[c] = DSum4{m, sx, sy, sz};
    nd.jpos[c] = make_float4(jx, jy, jz, d2f(m));
    nd.walk[c] = make_float4(__fmul_rn(__fsqrt_rn(d2max), GT_RADIUS_MARGIN), __uint_as_float(f),
                             __uint_as_float(k | GT_LEAF_FLAG), b2);
}

// What a cell's lane reads of the cell itself, before it waits for the level below.
struct CellInfo {
    uint32_t p, nch;
    int32_t ch0;
    double m;  // the stored mass (WITH_MASS: 0, it is summed)
};

template <bool WITH_MASS>
__device__ __forceinline__ CellInfo cell_info(const Nodes &nd, uint32_t p) {
    return CellInfo{p, nd.nchild[p], nd.child[p], WITH_MASS ? 0.0 : nd.sum[p].m};
}

// Cell p with children: its children's FP64 sums added in child order.  The children
// were written by other blocks of this launch: they are read through L2 (__ldcg), an
// SM's L1 may hold a line of them from before they were written.  Loads go out CU
// children at a time, so a level costs few L2 round trips.
template <bool WITH_MASS>
__device__ __forceinline__ void pseudo_cell(const Nodes &nd, const CellInfo &ci) {
    const uint32_t p = ci.p, nch = ci.nch;
    const int32_t ch0 = ci.ch0;
    double m = ci.m, sx = 0.0, sy = 0.0, sz = 0.0;
    for (uint32_t q0 = 0; q0 < nch; q0 += CU) {
        double2 s0[CU], s1[CU];  // (m, x), (y, z)
#pragma unroll
        for (uint32_t q = 0; q < CU; q++)
            if (q0 + q < nch) {
                const double2 *cs = (const double2 *)&nd.sum[ch0 + q0 + q];
                s0[q] = __ldcg(cs);
                s1[q] = __ldcg(cs + 1);
            }
#pragma unroll
        for (uint32_t q = 0; q < CU; q++)
            if (q0 + q < nch) {
                if (WITH_MASS) m = __dadd_rn(m, s0[q].x);
                sx = __dadd_rn(sx, s0[q].y);
                sy = __dadd_rn(sy, s1[q].x);
                sz = __dadd_rn(sz, s1[q].y);
            }
    }
    const float mf = d2f(m);
    const float jx = __fdiv_rn(d2f(sx), mf);
    const float jy = __fdiv_rn(d2f(sy), mf);
    const float jz = __fdiv_rn(d2f(sz), mf);
    float b = 0.0f, b2 = 0.0f;  // b2: B_2 by parallel axes
    for (uint32_t q0 = 0; q0 < nch; q0 += CU) {
        float4 cj[CU], cw[CU];
#pragma unroll
        for (uint32_t q = 0; q < CU; q++)
            if (q0 + q < nch) {
                cj[q] = __ldcg(&nd.jpos[ch0 + q0 + q]);
                cw[q] = __ldcg(&nd.walk[ch0 + q0 + q]);
            }
#pragma unroll
        for (uint32_t q = 0; q < CU; q++)
            if (q0 + q < nch) {
                const float d2 = sq3f(__fsub_rn(cj[q].x, jx), __fsub_rn(cj[q].y, jy), __fsub_rn(cj[q].z, jz));
                const float e = __fadd_rn(__fsqrt_rn(d2), cw[q].x);
                if (e > b) b = e;
                b2 = __fadd_rn(b2, __fadd_rn(cw[q].w, __fmul_rn(cj[q].w, d2)));
            }
    }
    nd.sum[p] = DSum4{m, sx, sy, sz};
    nd.jpos[p] = make_float4(jx, jy, jz, mf);
    nd.walk[p] = make_float4(__fmul_rn(b, GT_RADIUS_MARGIN), __uint_as_float((uint32_t)ch0),
                             __uint_as_float(nch), b2);
}

// The same cell with eight lanes, one child each (lanes 8g .. 8g + 7 of the warp hold cell
// g of four): the children's records arrive in one round of loads instead of one per
// pair of children.  The FP64 sums and the B_2 sum are formed in child order from the lanes'
// values (shuffles), so the operations and their
// order are those of pseudo_cell; the radius is a maximum, taken across the lanes.  For
// the levels near the root, whose few cells each wait for the level below.  Every lane
// of the warp must call it; `valid` marks groups that own a cell.
template <bool WITH_MASS>
__device__ __forceinline__ void pseudo_cell_coop(const Nodes &nd, const CellInfo &ci, bool valid) {
    const uint32_t p = ci.p, nch = ci.nch;
    const int32_t ch0 = ci.ch0;
    const unsigned FULL = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31u, j = lane & 7u, g0 = lane & ~7u;
    const bool has = j < nch;
    double2 s0 = make_double2(0.0, 0.0), s1 = make_double2(0.0, 0.0);  // (m, x), (y, z)
    float4 cj = make_float4(0.f, 0.f, 0.f, 0.f), cw = make_float4(0.f, 0.f, 0.f, 0.f);
    if (has) {
        const double2 *cs = (const double2 *)&nd.sum[ch0 + j];
        s0 = __ldcg(cs);
        s1 = __ldcg(cs + 1);
        cj = __ldcg(&nd.jpos[ch0 + j]);
        cw = __ldcg(&nd.walk[ch0 + j]);
    }
    // lanes 0 to 3 of the group sum a component each (the FP64 unit takes 16 cycles per warp instruction, so that the
    // four sums on every lane were half of a level's time)
    double acc = j == 0 ? ci.m : 0.0;
#pragma unroll
    for (uint32_t q = 0; q < 8; q++) {
        const double cm = __shfl_sync(FULL, s0.x, g0 + q), cx = __shfl_sync(FULL, s0.y, g0 + q);
        const double cy = __shfl_sync(FULL, s1.x, g0 + q), cz = __shfl_sync(FULL, s1.y, g0 + q);
        const double c = j == 0 ? cm : (j == 1 ? cx : (j == 2 ? cy : cz));
        if (q < nch && (WITH_MASS || j != 0)) acc = __dadd_rn(acc, c);
    }
    const float af = d2f(acc), mf = __shfl_sync(FULL, af, g0);
    const float jf = __fdiv_rn(af, mf);
    const float jx = __shfl_sync(FULL, jf, g0 + 1), jy = __shfl_sync(FULL, jf, g0 + 2),
                jz = __shfl_sync(FULL, jf, g0 + 3);
    const double m = __shfl_sync(FULL, acc, g0), sx = __shfl_sync(FULL, acc, g0 + 1),
                 sy = __shfl_sync(FULL, acc, g0 + 2), sz = __shfl_sync(FULL, acc, g0 + 3);
    const float d2 = sq3f(__fsub_rn(cj.x, jx), __fsub_rn(cj.y, jy), __fsub_rn(cj.z, jz));
    float b = 0.0f;
    if (has) {
        const float e = __fadd_rn(__fsqrt_rn(d2), cw.x);
        if (e > b) b = e;
    }
    const float t = __fadd_rn(cw.w, __fmul_rn(cj.w, d2));
    float b2 = 0.0f;
#pragma unroll
    for (uint32_t q = 0; q < 8; q++) {
        const float tq = __shfl_sync(FULL, t, g0 + q);
        if (q < nch) b2 = __fadd_rn(b2, tq);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const float bo = __shfl_xor_sync(FULL, b, o);
        if (bo > b) b = bo;
    }
    if (valid && j == 0) {
        nd.sum[p] = DSum4{m, sx, sy, sz};
        nd.jpos[p] = make_float4(jx, jy, jz, mf);
        nd.walk[p] = make_float4(__fmul_rn(b, GT_RADIUS_MARGIN), __uint_as_float((uint32_t)ch0),
                                 __uint_as_float(nch), b2);
    }
}

template <bool WITH_MASS>
__device__ __forceinline__ void pseudo_body(const unsigned bid, const unsigned nb, Nodes nd,
        const float4 *__restrict__ posm, DevCtl *ctl) {
    __shared__ uint32_t seg[NSEG + 1];
    __shared__ uint8_t olvl[NSEG], ocell[NSEG];      // ticket order: segment level and kind
    __shared__ uint32_t ocum[NSEG + 1];              // first ticket of every entry
    __shared__ uint32_t nchunk[NSEG];                // chunks of segment (2 l + kind)
    __shared__ uint8_t coop[NSEG];                   // cells of the segment taken eight lanes each
    __shared__ unsigned int t_sh;
    __shared__ int o_sh, bad_sh;
    for (int i = threadIdx.x; i <= NSEG; i += PL) seg[i] = ctl->seg[i];
    __syncthreads();
    for (int k = threadIdx.x; k < NSEG; k += PL) {
        const uint32_t cnt = seg[k + 1] - seg[k];
        coop[k] = (k & 1) && cnt <= (uint32_t)GT_PSEUDO_COOP;
        const uint32_t per = coop[k] ? PL / 8 : PL;
        nchunk[k] = (cnt + per - 1) / per;
        // the order of entries: the leaves of levels 21 and 20; then for l = 19 .. 0 the leaves of level l and the cells
        // with children of level l + 1; those of level 0; an empty entry (level 21 has no cells with children)
        const int kind = k < 2 ? 0 : (k < NSEG - 2 ? (k & 1) : k - (NSEG - 3));
        const int lvl = k < 2 ? GT_TREE_LEVELS - 1 - k : (k < NSEG - 2 ? GT_TREE_LEVELS - 2 + (k & 1) - k / 2 : 0);
        olvl[k] = (uint8_t)lvl;
        ocell[k] = (uint8_t)kind;
    }
    if (threadIdx.x == 0) bad_sh = 0;
    __syncthreads();
    if (threadIdx.x < 32) {  // first tickets: entries l and l + 32 of lane l
        const uint32_t l = threadIdx.x;
        auto chunks = [&](uint32_t k) { return k < NSEG && ocell[k] < 2 ? nchunk[2 * olvl[k] + ocell[k]] : 0u; };
        const uint32_t c0 = chunks(l), c1 = chunks(l + 32);
        const uint32_t i0 = warp_incl_scan(c0), half = __shfl_sync(0xffffffffu, i0, 31), i1 = half + warp_incl_scan(c1);
        ocum[l] = i0 - c0;
        if (l + 32 <= NSEG) ocum[l + 32] = i1 - c1;
    }
    __syncthreads();
    const uint32_t total = ocum[NSEG];
    for (;;) {
        if (threadIdx.x < 32) {
            unsigned int t = 0;
            if (threadIdx.x == 0) t = atomicAdd(&ctl->pl_ticket, 1u);
            t = __shfl_sync(0xffffffffu, t, 0);
            // the last entry that begins at or before t
            static_assert(NSEG <= 64, "two entries per lane");
            int o = __popc(__ballot_sync(0xffffffffu, ocum[threadIdx.x + 1] <= t));
            o += __popc(__ballot_sync(0xffffffffu, threadIdx.x + 33 <= NSEG && ocum[min(threadIdx.x + 33u, (uint32_t)NSEG)] <= t));
            if (threadIdx.x == 0) {
                t_sh = t;
                o_sh = o < NSEG ? o : NSEG - 1;
            }
        }
        __syncthreads();
        const unsigned int t = t_sh;
        const int o = o_sh;
        if (t >= total) break;
        const int lvl = olvl[o], kind = ocell[o], sg = 2 * lvl + kind;
#if GT_DEBUG
        {   // every node of the chunk: its particle or child range inside the tree
            const uint32_t nn = ctl->level_start[GT_TREE_LEVELS], np = nd.count[0];
            const uint32_t per = coop[sg] ? PL / 8 : PL;
            const long long i0 = (long long)seg[sg] + (long long)(t - ocum[o]) * per;
            bool bad = false;
            for (long long i = i0 + threadIdx.x; i < i0 + per && i < (long long)seg[sg + 1]; i += PL) {
                const uint32_t c = nd.cells[i];
                if (c >= nn) { bad = true; continue; }
                bad |= kind == 0 ? ((unsigned long long)nd.first[c] + nd.count[c] > np)
                                 : (nd.child[c] < 0 || (unsigned long long)nd.child[c] + nd.nchild[c] > nn);
            }
            if (__syncthreads_or(bad)) {  // the whole chunk is skipped
                if (threadIdx.x == 0) {
                    gt_set_error(ctl, GT_EINVAL, GTK_PSEUDO);
                    atomicAdd(&ctl->pl_done[lvl], 1u);
                }
                continue;
            }
        }
#endif
        const uint32_t per = coop[sg] ? PL / 8 : PL;  // coop: eight lanes each
        const long long idx = (long long)seg[sg] + (long long)(t - ocum[o]) * per + (coop[sg] ? threadIdx.x >> 3 : threadIdx.x);
        const bool valid = idx < (long long)seg[sg + 1];
        const uint32_t node = valid ? nd.cells[idx] : 0u;
        if (kind == 0) {
            if (valid) pseudo_leaf<WITH_MASS>(nd, posm, node);
        } else {
            CellInfo ci{0u, 0u, 0, 0.0};
            if (valid) ci = cell_info<WITH_MASS>(nd, node);
            if (threadIdx.x == 0 && lvl + 1 < GT_TREE_LEVELS) {
                const int l1 = lvl + 1;  // every chunk of that level first
                const unsigned int need = nchunk[2 * l1] + nchunk[2 * l1 + 1];
                unsigned int spins = 0;
                const unsigned int limit = gt_spin_limit(ctl);
                while (*((volatile unsigned int *)&ctl->pl_done[l1]) < need) {
                    if (++spins > limit) {
                        gt_set_error(ctl, GT_ETIMEOUT, GTK_PSEUDO);
                        bad_sh = 1;
                        break;
                    }
                    __nanosleep(20);
                }
                __threadfence();
            }
            __syncthreads();
            if (bad_sh) break;
            if (coop[sg]) pseudo_cell_coop<WITH_MASS>(nd, ci, valid);
            else if (valid) pseudo_cell<WITH_MASS>(nd, ci);
        }
        __syncthreads();
        if (threadIdx.x == 0) {  // the block's nodes are visible device-wide before the chunk counts as done
            __threadfence();
            atomicAdd(&ctl->pl_done[lvl], 1u);
        }
    }
}

template <bool WITH_MASS>
__global__ __launch_bounds__(PL, GT_PSEUDO_MINB) void k_pseudo(Nodes nd, const float4 *__restrict__ posm, DevCtl *ctl) {
    gt_grid_ready();
    pseudo_body<WITH_MASS>(blockIdx.x, gridDim.x, nd, posm, ctl);
}

// ---- a table of systems (two rounds of marks each: GT_GROUPED_MOST is below GT_FLAT_SMALL) ----
struct FlatScratch {
    uint16_t *dl;
    uint32_t *cnt, *tot;
    int ntiles;
    __host__ __device__ FlatScratch(uint8_t *scratch, long long n, int rounds) {
        ntiles = (int)((n + rounds * FB - 1) / (rounds * FB));
        dl = (uint16_t *)scratch;
        cnt = (uint32_t *)(scratch + (2 * (size_t)(n > 0 ? n : 1) + 15) / 16 * 16);
        tot = cnt + (size_t)NREC * ntiles;
    }
};

template <int MT>
__global__ __launch_bounds__(FB) void kg_flat_marks(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const FlatScratch f(s.bscratch, s.n, 2);
    if ((s.flags & GT_SYS_BUILD) && (int)blockIdx.y < f.ntiles)
        flat_marks_body<MT, 2>(blockIdx.y, (unsigned)f.ntiles, (const unsigned long long *)s.sb.key[0], s.n, s.leaf_max,
                               f.dl, f.cnt, f.ntiles);
}

__global__ __launch_bounds__(1024) void kg_flat_scan(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const FlatScratch f(s.bscratch, s.n, 2);
    if (s.flags & GT_SYS_BUILD) flat_scan_body(blockIdx.y, NREC, f.cnt, f.ntiles, f.tot, s.cap, s.ctl);
}

__global__ __launch_bounds__(FB) void kg_flat_scatter(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const FlatScratch f(s.bscratch, s.n, 2);
    if ((s.flags & GT_SYS_BUILD) && (int)blockIdx.y < f.ntiles)
        flat_scatter_body<2>(blockIdx.y, (unsigned)f.ntiles, f.dl, s.n, f.cnt, f.ntiles, s.cap, s.nd, s.ctl);
}

__global__ __launch_bounds__(256) void kg_flat_link(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 256, nsm * 8);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb) flat_link_body(blockIdx.y, nb, s.nd, s.cap, s.ctl);
}

__global__ __launch_bounds__(256) void kg_cell_count(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 512, nsm * 4);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb) cell_count_body(blockIdx.y, nb, s.nd, s.cap, s.ctl);
}

__global__ __launch_bounds__(256) void kg_cell_fill(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 1024, nsm * 2);
    if ((s.flags & GT_SYS_BUILD) && blockIdx.y < nb) cell_fill_body(blockIdx.y, nb, s.nd, s.cap, s.ctl);
}

__global__ __launch_bounds__(PL, GT_PSEUDO_MINB) void kg_pseudo(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    if (blockIdx.y >= gt_grid(s.n, 64, nsm * GT_PSEUDO_MINB)) return;
    if (s.flags & GT_SYS_BUILD) pseudo_body<true>(blockIdx.y, gridDim.y, s.nd, s.posm, s.ctl);
    else pseudo_body<false>(blockIdx.y, gridDim.y, s.nd, s.posm, s.ctl);
}

}  // namespace

size_t gt_build_scratch_bytes(int64_t n) {
    const size_t N = (size_t)(n > 0 ? n : 1);
    const size_t FT = (size_t)flat_rounds(n) * FB, tiles = (N + FT - 1) / FT;
    return (2 * N + 15) / 16 * 16 + 4 * (size_t)NREC * (tiles + 1);
}

namespace {

template <int ROUNDS>
void launch_flat(const unsigned long long *k, int64_t n, int leaf_max, Nodes nd, int64_t cap, uint8_t *scratch,
                 DevCtl *ctl, int nsm, cudaStream_t st) {
    const FlatScratch f(scratch, n, ROUNDS);
    if (f.ntiles > 0) {
        auto marks = k_flat_marks<0, ROUNDS>;
        switch (leaf_max) {
        case 4: marks = k_flat_marks<4, ROUNDS>; break;
        case 8: marks = k_flat_marks<8, ROUNDS>; break;
        case 16: marks = k_flat_marks<16, ROUNDS>; break;
        case 24: marks = k_flat_marks<24, ROUNDS>; break;
        case 32: marks = k_flat_marks<32, ROUNDS>; break;
        }
        gt_launch(marks, f.ntiles, FB, 0, st, k, n, leaf_max, f.dl, f.cnt, f.ntiles);
        gt_note_launches(1);
    }
    { gt_launch(k_flat_scan, NREC, 1024, 0, st, f.cnt, f.ntiles, f.tot, cap, ctl); gt_note_launches(1); }
    if (f.ntiles > 0) {
        gt_launch(k_flat_scatter<ROUNDS>, f.ntiles, FB, 0, st, f.dl, n, f.cnt, f.ntiles, cap, nd, ctl);
        { gt_launch(k_flat_link, gt_grid(n, 256, nsm * 8), 256, 0, st, nd, cap, ctl); }
        gt_note_launches(2);
    }
}

}  // namespace

void gt_launch_build(const uint64_t *skey, int64_t n, int leaf_max, Nodes nd, int64_t cap,
                     unsigned long long *status, uint8_t *scratch, DevCtl *ctl, int nsm, cudaStream_t st) {
    if (leaf_max <= FLAT_LWIN) {
        const unsigned long long *k = (const unsigned long long *)skey;
        if (flat_rounds(n) == 2) launch_flat<2>(k, n, leaf_max, nd, cap, scratch, ctl, nsm, st);
        else launch_flat<8>(k, n, leaf_max, nd, cap, scratch, ctl, nsm, st);
        return;
    }
    { k_build_init<<<1, 256, 0, st>>>(n, nd, ctl); gt_note_launches(1); }
    for (int l = 0; l < GT_TREE_LEVELS; l++)
        { k_build_level<<<nsm * 4, BT, 0, st>>>(l, (const unsigned long long *)skey, leaf_max, nd, cap,
                                              status, ctl); gt_note_launches(1); }
}

void gt_launch_cell_lists(Nodes nd, int64_t n, int64_t cap, DevCtl *ctl, int nsm, cudaStream_t st) {
    { gt_launch(k_cell_count, gt_grid(n, 512, nsm * 4), 256, 0, st, nd, cap, ctl); gt_note_launches(1); }
    { gt_launch(k_cell_fill, gt_grid(n, 1024, nsm * 2), 256, 0, st, nd, cap, ctl); gt_note_launches(1); }
}

void gt_launch_pseudo(Nodes nd, int64_t n, const float4 *posm, DevCtl *ctl, int nsm, bool with_mass,
                      cudaStream_t st) {
    // the ticket and the per-level counters were cleared by gt_launch_prepare
    const unsigned grid = gt_grid(n, 64, nsm * GT_PSEUDO_MINB);
    if (with_mass) { gt_launch(k_pseudo<true>, grid, PL, 0, st, nd, posm, ctl); }
    else { gt_launch(k_pseudo<false>, grid, PL, 0, st, nd, posm, ctl); }
    gt_note_launches(1);
}

void gt_grouped_build(const GroupedSys *t, const GroupedPlan &p, int nsm, cudaStream_t st) {
    static_assert(GT_GROUPED_MOST <= GT_FLAT_SMALL, "two rounds");
    const int64_t n = p.n_build;
    if (n <= 0) return;
    auto marks = kg_flat_marks<0>;
    switch (p.leaf_max) {
    case 4: marks = kg_flat_marks<4>; break;
    case 8: marks = kg_flat_marks<8>; break;
    case 16: marks = kg_flat_marks<16>; break;
    case 24: marks = kg_flat_marks<24>; break;
    case 32: marks = kg_flat_marks<32>; break;
    }
    const unsigned tiles = (unsigned)((n + 2 * FB - 1) / (2 * FB));
    gt_launch(marks, dim3(p.count, tiles), FB, 0, st, t);
    gt_launch(kg_flat_scan, dim3(p.count, NREC), 1024, 0, st, t);
    gt_launch(kg_flat_scatter, dim3(p.count, tiles), FB, 0, st, t);
    gt_launch(kg_flat_link, dim3(p.count, gt_grid(n, 256, nsm * 8)), 256, 0, st, t, nsm);
    gt_launch(kg_cell_count, dim3(p.count, gt_grid(n, 512, nsm * 4)), 256, 0, st, t, nsm);
    gt_launch(kg_cell_fill, dim3(p.count, gt_grid(n, 1024, nsm * 2)), 256, 0, st, t, nsm);
    gt_note_launches(6);
}

void gt_grouped_pseudo(const GroupedSys *t, const GroupedPlan &p, int nsm, cudaStream_t st) {
    // A block of a system waits for that system's blocks only, so all systems should have some at once: the systems
    // vary fastest, and four grids' worth of blocks let those of finished systems make room for the others'.
    const int most = nsm * GT_PSEUDO_MINB, share = (4 * most + p.count - 1) / p.count;
    gt_launch(kg_pseudo, dim3(p.count, gt_grid(p.n_all, 64, share < most ? share : most)), PL, 0, st, t, nsm);
    gt_note_launches(1);
}
