// Block time step (Sec. 1; Sec. 2.7, Eqs. 15-17), active sets and groups, and the
// particle-array plumbing:
//   k_prepare      per-phase bookkeeping (epoch, tickets, the step's block time)
//   k_predict      A8: r(T) = fma((T - t0) dt_min, v^{1/2}, r0) for every particle, FP64,
//                  rounded to FP32 for the tree                    (HBM: 60 B read, 16 B written)
//   k_permute      A3: gather every particle array into key order  (HBM: ~100 B each way)
//   k_compact      A6: order-preserving compaction with a block scan and a bounded decoupled
//                  look-back; selects by block time (t0 + ticks(level) == T) and writes the actives
//                  and, per 32 particles, their mask and the number of actives before (from
//                  which rank_at has the number below any i: 1/16 of the 4 B per particle of a prefix)
//                  (HBM: 9 B read per particle, 4 B per active)
//   k_compact_bits A6: the same for a bit mask (a caller's list, group starts), which it clears
//   k_group_cells  A6: groups bounded by tree cells (Sec. 2.4): the actives of every maximal
//                  cell with at most group_max of them (or of a leaf, cut into runs)
//   k_correct      A9: Eq. (17), the new level, the next half kick; the active particles'
//                  new step ends are folded into the next block time
//   k_init_levels  start: dt_max, levels and the first half kick
// Level of a particle: the smallest k with dt_k = dt_max 2^-k <= dt_i = sqrt(c/|a|),
// c = 2 eta eps, clamped to [0, L-1]; equivalently 2^(4(M-k)) A2 <= c2 with
// A2 = (ax^2 + ay^2) + az^2 and c2 = c c in FP64, decided exactly on the exponents
// (no root, no division: FP64 throughput is low on this GPU).  A shorter step is taken
// at once; a longer one only by one level and only when T is a multiple of it.  Every
// FP64 operation carries an explicit rounding, so results are reproducible bit for bit.
#include <float.h>

#include "gt_internal.cuh"

namespace {

__device__ __forceinline__ void prepare_body(const unsigned bid, const unsigned nb, DevCtl *ctl, int begin_step) {  // one warp
    static_assert(GT_TREE_LEVELS + 4 <= 32, "a lane per ticket");
    const int l = threadIdx.x;
    if (l < GT_TREE_LEVELS + 4) ctl->tile_ticket[l] = 0;
    if (l < GT_TREE_LEVELS) ctl->pl_done[l] = 0;
    if (l < 6) ctl->bbox[l] = gt_ordered(l < 3 ? FLT_MAX : -FLT_MAX);
    if (l != 0) return;
    ctl->epoch += 1u;
    ctl->group_next = 0;
    ctl->pl_ticket = 0;
    if (begin_step) {
        ctl->tnext = ctl->tnext_acc;
        ctl->tnext_acc = ~0ull;
    }
}

__global__ void k_prepare(DevCtl *ctl, int begin_step) {
    gt_grid_ready();
    prepare_body(blockIdx.x, gridDim.x, ctl, begin_step);
}

__global__ void k_set_nactive(DevCtl *ctl, unsigned int n_active) { ctl->n_active = n_active; }

__global__ void k_mirror(const DevCtl *ctl, StepMirror *dst) {
    gt_grid_ready();
    volatile StepMirror *d = dst;
    d->tnext_acc = ctl->tnext_acc;
    d->n_active = ctl->n_active;
    d->err = ctl->err;
    __threadfence_system();
}

// Two particles per thread with 16-byte loads (n even, so that every array of the state,
// and the second and third coordinate arrays inside its block, start 16-byte aligned).
__device__ __forceinline__ void predict2_body(const unsigned bid, const unsigned nb, State s, long long n,
        const DevCtl *__restrict__ ctl, float4 *__restrict__ posm, int ahead) {
    const long long i = 2 * (bid * 256ll + threadIdx.x);
    if (i >= n) return;
    const long long T = (long long)(ahead ? ctl->tnext_acc : ctl->tnext);
    const int k = (int)((__double_as_longlong(ctl->dt_max) >> 52) & 0x7ff) - 1023 - ctl->levels_m1;
    const longlong2 t0 = *(const longlong2 *)&s.t0[i];
    const double dt0 = ctl->dt_max > 0.0 ? i2d_scaled(T - t0.x, k) : 0.0;
    const double dt1 = ctl->dt_max > 0.0 ? i2d_scaled(T - t0.y, k) : 0.0;
    const double2 rx = *(const double2 *)&s.rx[i], ry = *(const double2 *)&s.ry[i], rz = *(const double2 *)&s.rz[i];
    const double2 vx = *(const double2 *)&s.vx[i], vy = *(const double2 *)&s.vy[i], vz = *(const double2 *)&s.vz[i];
    const float2 m = *(const float2 *)&s.mass[i];
    posm[i] = make_float4(d2f(__fma_rn(dt0, vx.x, rx.x)), d2f(__fma_rn(dt0, vy.x, ry.x)),
                          d2f(__fma_rn(dt0, vz.x, rz.x)), m.x);
    posm[i + 1] = make_float4(d2f(__fma_rn(dt1, vx.y, rx.y)), d2f(__fma_rn(dt1, vy.y, ry.y)),
                              d2f(__fma_rn(dt1, vz.y, rz.y)), m.y);
}

__global__ __launch_bounds__(256) void k_predict2(State s, long long n, const DevCtl *__restrict__ ctl,
        float4 *__restrict__ posm, int ahead) {
    gt_grid_ready();
    predict2_body(blockIdx.x, gridDim.x, s, n, ctl, posm, ahead);
}

__device__ __forceinline__ void predict_body(const unsigned bid, const unsigned nb, State s, long long n,
        const DevCtl *__restrict__ ctl, float4 *__restrict__ posm, int ahead) {
    const long long i = bid * 256ll + threadIdx.x;
    if (i >= n) return;
    const long long T = (long long)(ahead ? ctl->tnext_acc : ctl->tnext);
    // dt = (T - t0) dt_min with dt_min = dt_max 2^-(L-1) a power of two: exact, so it is
    // built from the bits; only the three fused multiply-adds run on the FP64 pipe
    const int k = (int)((__double_as_longlong(ctl->dt_max) >> 52) & 0x7ff) - 1023 - ctl->levels_m1;
    const double dt = ctl->dt_max > 0.0 ? i2d_scaled(T - s.t0[i], k) : 0.0;
    const float x = d2f(__fma_rn(dt, s.vx[i], s.rx[i]));
    const float y = d2f(__fma_rn(dt, s.vy[i], s.ry[i]));
    const float z = d2f(__fma_rn(dt, s.vz[i], s.rz[i]));
    posm[i] = make_float4(x, y, z, s.mass[i]);
}

__global__ __launch_bounds__(256) void k_predict(State s, long long n, const DevCtl *__restrict__ ctl,
        float4 *__restrict__ posm, int ahead) {
    gt_grid_ready();
    predict_body(blockIdx.x, gridDim.x, s, n, ctl, posm, ahead);
}

__global__ __launch_bounds__(256) void k_load(State s, long long n, float4 *__restrict__ posm) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n) return;
    posm[i] = make_float4(d2f(s.rx[i]), d2f(s.ry[i]), d2f(s.rz[i]), s.mass[i]);
    s.id[i] = (uint32_t)i;
    s.t0[i] = 0;
    s.level[i] = 0;
    s.aold[i] = 0.0f;
    s.acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// The same from a caller's device arrays: one pass of 52 B read and 109 B written per particle (through the scratch
// copies and k_deinterleave3 it was five passes, 201 B read and 205 B written).
__global__ __launch_bounds__(256) void k_load_from(State s, long long n, const double *__restrict__ pos,
                                                   const double *__restrict__ vel, const float *__restrict__ mass,
                                                   float4 *__restrict__ posm) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n) return;
    const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
    const float m = mass[i];
    s.rx[i] = x;
    s.ry[i] = y;
    s.rz[i] = z;
    s.vx[i] = vel[3 * i];
    s.vy[i] = vel[3 * i + 1];
    s.vz[i] = vel[3 * i + 2];
    s.mass[i] = m;
    posm[i] = make_float4(d2f(x), d2f(y), d2f(z), m);
    s.id[i] = (uint32_t)i;
    s.t0[i] = 0;
    s.level[i] = 0;
    s.aold[i] = 0.0f;
    s.acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

__device__ __forceinline__ void permute_body(const unsigned bid, const unsigned nb, State src, State dst,
        const float4 *__restrict__ pin, float4 *__restrict__ pout, const uint32_t *__restrict__ perm, long long n) {
    const long long i = bid * 256ll + threadIdx.x;
    if (i >= n) return;
    const uint32_t k = perm[i];
    dst.rx[i] = src.rx[k];
    dst.ry[i] = src.ry[k];
    dst.rz[i] = src.rz[k];
    dst.vx[i] = src.vx[k];
    dst.vy[i] = src.vy[k];
    dst.vz[i] = src.vz[k];
    dst.t0[i] = src.t0[k];
    dst.level[i] = src.level[k];
    dst.aold[i] = src.aold[k];
    dst.acc[i] = src.acc[k];
    dst.id[i] = src.id[k];
    const float4 p = pin[k];
    dst.mass[i] = p.w;  // the position's fourth word is the mass
    pout[i] = p;
}

__global__ __launch_bounds__(256) void k_permute(State src, State dst, const float4 *__restrict__ pin,
        float4 *__restrict__ pout, const uint32_t *__restrict__ perm, long long n) {
    gt_grid_ready();
    permute_body(blockIdx.x, gridDim.x, src, dst, pin, pout, perm, n);
}

// copy the permuted state back, so that buffer 0 always holds the current state
__device__ __forceinline__ void copy_state_body(const unsigned bid, const unsigned nb, State src, State dst,
        const float4 *__restrict__ pin, float4 *__restrict__ pout, long long n) {
    const long long i = bid * 256ll + threadIdx.x;
    if (i >= n) return;
    dst.rx[i] = src.rx[i];
    dst.ry[i] = src.ry[i];
    dst.rz[i] = src.rz[i];
    dst.vx[i] = src.vx[i];
    dst.vy[i] = src.vy[i];
    dst.vz[i] = src.vz[i];
    dst.t0[i] = src.t0[i];
    dst.level[i] = src.level[i];
    dst.aold[i] = src.aold[i];
    dst.acc[i] = src.acc[i];
    dst.id[i] = src.id[i];
    dst.mass[i] = src.mass[i];
    if (pin) pout[i] = pin[i];
}

__global__ __launch_bounds__(256) void k_copy_state(State src, State dst, const float4 *__restrict__ pin,
        float4 *__restrict__ pout, long long n) {
    gt_grid_ready();
    copy_state_body(blockIdx.x, gridDim.x, src, dst, pin, pout, n);
}

// n x 3 row-major <-> three arrays
__global__ __launch_bounds__(256) void k_deinterleave3(const double *__restrict__ in, long long n,
                                                       double *__restrict__ x, double *__restrict__ y,
                                                       double *__restrict__ z) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n) return;
    x[i] = in[3 * i];
    y[i] = in[3 * i + 1];
    z[i] = in[3 * i + 2];
}

__global__ __launch_bounds__(256) void k_interleave3(const double *__restrict__ x, const double *__restrict__ y,
                                                     const double *__restrict__ z, long long n,
                                                     double *__restrict__ out) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n) return;
    out[3 * i] = x[i];
    out[3 * i + 1] = y[i];
    out[3 * i + 2] = z[i];
}

// state out in the caller's particle order: row id[i] of pos/vel (n x 3) <- slot i
__global__ __launch_bounds__(256) void k_state_out(State t, long long n, double *__restrict__ pos,
                                                   double *__restrict__ vel) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n) return;
    const long long j = t.id[i];
    if (pos) {
        pos[3 * j] = t.rx[i];
        pos[3 * j + 1] = t.ry[i];
        pos[3 * j + 2] = t.rz[i];
    }
    if (vel) {
        vel[3 * j] = t.vx[i];
        vel[3 * j + 1] = t.vy[i];
        vel[3 * j + 2] = t.vz[i];
    }
}

__global__ __launch_bounds__(256) void k_gather_f(const float *__restrict__ in, const uint32_t *__restrict__ id,
                                                  long long n, float *__restrict__ out) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i < n) out[i] = in[id[i]];
}

// bit active[k] set for a caller's list; a list that is not strictly increasing or
// holds an index >= n latches GT_EINVAL (the cell grouping needs key order)
__global__ __launch_bounds__(256) void k_scatter_flags(const uint32_t *__restrict__ active, long long na,
                                                       long long n, uint32_t *__restrict__ bits, DevCtl *ctl) {
    gt_grid_ready();
    const long long k = blockIdx.x * 256ll + threadIdx.x;
    const uint32_t i = k < na ? active[k] : 0u;
    const bool bad = k < na && ((long long)i >= n || (k > 0 && active[k - 1] >= i)), on = k < na && !bad;
    if (bad) gt_set_error(ctl, GT_EINVAL, GTK_ACTIVE);
    // one atomic per word of the warp's entries (a tenth of 10^6 active: 2.9 us, one per entry 6.1 us)
    const unsigned int peers = __match_any_sync(0xffffffffu, on ? i >> 5 : ~0u);
    const uint32_t mask = __reduce_or_sync(peers, on ? 1u << (i & 31u) : 0u);
    if (on && __ffs(peers) - 1 == lane_id()) atomicOr(&bits[i >> 5], mask);
}

constexpr int AT = 256, AIPT = 16, ATILE = AT * AIPT;

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, v, o);
        v = t < v ? t : v;
    }
    return v;
}

// Order-preserving compaction of the particles whose step ends at the block time.  Writes their indices to out, the
// rank words (rank[n / 32] too), the count to ctl->n_active, and folds the others' step ends into the next block time.
__device__ __forceinline__ void compact_body(const unsigned bid, const unsigned nb, long long n,
        const long long *__restrict__ t0, const uint8_t *__restrict__ level, int L, DevCtl *ctl, int ticket,
        uint32_t tag_slot, uint32_t *__restrict__ out, uint2 *__restrict__ rank, unsigned long long *status) {
    __shared__ uint32_t tmp[AT / 32 + 1];
    __shared__ uint32_t tile_sh, excl_sh;
    const unsigned long long T = ctl->tnext;
    const uint32_t tag = ctl->epoch * 32u + tag_slot;
    const uint32_t ntiles = (uint32_t)((n + ATILE - 1) / ATILE);
    unsigned long long tmin = ~0ull;
    if (n == 0) {
        if (bid == 0 && threadIdx.x == 0) {
            ctl->n_active = 0;
            rank[0] = make_uint2(0u, 0u);
        }
        return;
    }
    for (;;) {
        if (threadIdx.x == 0) tile_sh = atomicAdd(&ctl->tile_ticket[ticket], 1u);
        __syncthreads();
        const uint32_t tile = tile_sh;
        __syncthreads();
        if (tile >= ntiles) break;
        // warp w owns items [wbase, wbase + 32 AIPT); row q is items wbase + 32 q + lane, so
        // every load and store of a row is one coalesced access, and rows then lanes
        // visit the items in index order (the compaction keeps it)
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const long long wbase = (long long)tile * ATILE + (long long)w * (32 * AIPT);
        unsigned int bal[AIPT];
        uint32_t wsel = 0;
#pragma unroll
        for (int q = 0; q < AIPT; q++) {
            const long long i = wbase + 32 * q + lane;
            bool on = false;
            if (i < n) {
                const unsigned long long tend = (unsigned long long)t0[i] + (1ull << (L - 1 - (int)level[i]));
                on = tend == T;
                if (!on) tmin = tend < tmin ? tend : tmin;
            }
            bal[q] = __ballot_sync(0xffffffffu, on);
            wsel += (uint32_t)__popc(bal[q]);
        }
        // the warps' counts in order: one value per warp into the block scan
        uint32_t total;
        const uint32_t wexcl = block_excl_scan<AT>(lane == 31 ? wsel : 0u, &total, tmp);
        const uint32_t wstart = __shfl_sync(0xffffffffu, wexcl, 31);
        if (threadIdx.x < 32) {
            const uint32_t e = lookback_warp(status, tile, total, tag, ctl, GTK_ACTIVE);
            if (threadIdx.x == 0) excl_sh = e;
        }
        __syncthreads();
        uint32_t pos = excl_sh + wstart;
        const unsigned int lt = lanemask_lt();
        uint2 mine = make_uint2(0u, 0u);  // lane q keeps row q's rank word
#pragma unroll
        for (int q = 0; q < AIPT; q++) {
            const long long i = wbase + 32 * q + lane;
            if (lane == q) mine = make_uint2(bal[q], pos);
            if ((bal[q] >> lane) & 1u) out[pos + (uint32_t)__popc(bal[q] & lt)] = (uint32_t)i;
            pos += (uint32_t)__popc(bal[q]);
        }
        if (lane < AIPT && wbase + 32 * lane < n) rank[(wbase >> 5) + lane] = mine;
        if (tile == ntiles - 1 && threadIdx.x == AT - 1) {
            ctl->n_active = excl_sh + total;
            if (n % 32 == 0) rank[n >> 5] = make_uint2(0u, excl_sh + total);
        }
    }
    tmin = warp_min_u64(tmin);
    if (lane_id() == 0 && tmin != ~0ull) atomicMin(&ctl->tnext_acc, tmin);
}

__global__ __launch_bounds__(AT) void k_compact(long long n, const long long *__restrict__ t0,
        const uint8_t *__restrict__ level, int L, DevCtl *ctl, int ticket, uint32_t tag_slot,
        uint32_t *__restrict__ out, uint2 *__restrict__ rank, unsigned long long *status) {
    gt_grid_ready();
    compact_body(blockIdx.x, gridDim.x, n, t0, level, L, ctl, ticket, tag_slot, out, rank, status);
}

// Order-preserving compaction of the bits of [0, n) (n from n_dev if given), which are cleared on the way (masks
// start at zero, so that no launch has to clear them).  Writes the indices to out, the rank words if rank != null
// (rank[n / 32] too), and the count to *count_out.  A lane takes a word of 32 items, 8192 items to a
// tile: at 2^24 items the masks are 2 MB, in L2, where a byte each was 16 MB to clear, write and read.  100 000 of 2^24
// active, the whole walk: 282 us with bytes, 236 with four words per lane (too few blocks), 225.
constexpr int BTILE = AT;  // words per tile, a word per lane

__device__ __forceinline__ void compact_bits_body(const unsigned bid, const unsigned nb, long long n_host,
        const unsigned int *n_dev, uint32_t *__restrict__ bits, DevCtl *ctl, int ticket, uint32_t tag_slot,
        uint32_t *__restrict__ out, uint2 *__restrict__ rank, unsigned int *count_out, unsigned long long *status) {
    __shared__ uint32_t tmp[AT / 32 + 1];
    __shared__ uint32_t tile_sh, excl_sh;
    const long long n = n_dev ? (long long)*n_dev : n_host;
    const uint32_t tag = ctl->epoch * 32u + tag_slot;
    const long long nwords = (n + 31) / 32;
    const uint32_t ntiles = (uint32_t)((nwords + BTILE - 1) / BTILE);
    if (n == 0) {
        if (bid == 0 && threadIdx.x == 0) {
            *count_out = 0;
            if (rank) rank[0] = make_uint2(0u, 0u);
        }
        return;
    }
    for (;;) {
        if (threadIdx.x == 0) tile_sh = atomicAdd(&ctl->tile_ticket[ticket], 1u);
        __syncthreads();
        const uint32_t tile = tile_sh;
        __syncthreads();
        if (tile >= ntiles) break;
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const long long wbase = (long long)tile * BTILE + 32 * w, i = wbase + lane;  // the warp's first word, the lane's
        const uint32_t word = i < nwords ? bits[i] : 0u;
        if (word) bits[i] = 0u;
        const uint32_t incl = warp_incl_scan((uint32_t)__popc(word));
        uint32_t total;
        const uint32_t wexcl = block_excl_scan<AT>(lane == 31 ? incl : 0u, &total, tmp);
        const uint32_t wstart = __shfl_sync(0xffffffffu, wexcl, 31);
        if (threadIdx.x < 32) {
            const uint32_t e = lookback_warp(status, tile, total, tag, ctl, GTK_ACTIVE);
            if (threadIdx.x == 0) excl_sh = e;
        }
        __syncthreads();
        const uint32_t start = excl_sh + wstart + incl - (uint32_t)__popc(word);
        if (rank && i < nwords) rank[i] = make_uint2(word, start);
        const unsigned int lt = lanemask_lt();
        for (unsigned int m = __ballot_sync(0xffffffffu, word != 0u); m; m &= m - 1) {  // a word at a time
            const int src = __ffs(m) - 1;
            const uint32_t b = __shfl_sync(0xffffffffu, word, src), at = __shfl_sync(0xffffffffu, start, src);
            if ((b >> lane) & 1u) out[at + (uint32_t)__popc(b & lt)] = (uint32_t)(32 * (wbase + src) + lane);
        }
        if (tile == ntiles - 1 && threadIdx.x == AT - 1) {
            *count_out = excl_sh + total;
            if (rank && n % 32 == 0) rank[n >> 5] = make_uint2(0u, excl_sh + total);
        }
    }
}

__global__ __launch_bounds__(AT) void k_compact_bits(long long n_host, const unsigned int *n_dev,
        uint32_t *__restrict__ bits, DevCtl *ctl, int ticket, uint32_t tag_slot, uint32_t *__restrict__ out,
        uint2 *__restrict__ rank, unsigned int *count_out, unsigned long long *status) {
    gt_grid_ready();
    compact_bits_body(blockIdx.x, gridDim.x, n_host, n_dev, bits, ctl, ticket, tag_slot, out, rank, count_out, status);
}

// The number of actives below i.
__device__ __forceinline__ uint32_t rank_at(const uint2 *__restrict__ rank, uint32_t i) {
    const uint2 r = rank[i >> 5];
    return r.y + (uint32_t)__popc(r.x & ((1u << (i & 31u)) - 1u));
}

// Mark the first active position of every group (Sec. 2.4 reading: groups never
// straddle two tree cells).  A cell qualifies when it holds at most gmax actives and is
// a leaf or no wider than r_crit (b_J <= r_crit; r_crit <= 0: no radius limit).  Counts
// and radii only shrink from a cell to its children, so a group cell is a qualifying
// cell whose parent does not qualify (or the root), or a leaf under no qualifying cell;
// its actives are cut into runs of gmax.
// ALL: every particle is active (the number below i is i).
template <bool ALL>
__device__ __forceinline__ bool group_cell_ok(const Nodes &nd, const uint2 *R, uint32_t c, int gmax, float r_crit) {
    const uint32_t f = nd.first[c], k = nd.count[c];
    if ((ALL ? k : rank_at(R, f + k) - rank_at(R, f)) > (uint32_t)gmax) return false;
    return nd.child[c] < 0 || r_crit <= 0.0f || nd.walk[c].x <= r_crit;
}

template <bool ALL>
__device__ __forceinline__ void group_cells_body(const unsigned bid, const unsigned nb, Nodes nd, long long n,
        long long cap, const uint2 *__restrict__ R, int gmax, float r_crit, uint32_t *__restrict__ marks, DevCtl *ctl) {
    long long nn = ctl->level_start[GT_TREE_LEVELS];
    if (nn > cap) nn = cap;
    if (ALL && bid == 0 && threadIdx.x == 0) ctl->n_active = (unsigned int)n;
    for (long long c = bid * 256ll + threadIdx.x; c < nn; c += (long long)nb * 256) {
        const uint32_t f = nd.first[c], k = nd.count[c];
        const uint32_t a0 = ALL ? f : rank_at(R, f), A = ALL ? k : rank_at(R, f + k) - a0;
        if (A == 0) continue;
        const int32_t p = nd.parent[c];
        if (p >= 0 && group_cell_ok<ALL>(nd, R, (uint32_t)p, gmax, r_crit)) continue;  // inside a group cell
        if (nd.child[c] >= 0 && !group_cell_ok<ALL>(nd, R, (uint32_t)c, gmax, r_crit)) continue;  // children decide
        for (uint32_t s = a0; s < a0 + A; s += (uint32_t)gmax) atomicOr(&marks[s >> 5], 1u << (s & 31u));
    }
}

template <bool ALL>
__global__ __launch_bounds__(256) void k_group_cells(Nodes nd, long long n, long long cap,
        const uint2 *__restrict__ R, int gmax, float r_crit, uint32_t *__restrict__ marks, DevCtl *ctl) {
    gt_grid_ready();
    group_cells_body<ALL>(blockIdx.x, gridDim.x, nd, n, cap, R, gmax, r_crit, marks, ctl);
}

// a batch member's accelerations and ids to the caller
__global__ __launch_bounds__(256) void k_acc_out(const float4 *__restrict__ acc, const uint32_t *__restrict__ id,
                                                 long long n, float4 *__restrict__ acc_out,
                                                 uint32_t *__restrict__ id_out) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n) return;
    if (acc_out) acc_out[i] = acc[i];
    if (id_out) id_out[i] = id[i];
}

__global__ __launch_bounds__(256) void k_iota(uint32_t *__restrict__ out, long long n) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i < n) out[i] = (uint32_t)i;
}

__device__ __forceinline__ double a2_of(float4 a) {
    const double ax = f2d(a.x), ay = f2d(a.y), az = f2d(a.z);  // exact widenings, integer pipe
    // the squares are exact in FP64, so the fused forms round only at the additions
    return __fma_rn(az, az, __fma_rn(ay, ay, __dmul_rn(ax, ax)));
}

__device__ __forceinline__ long long floordiv4(long long d) { return d >= 0 ? d / 4 : -((-d + 3) / 4); }

__device__ __forceinline__ int level_from_a2(double a2, double c2, int M, int L) {
    if (!(a2 > 0.0) || !isfinite(a2)) return 0;
    int ea, ec;
    const double fa = frexp(a2, &ea), fc = frexp(c2, &ec);
    // level k qualifies iff 4k > D, or 4k == D and fa <= fc, with D = ea + 4M - ec
    const long long D = (long long)ea + 4ll * M - ec;
    const long long q = floordiv4(D);
    long long k = (4 * q == D && fa <= fc) ? q : q + 1;
    k = k < 0 ? 0 : k;
    k = k > L - 1 ? L - 1 : k;
    return (int)k;
}

__device__ __forceinline__ void correct_body(const unsigned bid, const unsigned nb, State s,
        const uint32_t *__restrict__ active, const float4 *__restrict__ acc, DevCtl *ctl, long long n, int L,
        double c2) {
    const uint32_t na = ctl->n_active;
    const long long T = (long long)ctl->tnext;
    const int M = ctl->M;  // dt_max = 2^M
    // the step's powers of two and the exact widenings are built on the integer pipe (the
    // FP64 pipe of this GPU is narrow); only the kicks, drifts and |a|^2 use it
    auto p2 = [](int e) {  // 2^e
        return (e > -1023 && e < 1024) ? __longlong_as_double((long long)(e + 1023) << 52) : ldexp(1.0, e);
    };
    unsigned long long tmin = ~0ull;
    for (uint32_t k = bid * 256u + threadIdx.x; k < na; k += nb * 256u) {
        const uint32_t i = active[k];
        if ((long long)i >= n) {  // an index outside the system: report it and skip
            gt_set_error(ctl, GT_EINVAL, GTK_CORRECT);
            continue;
        }
        const float4 a = acc[k];
        const int kold = s.level[i];
        const double hold = p2(M - kold - 1);                  // dt(kold) / 2
        const double dtp = i2d_scaled(T - s.t0[i], M - (L - 1));  // (T - t0) dt_min, exact
        const double ax = f2d(a.x), ay = f2d(a.y), az = f2d(a.z);
        const double vx0 = s.vx[i], vy0 = s.vy[i], vz0 = s.vz[i];
        s.rx[i] = __fma_rn(dtp, vx0, s.rx[i]);
        s.ry[i] = __fma_rn(dtp, vy0, s.ry[i]);
        s.rz[i] = __fma_rn(dtp, vz0, s.rz[i]);
        const double vx = __fma_rn(hold, ax, vx0);
        const double vy = __fma_rn(hold, ay, vy0);
        const double vz = __fma_rn(hold, az, vz0);
        const double a2 = a2_of(a);
        const int kc = level_from_a2(a2, c2, M, L);
        int knew = kold;
        if (kc > kold) {
            knew = kc;
        } else if (kc < kold) {
            const long long span = 1ll << (L - 1 - (kold - 1));
            if (T % span == 0) knew = kold - 1;
        }
        const double hnew = p2(M - knew - 1);
        s.vx[i] = __fma_rn(hnew, ax, vx);
        s.vy[i] = __fma_rn(hnew, ay, vy);
        s.vz[i] = __fma_rn(hnew, az, vz);
        s.level[i] = (uint8_t)knew;
        s.t0[i] = T;
        s.aold[i] = __fsqrt_rn(d2f(a2));
        s.acc[i] = a;
        const unsigned long long tend = (unsigned long long)T + (1ull << (L - 1 - knew));
        tmin = tend < tmin ? tend : tmin;
    }
    tmin = warp_min_u64(tmin);
    if (lane_id() == 0 && tmin != ~0ull) atomicMin(&ctl->tnext_acc, tmin);
}

__global__ __launch_bounds__(256) void k_correct(State s, const uint32_t *__restrict__ active,
        const float4 *__restrict__ acc, DevCtl *ctl, long long n, int L, double c2) {
    gt_grid_ready();
    correct_body(blockIdx.x, gridDim.x, s, active, acc, ctl, n, L, c2);
}

__device__ __forceinline__ void aold_body(const unsigned bid, const unsigned nb, const float4 *__restrict__ acc,
        long long n, float *__restrict__ aold) {
    const long long i = bid * 256ll + threadIdx.x;
    if (i < n) aold[i] = __fsqrt_rn(__double2float_rn(a2_of(acc[i])));
}

__global__ __launch_bounds__(256) void k_aold(const float4 *__restrict__ acc, long long n, float *__restrict__ aold) {
    gt_grid_ready();
    aold_body(blockIdx.x, gridDim.x, acc, n, aold);
}

// start, phase 1: the smallest positive A2 (bit pattern of a positive double)
__device__ __forceinline__ void min_a2_body(const unsigned bid, const unsigned nb, const float4 *__restrict__ acc,
        long long n, DevCtl *ctl) {
    unsigned long long best = ~0ull;
    for (long long i = bid * 256ll + threadIdx.x; i < n; i += (long long)nb * 256) {
        const double a2 = a2_of(acc[i]);
        if (!(a2 > 0.0) || !isfinite(a2)) continue;
        const unsigned long long b = (unsigned long long)__double_as_longlong(a2);
        best = b < best ? b : best;
    }
    best = warp_min_u64(best);
    if (lane_id() == 0 && best != ~0ull) atomicMin(&ctl->max_dt_bits, best);
}

__global__ __launch_bounds__(256) void k_min_a2(const float4 *__restrict__ acc, long long n, DevCtl *ctl) {
    gt_grid_ready();
    min_a2_body(blockIdx.x, gridDim.x, acc, n, ctl);
}

// start, phase 2: dt_max (the largest 2^M with 2^(4M) A2min <= c2), levels, t0 = 0,
// first half kick v^{1/2} = fma(dt/2, a, v)
__device__ __forceinline__ void init_levels_body(const unsigned bid, const unsigned nb, State s,
        const float4 *__restrict__ acc, long long n, int L, double c2, int M_given, int have_M, DevCtl *ctl) {
    int M = M_given;
    if (!have_M) {
        M = 0;
        if (ctl->max_dt_bits != ~0ull) {
            const double a2min = __longlong_as_double((long long)ctl->max_dt_bits);
            int ea, ec;
            const double fa = frexp(a2min, &ea), fc = frexp(c2, &ec);
            const long long D = (long long)ec - ea;  // M qualifies iff 4M < D, or 4M == D and fa <= fc
            const long long q = floordiv4(D);
            M = (int)(4 * q == D ? (fa <= fc ? q : q - 1) : q);
        }
    }
    const double dt_max = ldexp(1.0, M);
    if (bid == 0 && threadIdx.x == 0) {
        ctl->M = M;
        ctl->dt_max = dt_max;
        ctl->levels_m1 = L - 1;
    }
    unsigned long long tmin = ~0ull;
    for (long long i = bid * 256ll + threadIdx.x; i < n; i += (long long)nb * 256) {
        const float4 a = acc[i];
        const double a2 = a2_of(a);
        const int k = level_from_a2(a2, c2, M, L);
        const double h = 0.5 * ldexp(dt_max, -k);
        s.vx[i] = __fma_rn(h, (double)a.x, s.vx[i]);
        s.vy[i] = __fma_rn(h, (double)a.y, s.vy[i]);
        s.vz[i] = __fma_rn(h, (double)a.z, s.vz[i]);
        s.level[i] = (uint8_t)k;
        s.t0[i] = 0;
        s.aold[i] = __fsqrt_rn(__double2float_rn(a2));
        s.acc[i] = a;
        const unsigned long long tend = 1ull << (L - 1 - k);
        tmin = tend < tmin ? tend : tmin;
    }
    tmin = warp_min_u64(tmin);
    if (lane_id() == 0 && tmin != ~0ull) atomicMin(&ctl->tnext_acc, tmin);
}

__global__ __launch_bounds__(256) void k_init_levels(State s, const float4 *__restrict__ acc, long long n, int L,
        double c2, int M_given, int have_M, DevCtl *ctl) {
    gt_grid_ready();
    init_levels_body(blockIdx.x, gridDim.x, s, acc, n, L, c2, M_given, have_M, ctl);
}

// resume: scalars of the integration and the next block time over all particles
__global__ void k_set_clock(DevCtl *ctl, int M, int L, long long T) {
    gt_grid_ready();
    ctl->M = M;
    ctl->dt_max = ldexp(1.0, M);
    ctl->levels_m1 = L - 1;
    ctl->tnext = (unsigned long long)T;
    ctl->tnext_acc = ~0ull;
}

__global__ void k_set_tnext(DevCtl *ctl, long long T) { ctl->tnext = (unsigned long long)T; }

__global__ void k_set_u32(unsigned int *dst, unsigned int v) { *dst = v; }

__global__ __launch_bounds__(256) void k_tnext_all(const long long *__restrict__ t0,
                                                   const uint8_t *__restrict__ level, long long n, int L,
                                                   DevCtl *ctl) {
    gt_grid_ready();
    unsigned long long tmin = ~0ull;
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
        const unsigned long long tend = (unsigned long long)t0[i] + (1ull << (L - 1 - (int)level[i]));
        tmin = tend < tmin ? tend : tmin;
    }
    tmin = warp_min_u64(tmin);
    if (lane_id() == 0 && tmin != ~0ull) atomicMin(&ctl->tnext_acc, tmin);
}

__global__ __launch_bounds__(256) void k_gather_resume(const uint8_t *__restrict__ lv, const long long *__restrict__ t0,
                                                       const float *__restrict__ ao, const float4 *__restrict__ acc,
                                                       const uint32_t *__restrict__ id, long long n, State s) {
    gt_grid_ready();
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n) return;
    const uint32_t k = id[i];
    s.level[i] = lv[k];
    s.t0[i] = t0[k];
    s.aold[i] = ao[k];
    s.acc[i] = acc ? acc[k] : make_float4(0.f, 0.f, 0.f, 0.f);
}

__global__ void k_reset_start(DevCtl *ctl) {
    gt_grid_ready();
    ctl->max_dt_bits = ~0ull;
    ctl->tnext_acc = ~0ull;
    ctl->tnext = 0;
}

// ---- a table of systems ----
__global__ void kg_prepare(const GroupedSys *__restrict__ t) {  // a warp each
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    prepare_body(0, 1, s.ctl, (s.flags & GT_SYS_STEP) ? 1 : 0);
    if ((s.flags & GT_SYS_START) && threadIdx.x == 0) {
        s.ctl->max_dt_bits = ~0ull;
        s.ctl->tnext_acc = ~0ull;
        s.ctl->tnext = 0;
    }
}

__global__ __launch_bounds__(256) void kg_predict(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    if (!(s.flags & GT_SYS_STEP)) return;
    float4 *dst = (s.flags & GT_SYS_BUILD) ? s.posm_tmp : s.posm;
    // (a system's arrays start 256-byte aligned, so an even number of particles keeps the pairs aligned)
    if (s.n % 2 == 0) predict2_body(blockIdx.y, gridDim.y, s.st0, s.n, s.ctl, dst, 0);
    else predict_body(blockIdx.y, gridDim.y, s.st0, s.n, s.ctl, dst, 0);
}

__global__ __launch_bounds__(256) void kg_permute(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    if (!(s.flags & GT_SYS_BUILD)) return;
    const bool tmp = (s.flags & GT_SYS_PREDICTED) != 0;
    permute_body(blockIdx.y, gridDim.y, s.st0, s.st1, tmp ? s.posm_tmp : s.posm, tmp ? s.posm : s.posm_tmp, s.sb.val[0],
                 s.n);
}

__global__ __launch_bounds__(256) void kg_copy_state(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    if (!(s.flags & GT_SYS_BUILD)) return;
    const bool tmp = (s.flags & GT_SYS_PREDICTED) != 0;
    copy_state_body(blockIdx.y, gridDim.y, s.st1, s.st0, tmp ? nullptr : s.posm_tmp, tmp ? nullptr : s.posm, s.n);
}

__global__ __launch_bounds__(AT) void kg_compact(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, ATILE, nsm * 4);
    if (!(s.flags & GT_SYS_STEP) || blockIdx.y >= nb) return;
    compact_body(blockIdx.y, nb, s.n, s.st0.t0, s.st0.level, s.levels, s.ctl, GT_TREE_LEVELS, 30u, s.active, s.rank,
                 s.status);
}

__global__ __launch_bounds__(256) void kg_group_cells(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 256, nsm * 8);
    if (blockIdx.y >= nb) return;
    if (!s.cells) {
        if (!(s.flags & GT_SYS_STEP) && blockIdx.y == 0 && threadIdx.x == 0) s.ctl->n_active = (unsigned int)s.n;
    } else if (s.flags & GT_SYS_STEP) {
        group_cells_body<false>(blockIdx.y, nb, s.nd, s.n, s.cap, s.rank, s.gmax, s.r_crit, s.marks, s.ctl);
    } else {
        group_cells_body<true>(blockIdx.y, nb, s.nd, s.n, s.cap, nullptr, s.gmax, s.r_crit, s.marks, s.ctl);
    }
}

__global__ __launch_bounds__(AT) void kg_groups(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 32 * BTILE, nsm * 4);
    if (!s.cells || blockIdx.y >= nb) return;
    compact_bits_body(blockIdx.y, nb, 0, &s.ctl->n_active, s.marks, s.ctl, GT_TREE_LEVELS + 1, 31u, s.gstart, nullptr,
                      &s.ctl->n_groups, s.status);
}

__global__ __launch_bounds__(256) void kg_aold(const GroupedSys *__restrict__ t) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    if (s.flags & GT_SYS_START) aold_body(blockIdx.y, gridDim.y, s.acc, s.n, s.st0.aold);
}

__global__ __launch_bounds__(256) void kg_min_a2(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 256, nsm * 4);
    if ((s.flags & GT_SYS_START) && !s.have_M && blockIdx.y < nb) min_a2_body(blockIdx.y, nb, s.acc, s.n, s.ctl);
}

__global__ __launch_bounds__(256) void kg_init_levels(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 256, nsm * 8);
    if ((s.flags & GT_SYS_START) && blockIdx.y < nb)
        init_levels_body(blockIdx.y, nb, s.st0, s.acc, s.n, s.levels, s.c2, s.M, s.have_M, s.ctl);
}

__global__ __launch_bounds__(256) void kg_correct(const GroupedSys *__restrict__ t, int nsm) {
    gt_grid_ready();
    const GroupedSys &s = t[blockIdx.x];
    const unsigned nb = gt_grid(s.n, 256, nsm * 8);
    if ((s.flags & GT_SYS_STEP) && blockIdx.y < nb)
        correct_body(blockIdx.y, nb, s.st0, s.active, s.acc, s.ctl, s.n, s.levels, s.c2);
}

inline unsigned nblk(long long n) { return (unsigned)((n + 255) / 256); }

}  // namespace

void gt_launch_prepare(DevCtl *ctl, int begin_step, cudaStream_t st) {
    { k_prepare<<<1, 32, 0, st>>>(ctl, begin_step); gt_note_launches(1); }
}

void gt_launch_set_nactive(DevCtl *ctl, unsigned int n_active, cudaStream_t st) {
    { k_set_nactive<<<1, 1, 0, st>>>(ctl, n_active); gt_note_launches(1); }
}

void gt_launch_predict(const State &s, int64_t n, const DevCtl *ctl, float4 *posm, cudaStream_t st, bool ahead) {
    if (n <= 0) return;
    const bool aligned = ((uintptr_t)s.rx | (uintptr_t)s.ry | (uintptr_t)s.rz | (uintptr_t)s.vx | (uintptr_t)s.vy |
                          (uintptr_t)s.vz | (uintptr_t)s.t0 | (uintptr_t)s.mass) % 16 == 0;
    if (n % 2 == 0 && aligned) gt_launch(k_predict2, nblk(n / 2), 256, 0, st, s, n, ctl, posm, ahead ? 1 : 0);
    else gt_launch(k_predict, nblk(n), 256, 0, st, s, n, ctl, posm, ahead ? 1 : 0);
    gt_note_launches(1);
}

void gt_launch_mirror(const DevCtl *ctl, StepMirror *dst, cudaStream_t st) {
    { k_mirror<<<1, 1, 0, st>>>(ctl, dst); gt_note_launches(1); }
}

void gt_launch_load(const State &s, float4 *posm, int64_t n, cudaStream_t st) {
    if (n > 0) { k_load<<<nblk(n), 256, 0, st>>>(s, n, posm); gt_note_launches(1); }
}

void gt_launch_load_from(const State &s, float4 *posm, int64_t n, const double *pos, const double *vel,
                         const float *mass, cudaStream_t st) {
    if (n > 0) { k_load_from<<<nblk(n), 256, 0, st>>>(s, n, pos, vel, mass, posm); gt_note_launches(1); }
}

void gt_launch_permute(const State &src, const State &dst, const float4 *posm_in, float4 *posm_out,
                       const uint32_t *perm, int64_t n, cudaStream_t st) {
    if (n > 0) { gt_launch(k_permute, nblk(n), 256, 0, st, src, dst, posm_in, posm_out, perm, n); gt_note_launches(1); }
}

void gt_launch_copy_state(const State &src, const State &dst, const float4 *posm_in, float4 *posm_out,
                          int64_t n, cudaStream_t st) {
    if (n > 0) { gt_launch(k_copy_state, nblk(n), 256, 0, st, src, dst, posm_in, posm_out, n); gt_note_launches(1); }
}

void gt_launch_deinterleave3(const double *in, int64_t n, double *x, double *y, double *z,
                             cudaStream_t st) {
    if (n > 0) { k_deinterleave3<<<nblk(n), 256, 0, st>>>(in, n, x, y, z); gt_note_launches(1); }
}

void gt_launch_interleave3(const double *x, const double *y, const double *z, int64_t n, double *out,
                           cudaStream_t st) {
    if (n > 0) { k_interleave3<<<nblk(n), 256, 0, st>>>(x, y, z, n, out); gt_note_launches(1); }
}

void gt_launch_state_out(const State &t, int64_t n, double *pos, double *vel, cudaStream_t st) {
    if (n > 0) { k_state_out<<<nblk(n), 256, 0, st>>>(t, n, pos, vel); gt_note_launches(1); }
}

void gt_launch_gather_f(const float *in, const uint32_t *id, int64_t n, float *out, cudaStream_t st) {
    if (n > 0) { k_gather_f<<<nblk(n), 256, 0, st>>>(in, id, n, out); gt_note_launches(1); }
}

void gt_launch_active(const State &s, int64_t n, int L, DevCtl *ctl, uint32_t *active, uint2 *rank,
                      unsigned long long *status, int nsm, cudaStream_t st) {
    { gt_launch(k_compact, gt_grid(n, ATILE, nsm * 4), AT, 0, st, n, s.t0, s.level, L, ctl, GT_TREE_LEVELS, 30u,
                active, rank, status);
      gt_note_launches(1); }
}

void gt_launch_active_from_list(const uint32_t *list, int64_t n_list, int64_t n, uint32_t *flags, DevCtl *ctl,
                                uint32_t *active, uint2 *rank, unsigned long long *status, int nsm, cudaStream_t st) {
    if (n_list > 0) { k_scatter_flags<<<nblk(n_list), 256, 0, st>>>(list, n_list, n, flags, ctl); gt_note_launches(1); }
    { gt_launch(k_compact_bits, gt_grid(n, 32 * BTILE, nsm * 4), AT, 0, st, n, nullptr, flags, ctl, GT_TREE_LEVELS,
                30u, active, rank, &ctl->n_active, status);
      gt_note_launches(1); }
}

void gt_launch_acc_out(const float4 *acc, const uint32_t *id, int64_t n, float4 *acc_out, uint32_t *id_out,
                       cudaStream_t st) {
    if (n > 0) { k_acc_out<<<nblk(n), 256, 0, st>>>(acc, id, n, acc_out, id_out); gt_note_launches(1); }
}

void gt_launch_iota(uint32_t *out, int64_t n, cudaStream_t st) {
    if (n > 0) { k_iota<<<nblk(n), 256, 0, st>>>(out, n); gt_note_launches(1); }
}

void gt_launch_groups(Nodes nd, int64_t cap, const uint2 *rank, int gmax, float r_crit, int64_t n, uint32_t *marks,
                      DevCtl *ctl, uint32_t *gstart, unsigned long long *status, int nsm, cudaStream_t st) {
    const unsigned grid = gt_grid(n, 256, nsm * 8);
    if (rank) gt_launch(k_group_cells<false>, grid, 256, 0, st, nd, n, cap, rank, gmax, r_crit, marks, ctl);
    else gt_launch(k_group_cells<true>, grid, 256, 0, st, nd, n, cap, rank, gmax, r_crit, marks, ctl);
    gt_launch(k_compact_bits, gt_grid(n, 32 * BTILE, nsm * 4), AT, 0, st, 0, &ctl->n_active, marks, ctl,
              GT_TREE_LEVELS + 1, 31u, gstart, nullptr, &ctl->n_groups, status);
    gt_note_launches(2);
}

void gt_launch_correct(const State &s, const uint32_t *active, const float4 *acc, DevCtl *ctl,
                       int64_t n, int L, double c2, int nsm, cudaStream_t st) {
    if (n > 0) { k_correct<<<gt_grid(n, 256, nsm * 8), 256, 0, st>>>(s, active, acc, ctl, n, L, c2); gt_note_launches(1); }
}

void gt_launch_aold(const float4 *acc, int64_t n, float *aold, cudaStream_t st) {
    if (n > 0) { k_aold<<<nblk(n), 256, 0, st>>>(acc, n, aold); gt_note_launches(1); }
}

void gt_launch_set_clock(DevCtl *ctl, int M, int L, long long T, cudaStream_t st) {
    { k_set_clock<<<1, 1, 0, st>>>(ctl, M, L, T); gt_note_launches(1); }
}

void gt_launch_set_tnext(DevCtl *ctl, long long T, cudaStream_t st) {
    { k_set_tnext<<<1, 1, 0, st>>>(ctl, T); gt_note_launches(1); }
}

void gt_launch_set_u32(unsigned int *dst, unsigned int v, cudaStream_t st) {
    { k_set_u32<<<1, 1, 0, st>>>(dst, v); gt_note_launches(1); }
}

void gt_launch_tnext_all(const State &s, int64_t n, int L, DevCtl *ctl, int nsm, cudaStream_t st) {
    if (n > 0) { k_tnext_all<<<gt_grid(n, 256, nsm * 4), 256, 0, st>>>(s.t0, s.level, n, L, ctl); gt_note_launches(1); }
}

void gt_launch_gather_resume(const uint8_t *lv, const long long *t0, const float *ao, const float4 *acc,
                             const State &s, int64_t n, cudaStream_t st) {
    if (n > 0) { k_gather_resume<<<nblk(n), 256, 0, st>>>(lv, t0, ao, acc, s.id, n, s); gt_note_launches(1); }
}

void gt_launch_init_levels(const State &s, const float4 *acc, int64_t n, int L, double c2, int M_given,
                           int have_M, DevCtl *ctl, int nsm, cudaStream_t st) {
    { k_reset_start<<<1, 1, 0, st>>>(ctl); gt_note_launches(1); }
    if (!have_M && n > 0) { gt_launch(k_min_a2, gt_grid(n, 256, nsm * 4), 256, 0, st, acc, n, ctl); gt_note_launches(1); }
    { gt_launch(k_init_levels, gt_grid(n, 256, nsm * 8), 256, 0, st, s, acc, n, L, c2, M_given, have_M, ctl); gt_note_launches(1); }
}

// ---- a table of systems ----
void gt_grouped_prepare(const GroupedSys *t, const GroupedPlan &p, int, cudaStream_t st) {
    kg_prepare<<<p.count, 32, 0, st>>>(t);
    gt_note_launches(1);
}

void gt_grouped_predict(const GroupedSys *t, const GroupedPlan &p, int, cudaStream_t st) {
    if (p.n_step <= 0) return;
    gt_launch(kg_predict, dim3(p.count, nblk(p.n_step)), 256, 0, st, t);
    gt_note_launches(1);
}

void gt_grouped_gather(const GroupedSys *t, const GroupedPlan &p, int, cudaStream_t st) {
    if (p.n_build <= 0) return;
    gt_launch(kg_permute, dim3(p.count, nblk(p.n_build)), 256, 0, st, t);
    gt_launch(kg_copy_state, dim3(p.count, nblk(p.n_build)), 256, 0, st, t);
    gt_note_launches(2);
}

void gt_grouped_groups(const GroupedSys *t, const GroupedPlan &p, int nsm, cudaStream_t st) {
    if (p.n_step > 0) {
        gt_launch(kg_compact, dim3(p.count, gt_grid(p.n_step, ATILE, nsm * 4)), AT, 0, st, t, nsm);
        gt_note_launches(1);
    }
    gt_launch(kg_group_cells, dim3(p.count, gt_grid(p.n_all, 256, nsm * 8)), 256, 0, st, t, nsm);
    gt_launch(kg_groups, dim3(p.count, gt_grid(p.n_all, 32 * BTILE, nsm * 4)), AT, 0, st, t, nsm);
    gt_note_launches(2);
}

void gt_grouped_aold(const GroupedSys *t, const GroupedPlan &p, int, cudaStream_t st) {
    if (p.n_start <= 0) return;
    kg_aold<<<dim3(p.count, nblk(p.n_start)), 256, 0, st>>>(t);
    gt_note_launches(1);
}

void gt_grouped_correct(const GroupedSys *t, const GroupedPlan &p, int nsm, cudaStream_t st) {
    if (p.n_start > 0) {
        kg_min_a2<<<dim3(p.count, gt_grid(p.n_start, 256, nsm * 4)), 256, 0, st>>>(t, nsm);
        gt_launch(kg_init_levels, dim3(p.count, gt_grid(p.n_start, 256, nsm * 8)), 256, 0, st, t, nsm);
        gt_note_launches(2);
    }
    if (p.n_step > 0) {
        kg_correct<<<dim3(p.count, gt_grid(p.n_step, 256, nsm * 8)), 256, 0, st>>>(t, nsm);
        gt_note_launches(1);
    }
}
