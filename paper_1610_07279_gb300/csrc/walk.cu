// Step A7: the tree walk for groups of active i-particles (Sec. 2.3) with the
// ij-parallelisation of Sec. 2.5.
//
// One warp walks one group at a time (a persistent grid; groups are taken from an
// atomic counter, so slow groups do not hold a fixed share of the GPU).  A group is a
// range of the active list: the actives of one tree cell (Sec. 2.4 reading) or a run
// of group_max.  Per group:
//   * S lanes per member (Sec. 2.5): fixed, or 32 / (members rounded up to a power of
//     two) so that small groups still fill the warp; the members above 32 share the lanes
//     a second time in the same way;
//   * pseudo i-particle: the sphere about the centre of the members' bounding box
//     (Appendix B, "GEO"), the FP32 radius widened by (1 + 2^-20); |a_old| of the
//     group is the smallest of its members';
//   * breadth-first traversal: a ring-buffer queue in a per-warp slice of global memory, one
//     entry (first child, number of children) per opened cell.  An octree cell of more than
//     leaf_max particles has nearly always all eight children in a solid body (7.5 to 7.95 on
//     average on the models here), so four entries fill a batch of 32 lanes without any search
//     for the lanes' cells, their records are read in runs, and an opened cell costs one queue
//     store.  When the queue fills up, the newest entries are taken first, i.e.
//     depth-first, which bounds its size (the order does not change the set of
//     interactions).  The cells are tested with the MAC at distance lambda r_JI (Eqs. 2, 5-7)
//     in FP32 with explicit rounding (so the decision is reproducible); accepted cells and the
//     particles of opened leaves join the shared-memory interaction list in the cells'
//     order, the particles by asynchronous global-to-shared copies (cp.async), waited for
//     only when the list is summed;
//   * the list is kept as structure of arrays (x, y, z, m), so two consecutive entries
//     load as packed pairs; every 128 entries are summed through Eq. (1) from zero and the
//     partial sums added in order (so the result does not depend on when, or by which warp,
//     a chunk is summed): each i-particle is held by S lanes that take every S-th quad of
//     entries on the packed FP32 pipe (f32x2 add, mul and fma: two interactions per
//     instruction; rsqrt on the SFU), the two halves and the S lanes summed at the end.
//     The potential is accumulated too; the member's own term -G m_i/eps is removed at the
//     end (Eq. 1 excludes j = i).
// Bound: instruction issue and the FP32 pipe (per quad of entries 24 packed operations of two
// cycles, 4 rsqrt, 4 loads); the node records (32 B per cell) stay in L2.  80 registers and
// 48 KB of shared memory at three blocks per SM; members and sums wait in shared memory
// during the traversal (held in registers they spill, and a spilling force loop costs 15 %;
// two blocks at 95 registers 12 % more time, four at 64 10 %).  What still spills is outside of
// the force loop: 12 B of stores and 36 B of loads in k_walk (44 and 36 with levels, and 44 and 116
// in walk_group_ordered), 64 and 116 in k_walk_batch.  The full walk of the
// Andromeda-like model at 2^22, leaves of 32: 2.55 ms, 0.69 warp instructions per interaction
// (3.03 ms and 0.81 with a queue of single cells).
#include <limits.h>
#include <math.h>

#include "gt_internal.cuh"
#include "walk_levels.cuh"
#include "walk_list.cuh"

namespace {

#ifndef GT_WALK_MINB
#define GT_WALK_MINB 3            // resident blocks per SM the register budget is sized for
#endif
constexpr int WT = 256;             // threads per block
constexpr int NWARP = WT / 32;
constexpr uint32_t LIST_CAP = 256;  // interaction-list entries per warp
constexpr uint32_t CHUNK = 128;     // entries whose forces are summed from zero before they join a member's sums
constexpr uint32_t WARP_SM = 4 * LIST_CAP + 4 * 4 * 32;  // the list, then the lanes' members and sums
// walk_group_ordered: the whole of a warp's words is the list; a batch that leaves FLUSH_AT entries has it summed
constexpr uint32_t SEG_CAP = 384, FLUSH_AT = 256;
static_assert(4 * SEG_CAP <= WARP_SM, "the list of walk_group_ordered");
// Depth-first reserve of the queue: popping the newest 32 cells and pushing at most
// 8 children each grows the queue by <= 224 per tree level, <= ~22 x 256 in all.
constexpr int LIFO_ROOM = 6144;

// MAC >= 0: the criterion is known at compile time; MAC_ANY takes the argument's
constexpr int MAC_ANY = -1;

template <int MAC>
__device__ __forceinline__ bool mac_accept(int mac_arg, float theta, float dacc_amin, float delta, float G, float cx,
                                           float cy, float cz, float bI, float4 jp, float bJ, float B2) {
    const int mac = MAC == MAC_ANY ? mac_arg : MAC;
    const float dx = __fsub_rn(jp.x, cx);
    const float dy = __fsub_rn(jp.y, cy);
    const float dz = __fsub_rn(jp.z, cz);
    const float r2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
    const float r = __fsqrt_rn(r2);
    const float d = (bI < r) ? __fsub_rn(r, bI) : 0.0f;   // lambda r_JI, Eqs. (6)-(7)
    if (mac == GT_MAC_OPENING_ANGLE) return bJ <= __fmul_rn(theta, d);  // Eq. (2)
    if (mac == GT_MAC_MULTIPOLE)  // Warren & Salmon: d >= b/2 + sqrt(b^2/4 + sqrt(3 B_2 / Delta_mul))
        return d >= __fadd_rn(__fmul_rn(0.5f, bJ),
                              __fsqrt_rn(__fadd_rn(__fmul_rn(__fmul_rn(0.25f, bJ), bJ),
                                                   __fsqrt_rn(__fdiv_rn(__fmul_rn(3.0f, B2), delta)))));
    const float d2 = __fmul_rn(d, d);                                   // Eq. (5), raised to the 4th power
    return __fmul_rn(__fmul_rn(d2, d2), dacc_amin) >= __fmul_rn(__fmul_rn(G, jp.w), __fmul_rn(bJ, bJ));
}

__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// 1/sqrt(r2) on the special-function unit; r2 >= eps^2 > 0 is never subnormal, so the
// flush-to-zero form needs no range handling
__device__ __forceinline__ float rsqrt_sfu(float r2) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(r2));
    return r;
}

// Two list entries (packed: x = (x_e, x_e+1), ...) against one i-particle (negated
// coordinates nx, ny, nz) on the packed FP32 pipe; the sums keep the two entries' shares
// in their two halves.
__device__ __forceinline__ void interact_pairs(float2 X, float2 Y, float2 Z, float2 W, float2 nx, float2 ny,
                                               float2 nz, float2 e2, float2 &ax, float2 &ay, float2 &az,
                                               float2 &ph) {
    const float2 dx = __fadd2_rn(X, nx), dy = __fadd2_rn(Y, ny), dz = __fadd2_rn(Z, nz);
    const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __ffma2_rn(dx, dx, e2)));
    const float2 rinv = make_float2(rsqrt_sfu(r2.x), rsqrt_sfu(r2.y));
    const float2 mr = __fmul2_rn(W, rinv);
    const float2 mr3 = __fmul2_rn(__fmul2_rn(mr, rinv), rinv);
    ax = __ffma2_rn(mr3, dx, ax);
    ay = __ffma2_rn(mr3, dy, ay);
    az = __ffma2_rn(mr3, dz, az);
    ph = __fadd2_rn(ph, mr);
}

// (value, member) of the extreme member on one axis: the smallest (want_max false) or
// largest value, the lowest member index on ties
__device__ __forceinline__ void warp_arg_ext(float &v, int &m, bool want_max) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const int m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const bool take = want_max ? (v2 > v || (v2 == v && m2 < m)) : (v2 < v || (v2 == v && m2 < m));
        if (take) { v = v2; m = m2; }
    }
}

// Centre of Ritter's efficient bounding sphere of the group's members (Appendix B): the
// first diameter joins the extreme members of the axis whose pair is farthest apart; the
// sphere then grows towards the first member outside it (member order) until none is,
// at most cnt times.  FP32, every operation rounded as written.  Member k < 32 is the
// first member of the lanes holding slot k (pi), the others the second of the lanes holding slot2 (pi2).
__device__ __forceinline__ void ebs_centre(float4 pi, float4 pi2, bool mine1, bool mine2, int slot, int slot2,
                                           int logS, int logS2, uint32_t cnt, float &cx, float &cy, float &cz) {
    const unsigned FULL = 0xffffffffu;
    const float INF = __int_as_float(0x7f800000);
    auto coord = [](const float4 &p, int a) { return a == 0 ? p.x : (a == 1 ? p.y : p.z); };
    // the member's position, fetched from the lane that holds it
    auto fetch = [&](int m, float &x, float &y, float &z) {
        const bool second = m >= 32;
        const int src = second ? (m - 32) << logS2 : (m << logS);
        const float4 a1 = make_float4(__shfl_sync(FULL, pi.x, src), __shfl_sync(FULL, pi.y, src),
                                      __shfl_sync(FULL, pi.z, src), 0.f);
        const float4 a2 = make_float4(__shfl_sync(FULL, pi2.x, src), __shfl_sync(FULL, pi2.y, src),
                                      __shfl_sync(FULL, pi2.z, src), 0.f);
        x = second ? a2.x : a1.x; y = second ? a2.y : a1.y; z = second ? a2.z : a1.z;
    };
    float bd2 = -1.0f, lx = 0.f, ly = 0.f, lz = 0.f, hx = 0.f, hy = 0.f, hz = 0.f;
    for (int ax = 0; ax < 3; ax++) {
        float vmin = mine1 ? coord(pi, ax) : INF, vmax = mine1 ? coord(pi, ax) : -INF;
        int mmin = mine1 ? slot : 1 << 20, mmax = mmin;
        if (mine2) {
            const float v2 = coord(pi2, ax);
            if (v2 < vmin) { vmin = v2; mmin = slot2; }  // the second member has the larger index
            if (v2 > vmax) { vmax = v2; mmax = slot2; }
        }
        warp_arg_ext(vmin, mmin, false);
        warp_arg_ext(vmax, mmax, true);
        float ax0, ay0, az0, ax1, ay1, az1;
        fetch(mmin, ax0, ay0, az0);
        fetch(mmax, ax1, ay1, az1);
        const float dx = __fsub_rn(ax1, ax0), dy = __fsub_rn(ay1, ay0), dz = __fsub_rn(az1, az0);
        const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
        if (d2 > bd2) { bd2 = d2; lx = ax0; ly = ay0; lz = az0; hx = ax1; hy = ay1; hz = az1; }
    }
    cx = __fmul_rn(0.5f, __fadd_rn(lx, hx));
    cy = __fmul_rn(0.5f, __fadd_rn(ly, hy));
    cz = __fmul_rn(0.5f, __fadd_rn(lz, hz));
    float r = __fmul_rn(0.5f, __fsqrt_rn(bd2));
    for (uint32_t it = 0; it < cnt; it++) {
        const float r2 = __fmul_rn(r, r);
        auto outside = [&](const float4 &p) {
            const float dx = __fsub_rn(p.x, cx), dy = __fsub_rn(p.y, cy), dz = __fsub_rn(p.z, cz);
            return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz)) > r2;
        };
        const unsigned b1 = __ballot_sync(FULL, mine1 && outside(pi));
        const unsigned b2 = __ballot_sync(FULL, mine2 && outside(pi2));
        int m;
        if (b1) m = (__ffs(b1) - 1) >> logS;
        else if (b2) m = 32 + ((__ffs(b2) - 1) >> logS2);
        else break;
        float px, py, pz;
        fetch(m, px, py, pz);
        const float dx = __fsub_rn(px, cx), dy = __fsub_rn(py, cy), dz = __fsub_rn(pz, cz);
        const float d = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz)));
        const float rn = __fmul_rn(0.5f, __fadd_rn(r, d));
        const float f = __fdiv_rn(__fsub_rn(d, rn), d);
        cx = __fadd_rn(cx, __fmul_rn(f, dx));
        cy = __fadd_rn(cy, __fmul_rn(f, dy));
        cz = __fadd_rn(cz, __fmul_rn(f, dz));
        r = rn;
    }
}

// members [a0, a1) of group g in the active list
__device__ __forceinline__ void group_range(const WalkArgs &a, uint32_t g, uint32_t ngroups, uint32_t &a0, uint32_t &a1) {
    const uint32_t na = a.ctl->n_active;
    if (a.gstart) {
        a0 = a.gstart[g];
        a1 = g + 1 < ngroups ? a.gstart[g + 1] : na;
    } else {
        a0 = g * (uint32_t)a.gmax;
        a1 = min(a0 + (uint32_t)a.gmax, na);
    }
}

// The i-particle of active position k; an index outside the system is reported and particle 0 walked instead.
__device__ __forceinline__ uint32_t member_of(const WalkArgs &a, uint32_t k) {
    uint32_t i = a.active ? a.active[k] : k;
    if (i >= a.n) {
        gt_set_error(a.ctl, GT_EINVAL, GTK_WALK);
        i = 0u;
    }
    return i;
}

struct Pseudo {
    float x, y, z, b, dacc_amin;  // centre and radius of the group's sphere; Delta_acc times its smallest |a_old|
};

// A group's pseudo i-particle, and the lane's members: mem[0], mem[MS] the first and second, negated, with the
// first quad and the quad step of the lane's share in the fourth word; mem[2 MS], mem[3 MS] their sums, zero (MS 32:
// in shared memory; 1: the lane's own).  ORDERED: a second member has one lane.  False for a malformed group.
template <bool ORDERED, uint32_t MS>
__device__ __forceinline__ bool group_setup(const WalkArgs &a, uint32_t a0, uint32_t cnt, float4 *mem, Pseudo &ps) {
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    // a group of more than 32: member k < 32 has lane k, the others share the lanes a second time
    const bool two = cnt > 32u;
    if (cnt == 0u || cnt > 64u || (two && a.ij_share > 1)) return false;
    const int S = two ? 1 : (a.ij_share ? a.ij_share : 32 >> (cnt <= 1 ? 0 : 32 - __clz(cnt - 1)));
    const int logS = __ffs(S) - 1;
    const int slot = lane >> logS, sub = lane & (S - 1);
    const bool have = (uint32_t)slot < cnt;
    // lanes of one second member: like S, as many as their count (1 to 32) leaves, so that they don't idle
    const int logS2 = (!ORDERED && two && !a.ij_share) ? 5 - (cnt <= 33u ? 0 : 32 - __clz(cnt - 33u)) : 0;
    const int slot2 = 32 + (lane >> logS2), sub2 = lane & ((1 << logS2) - 1);
    const bool have2 = two && (uint32_t)slot2 < cnt;
    const uint32_t i = member_of(a, a0 + (have ? (uint32_t)slot : 0u));
    const uint32_t i2 = have2 ? member_of(a, a0 + (uint32_t)slot2) : i;
    const float4 pi = a.posm[i];
    const float4 pi2 = have2 ? a.posm[i2] : pi;
    float ao = have ? (a.aold ? a.aold[i] : 0.0f) : INFINITY;
    if (have2) ao = fminf(ao, a.aold ? a.aold[i2] : 0.0f);

    // lanes without a member repeat member 0: no effect on the box
    float mnx = fminf(pi.x, pi2.x), mny = fminf(pi.y, pi2.y), mnz = fminf(pi.z, pi2.z);
    float mxx = fmaxf(pi.x, pi2.x), mxy = fmaxf(pi.y, pi2.y), mxz = fmaxf(pi.z, pi2.z);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mnx = fminf(mnx, __shfl_xor_sync(FULL, mnx, o));
        mny = fminf(mny, __shfl_xor_sync(FULL, mny, o));
        mnz = fminf(mnz, __shfl_xor_sync(FULL, mnz, o));
        mxx = fmaxf(mxx, __shfl_xor_sync(FULL, mxx, o));
        mxy = fmaxf(mxy, __shfl_xor_sync(FULL, mxy, o));
        mxz = fmaxf(mxz, __shfl_xor_sync(FULL, mxz, o));
        ao = fminf(ao, __shfl_xor_sync(FULL, ao, o));
    }
    float cx = __fmul_rn(0.5f, __fadd_rn(mnx, mxx));
    float cy = __fmul_rn(0.5f, __fadd_rn(mny, mxy));
    float cz = __fmul_rn(0.5f, __fadd_rn(mnz, mxz));
    if (a.sphere == 1) ebs_centre(pi, pi2, have && sub == 0, have2 && sub2 == 0, slot, slot2, logS, logS2, cnt, cx, cy, cz);
    const float ddx = __fsub_rn(pi.x, cx), ddy = __fsub_rn(pi.y, cy), ddz = __fsub_rn(pi.z, cz);
    float d2 = __fadd_rn(__fadd_rn(__fmul_rn(ddx, ddx), __fmul_rn(ddy, ddy)), __fmul_rn(ddz, ddz));
    {
        const float ex = __fsub_rn(pi2.x, cx), ey = __fsub_rn(pi2.y, cy), ez = __fsub_rn(pi2.z, cz);
        d2 = fmaxf(d2, __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d2 = fmaxf(d2, __shfl_xor_sync(FULL, d2, o));
    ps = Pseudo{cx, cy, cz, __fmul_rn(__fsqrt_rn(d2), GT_RADIUS_MARGIN), __fmul_rn(a.delta_acc, ao)};
    mem[0] = make_float4(-pi.x, -pi.y, -pi.z, __uint_as_float((uint32_t)sub | (1u << logS << 8)));
    mem[MS] = make_float4(-pi2.x, -pi2.y, -pi2.z, __uint_as_float((uint32_t)sub2 | (1u << logS2 << 8)));
    mem[2 * MS] = mem[3 * MS] = make_float4(0.f, 0.f, 0.f, 0.f);
    return true;
}

// Forces of quads [k0, k1) of a list (arrays of `cap` entries) on one member of every lane, summed from zero.
__device__ __forceinline__ float4 chunk_force(const float *lx, uint32_t cap, float4 p, float eps2, uint32_t k0,
                                              uint32_t k1) {
    const float4 *px = (const float4 *)lx, *py = (const float4 *)(lx + cap), *pz = (const float4 *)(lx + 2 * cap),
                 *pw = (const float4 *)(lx + 3 * cap);
    const uint32_t share = __float_as_uint(p.w), step = share >> 8;
    const float2 e2 = make_float2(eps2, eps2);
    const float2 nx = make_float2(p.x, p.x), ny = make_float2(p.y, p.y), nz = make_float2(p.z, p.z);
    float2 sx = make_float2(0.f, 0.f), sy = sx, sz = sx, sp = sx;
#pragma unroll 1
    for (uint32_t k = k0 + (share & 0xffu); k < k1; k += step) {
        const float4 X = px[k], Y = py[k], Z = pz[k], W = pw[k];
        interact_pairs(make_float2(X.x, X.y), make_float2(Y.x, Y.y), make_float2(Z.x, Z.y), make_float2(W.x, W.y),
                       nx, ny, nz, e2, sx, sy, sz, sp);
        interact_pairs(make_float2(X.z, X.w), make_float2(Y.z, Y.w), make_float2(Z.z, Z.w), make_float2(W.z, W.w),
                       nx, ny, nz, e2, sx, sy, sz, sp);
    }
    return make_float4(__fadd_rn(sx.x, sx.y), __fadd_rn(sy.x, sy.y), __fadd_rn(sz.x, sz.y), __fadd_rn(sp.x, sp.y));
}

__device__ __forceinline__ void add_force(float4 &sum, float4 f) {
    float4 t = sum;
    t.x = __fadd_rn(t.x, f.x); t.y = __fadd_rn(t.y, f.y); t.z = __fadd_rn(t.z, f.z); t.w = __fsub_rn(t.w, f.w);
    sum = t;
}

// Massless entries behind the last of a list up to a multiple of four: they add exactly nothing.
__device__ __forceinline__ void pad_list(float *lx, uint32_t cap, uint32_t list_n) {
    const uint32_t lane = threadIdx.x & 31u;
    if (lane < ((0u - list_n) & 3u)) {
        float *e = lx + list_n + lane;
        e[0] = e[cap] = e[2 * cap] = e[3 * cap] = 0.f;
    }
    __syncwarp();
}

// The warp of walk_list.cuh.
struct Lanes {
    __device__ __forceinline__ uint32_t lane() const { return threadIdx.x & 31u; }
    __device__ __forceinline__ void sync() const { __syncwarp(); }
};

// A team's list: the first list_n (< CHUNK) entries from quad `from` on moved to the front of the list, by one warp.
__device__ __forceinline__ void move_rest(float *lx, uint32_t cap, uint32_t list_n, uint32_t from) {
    const uint32_t lane = threadIdx.x & 31u;
    if (4u * lane < list_n) {
        float4 *q = (float4 *)lx;
#pragma unroll
        for (uint32_t c = 0; c < 4; c++) q[c * (cap / 4) + lane] = q[c * (cap / 4) + from + lane];
    }
}

struct Batch {
    float4 jp;
    uint32_t l0, mine;  // first child or first particle; entries for the list: one, a leaf's particles, none
    uint32_t nch;       // children of an opened cell
    bool ok;            // accepted
};

// A batch of cells, one per lane.
struct Take {
    uint32_t node, nb;  // nb: queue entries taken
    bool valid;
};

// The children of the next four queue entries, eight lanes each (sib: the lane's entry).
__device__ __forceinline__ Take take_four(uint2 sib, uint32_t avail) {
    const uint32_t lane = threadIdx.x & 31u, nb = min(avail, 4u);
    const bool valid = (lane >> 3) < nb && (lane & 7u) < sib.y;
    return Take{valid ? sib.x + (lane & 7u) : 0u, nb, valid};
}

// The children of as many whole entries from the queue's head on as fill the lanes: for flat trees (DevCtl::flat), whose
// cells have four children on a sheet and two on a filament, so that four entries would leave half or three quarters of
// the lanes idle.  Every particle, with four entries and packed, us: a sheet of 2^20 (leaves of 4) 887 and 762, a line
// 1144 and 720, a sheet of 2^22 3653 and 3102, a line 6048 and 3632; solid bodies gain nothing by it (a Plummer sphere of
// 2^22, leaves of 16: 2489 and 2692), nor do filaments and slabs that are solid at the scale of the groups (2^18, a
// hundredth thick, leaves of 16: 1361 and 1480, 354 and 356).  So a tree is flat if its cells have fewer than five children,
// on average over all cells (sheets up to 4, slabs of a thousandth at 2^22 4.3, thicker ones and filaments 5 to 8) and
// fewer than 4.5 on average over the levels (solid models with leaves of one or two particles have 3 to 4.3 over all
// cells, most of which are the last two levels', but 4.5 and more over the levels from 2^16 on).  Both in one kernel would
// cost solid bodies 2 % (batches) to 3 % (registers, code), so each has its own, and the one that isn't meant ends at
// once (1 to 3 us a call).
__device__ __forceinline__ Take take_packed(const uint2 *q, uint32_t head, uint32_t avail, uint32_t qmask) {
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned FULL = 0xffffffffu;
    uint2 e = make_uint2(0u, 0u);
    if (lane < avail) e = q[(head + lane) & qmask];
    const uint32_t incl = warp_incl_scan(e.y), excl = incl - e.y;
    const unsigned taken = __ballot_sync(FULL, e.y && incl <= 32u);
    const uint32_t nb = __popc(taken);
    // bit p: the first child of an entry has lane p
    const unsigned m = __reduce_or_sync(FULL, e.y && incl <= 32u ? 1u << excl : 0u) & (0xffffffffu >> (31u - lane));
    const uint32_t node = __shfl_sync(FULL, e.x, __popc(m) - 1) + lane - (31u - (uint32_t)__clz(m));
    const bool valid = lane < __shfl_sync(FULL, incl, nb - 1u);
    return Take{valid ? node : 0u, nb, valid};
}

// One batch: a cell per lane, and what the MAC says.
template <int MAC>
__device__ __forceinline__ Batch test_batch(const WalkArgs &a, const Pseudo &ps, const Take &k, uint32_t &tests) {
    bool valid = k.valid;
    uint32_t node = k.node;
#if GT_DEBUG
    const uint32_t nnodes = a.ctl->level_start[GT_TREE_LEVELS];
    if (node >= nnodes) {
        gt_set_error(a.ctl, GT_EINVAL, GTK_WALK);
        valid = false;
        node = 0u;
    }
#endif
    Batch t;
    t.jp = a.jpos[node];
    const float4 wk = a.walk[node];
    const uint32_t l1 = __float_as_uint(wk.z);
    const bool leaf = (l1 & GT_LEAF_FLAG) != 0u;
    t.l0 = __float_as_uint(wk.y);
#if GT_DEBUG
    if (valid && (unsigned long long)t.l0 + (l1 & ~GT_LEAF_FLAG) > (leaf ? a.n : nnodes)) {
        gt_set_error(a.ctl, GT_EINVAL, GTK_WALK);
        valid = false;
    }
#endif
    tests += valid ? 1u : 0u;
    t.ok = valid && mac_accept<MAC>(a.mac, a.theta, ps.dacc_amin, a.delta_acc, a.G, ps.x, ps.y, ps.z, ps.b, t.jp, wk.x,
                                    wk.w);
    const bool opened = valid && !t.ok;
    t.nch = opened && !leaf ? l1 : 0u;
    t.mine = opened && leaf ? (l1 & ~GT_LEAF_FLAG) : (t.ok ? 1u : 0u);
    return t;
}

// The entries of a batch with index in [w0, w1) into the list: entry e goes to slot to + e.  `excl`: the index
// of the lane's first; lm: lanes with an opened leaf.
template <bool PACK>
__device__ __forceinline__ void write_entries(const WalkArgs &a, const Batch &t, uint32_t excl, unsigned lm, float *lx,
                                              uint32_t cap, uint32_t to, uint32_t w0, uint32_t w1) {
    const unsigned FULL = 0xffffffffu;
    if (t.ok && excl >= w0 && excl < w1) {
        float *e = list_at(lx, to, excl);
        e[0] = t.jp.x; e[cap] = t.jp.y; e[2 * cap] = t.jp.z; e[3 * cap] = t.jp.w;
    }
    // opened leaves next to each other that hold one range of particles are copied together, asynchronously: those among
    // one entry's children (eight lanes each), or, where entries are packed, that begin where the one before ends
    unsigned starts = lm & ~((lm << 1) & 0xfefefefeu);
    if (PACK) {
        const uint32_t before = __shfl_up_sync(FULL, t.l0 + t.mine, 1);  // where the lane before ends
        starts = lm & ~(__ballot_sync(FULL, before == t.l0) & (lm << 1));
    }
    for (unsigned m = starts; m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        // the run's last lane: before the next lane that is no leaf or starts a run of its own
        const unsigned stop = (~lm | (m & (m - 1))) & (0xfffffffeu << src);
        const int end = PACK ? (stop ? __ffs(stop) - 2 : 31)
                             : min(src + __ffs(~((lm >> src) & 0xffu)) - 2, src | 7);
        const uint32_t le = __shfl_sync(FULL, excl, src);
        const uint32_t e1 = min(__shfl_sync(FULL, excl + t.mine, end), w1);
        const float4 *p = a.posm + __shfl_sync(FULL, t.l0, src);
        for (uint32_t e = max(le, w0) + (threadIdx.x & 31u); e < e1; e += 32) {
            const float *from = (const float *)&p[e - le];
            float *d = list_at(lx, to, e);
            cp_async4(d, from);
            cp_async4(d + cap, from + 1);
            cp_async4(d + 2 * cap, from + 2);
            cp_async4(d + 3 * cap, from + 3);
        }
    }
}

// The members' sums, reduced over their lanes, to the caller's accelerations.  True (for the warp) if LEVELS, the walk
// is one that chooses levels (inv_c2 > 0), and one of them is near a level's threshold.
template <bool LEVELS, uint32_t MS>
__device__ __forceinline__ bool store_group(const WalkArgs &a, uint32_t a0, uint32_t a1, const float4 *mem) {
    const uint32_t lane = threadIdx.x & 31u;
    bool near = false;
    for (uint32_t who = 0; who < a1 - a0; who += 32) {
        const uint32_t share = __float_as_uint(mem[who / 32 * MS].w), S = share >> 8;
        float4 sum = mem[2 * MS + who / 32 * MS];
        for (uint32_t o = 1; o < S; o <<= 1) {
            sum.x += __shfl_xor_sync(0xffffffffu, sum.x, o);
            sum.y += __shfl_xor_sync(0xffffffffu, sum.y, o);
            sum.z += __shfl_xor_sync(0xffffffffu, sum.z, o);
            sum.w += __shfl_xor_sync(0xffffffffu, sum.w, o);
        }
        const uint32_t k = a0 + who + lane / S;
        if ((share & 0xffu) == 0u && k < a1) {
            const uint32_t i = a.active ? a.active[k] : k;
            const float phi = fmaf(a.posm[i < a.n ? i : 0u].w, a.inv_eps, sum.w);
            const float4 f = make_float4(a.G * sum.x, a.G * sum.y, a.G * sum.z, a.G * phi);
            a.acc[k] = f;
            if (LEVELS) near = near || near_level((f.x * f.x + f.y * f.y + f.z * f.z) * a.inv_c2);
        }
    }
    return LEVELS && __any_sync(0xffffffffu, near);
}

// Forces of a list's first nquad quads (arrays of `cap` entries from lx on) on one member of every lane, added to
// its sums.
__device__ __forceinline__ void sum_segment(const float *lx, uint32_t cap, float4 *member, float4 *sum, float eps2,
                                            uint32_t nquad) {
    const float4 *px = (const float4 *)lx, *py = (const float4 *)(lx + cap), *pz = (const float4 *)(lx + 2 * cap),
                 *pw = (const float4 *)(lx + 3 * cap);
    const float4 p = *member, s = *sum;
    const uint32_t share = __float_as_uint(p.w), step = share >> 8;
    const float2 e2 = make_float2(eps2, eps2);
    const float2 nx = make_float2(p.x, p.x), ny = make_float2(p.y, p.y), nz = make_float2(p.z, p.z);
    float2 sx = make_float2(s.x, 0.f), sy = make_float2(s.y, 0.f), sz = make_float2(s.z, 0.f);
    float2 sp = make_float2(-s.w, 0.f);
#pragma unroll 1
    for (uint32_t k = share & 0xffu; k < nquad; k += step) {
        const float4 X = px[k], Y = py[k], Z = pz[k], W = pw[k];
        interact_pairs(make_float2(X.x, X.y), make_float2(Y.x, Y.y), make_float2(Z.x, Z.y), make_float2(W.x, W.y),
                       nx, ny, nz, e2, sx, sy, sz, sp);
        interact_pairs(make_float2(X.z, X.w), make_float2(Y.z, Y.w), make_float2(Z.z, Z.w), make_float2(W.z, W.w),
                       nx, ny, nz, e2, sx, sy, sz, sp);
    }
    *sum = make_float4(__fadd_rn(sx.x, sx.y), __fadd_rn(sy.x, sy.y), __fadd_rn(sz.x, sz.y), -__fadd_rn(sp.x, sp.y));
}

struct Cell {
    float4 jp;
    uint32_t l0;      // first child or first particle
    uint32_t nch, lc; // children of an opened cell, particles of an opened leaf
    bool ok;          // accepted
};

// One cell per lane, and what the MAC says.
template <int MAC>
__device__ __forceinline__ Cell test_cell(const WalkArgs &a, const Pseudo &ps, uint32_t node, bool valid) {
#if GT_DEBUG
    const uint32_t nnodes = a.ctl->level_start[GT_TREE_LEVELS];
    if (valid && node >= nnodes) {
        gt_set_error(a.ctl, GT_EINVAL, GTK_WALK);
        valid = false;
    }
#endif
    if (!valid) node = 0u;
    Cell t;
    t.jp = a.jpos[node];
    const float4 wk = a.walk[node];
    const uint32_t l1 = __float_as_uint(wk.z);
    const bool leaf = (l1 & GT_LEAF_FLAG) != 0u;
    t.l0 = __float_as_uint(wk.y);
#if GT_DEBUG
    if (valid && (unsigned long long)t.l0 + (l1 & ~GT_LEAF_FLAG) > (leaf ? a.n : nnodes)) {
        gt_set_error(a.ctl, GT_EINVAL, GTK_WALK);
        valid = false;
    }
#endif
    t.ok = valid && mac_accept<MAC>(a.mac, a.theta, ps.dacc_amin, a.delta_acc, a.G, ps.x, ps.y, ps.z, ps.b, t.jp, wk.x,
                                    wk.w);
    const bool opened = valid && !t.ok;
    t.nch = opened && !leaf ? l1 : 0u;
    t.lc = opened && leaf ? (l1 & ~GT_LEAF_FLAG) : 0u;
    return t;
}

// An accepted cell's entry.
__device__ __forceinline__ void write_cell(const Cell &t, float *e, uint32_t cap) {
    e[0] = t.jp.x; e[cap] = t.jp.y; e[2 * cap] = t.jp.z; e[3 * cap] = t.jp.w;
}

// The particles of a batch's opened leaves with index in [w0, w1) into the list: particle e goes to slot to + e.
// `incl`: the warp scan of lc; lm: lanes with an opened leaf.  Opened leaves next to each other in the batch that
// hold one range of particles (siblings) are copied together, asynchronously.
__device__ __forceinline__ void write_particles(const WalkArgs &a, const Cell &t, uint32_t incl, unsigned lm, float *lx,
                                                uint32_t cap, uint32_t to, uint32_t w0, uint32_t w1) {
    const unsigned FULL = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t before = __shfl_up_sync(FULL, t.l0 + t.lc, 1);  // where the lane before ends
    const bool joins = lane > 0 && t.lc && (lm >> (lane - 1u) & 1u) && before == t.l0;
    const unsigned starts = lm & ~__ballot_sync(FULL, joins);
    for (unsigned m = starts; m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        // the run's last lane: before the next lane that is no leaf or starts a run of its own
        const unsigned stop = (~lm | (starts & ~(1u << src))) & (0xfffffffeu << src);
        const int end = stop ? __ffs(stop) - 2 : 31;
        const uint32_t le = __shfl_sync(FULL, incl - t.lc, src);
        const uint32_t e1 = min(__shfl_sync(FULL, incl, end), w1);
        const float4 *p = a.posm + __shfl_sync(FULL, t.l0, src);
        for (uint32_t e = max(le, w0) + lane; e < e1; e += 32) {
            const float *from = (const float *)&p[e - le];
            float *d = list_at(lx, to, e);
            cp_async4(d, from);
            cp_async4(d + cap, from + 1);
            cp_async4(d + 2 * cap, from + 2);
            cp_async4(d + 3 * cap, from + 3);
        }
    }
}

// Particles among the batch's children and particles number 32 r to 32 r + 31 (they are counted together, lane by
// lane; `first`: the number of the lane's first).  A batch whose particles don't fit behind the list goes on in
// steps of these 32: a segment ends before the step that would overflow it.
__device__ __forceinline__ uint32_t particles_of_step(uint32_t first, uint32_t lc, uint32_t r) {
    const uint32_t lo = max(first, 32u * r), hi = min(first + lc, 32u * r + 32u);
    return __reduce_add_sync(0xffffffffu, hi > lo ? hi - lo : 0u);
}

// One group again, in a fixed order of summation: a batch is the queue's next 32 cells, its accepted cells precede
// the particles of its opened leaves in the list, the list is summed whenever a batch leaves FLUSH_AT entries or
// would overflow it, every chain of additions runs over the whole walk, and a second member has one lane.  Block
// steps turn forces into discrete levels, and a particle whose |a| is within a rounding of a level's threshold
// would get another step from any other order of the same sums (1 particle in 10^7 and step).  The groups of
// particles near a threshold (near_level: 2 groups in 10^4) are walked a second time by this function, so that their levels
// don't depend on how walk_group arranges its sums; where a force's terms cancel so far that the rounding errors exceed
// near_level's window, a level can still do so (walk_group's own order is fixed too: levels never depend on the teams or
// on the run).  As the only walk it would take 2.9 ms against walk_group's 2.6 (every particle at 2^22).  lx: the warp's
// WARP_SM words of shared memory.
__device__ __noinline__ void walk_group_ordered(const WalkArgs &a, uint32_t g, uint32_t ngroups, float *lx, uint2 *q) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t qmask = gt_queue_ring(a.qcap) - 1u;
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = lanemask_lt();
    float4 mem[4];
    uint32_t a0, a1;
    group_range(a, g, ngroups, a0, a1);
    const bool two = a1 - a0 > 32u;
    Pseudo ps;
    if (!group_setup<true, 1>(a, a0, a1 - a0, mem, ps)) return;
    uint32_t list_n = 0;
    auto flush = [&]() {
        cp_async_wait_all();
        __syncwarp();
        pad_list(lx, SEG_CAP, list_n);
        const uint32_t nquad = (list_n + 3) >> 2;
        sum_segment(lx, SEG_CAP, &mem[0], &mem[2], a.eps2, nquad);
        if (two) sum_segment(lx, SEG_CAP, &mem[1], &mem[3], a.eps2, nquad);
        list_n = 0;
        __syncwarp();
    };
    uint32_t head = 0, tail = 1, off = 0;  // queue entries; children of the head's entry already taken
    if (lane == 0) q[0] = make_uint2(0u, 1u);  // the root
    __syncwarp();
    bool overflow = false;
    while (head != tail) {
        // the next 32 cells: breadth-first from the head while there is room, depth-first from the tail after
        const uint32_t avail = tail - head;
        uint32_t node, ncell;
        if (8 * (int)avail <= a.qcap - LIFO_ROOM) {
            uint2 e = make_uint2(0u, 0u);
            if (lane < avail) e = q[(head + lane) & qmask];
            if (lane == 0) {
                e.x += off;
                e.y -= off;
            }
            if ((__ballot_sync(FULL, e.y == 8u) & 0xfu) == 0xfu) {  // four whole entries of eight
                node = __shfl_sync(FULL, e.x, lane >> 3) + (lane & 7u);
                ncell = 32u;
                head += 4u;
                off = 0u;
            } else {
                const uint32_t incl = warp_incl_scan(e.y), excl = incl - e.y;
                // bit p: an entry's first cell has lane p; the entries before it are one after another from lane 0
                const unsigned m = __reduce_or_sync(FULL, e.y && excl < 32u ? 1u << excl : 0u) & (lt | (1u << lane));
                node = __shfl_sync(FULL, e.x, __popc(m) - 1) + lane - (31u - (uint32_t)__clz(m));
                ncell = min(__shfl_sync(FULL, incl, 31), 32u);
                const uint32_t whole = __popc(__ballot_sync(FULL, e.y && incl <= 32u));
                const uint32_t cut = __shfl_sync(FULL, excl, whole & 31u), left = __shfl_sync(FULL, incl, 31);
                head += whole;
                off = left > 32u ? 32u - cut : 0u;
            }
        } else {
            const uint32_t nb = min(avail, 4u), o = lane >> 3;
            tail -= nb;
            uint2 e = o < nb ? q[(tail + o) & qmask] : make_uint2(0u, 0u);
            if (o < nb && tail + o == head) {
                e.x += off;
                e.y -= off;
            }
            if (tail == head) off = 0u;
            // the cells side by side in the lanes, as from the head
            const uint32_t n0 = __shfl_sync(FULL, e.y, 0), n1 = n0 + __shfl_sync(FULL, e.y, 8),
                           n2 = n1 + __shfl_sync(FULL, e.y, 16), n3 = n2 + __shfl_sync(FULL, e.y, 24);
            const uint32_t own = (lane >= n0 ? 1u : 0u) + (lane >= n1 ? 1u : 0u) + (lane >= n2 ? 1u : 0u);
            node = __shfl_sync(FULL, e.x, 8u * own) + lane - (own == 0 ? 0u : own == 1 ? n0 : own == 2 ? n1 : n2);
            ncell = n3;
        }
        const Cell t = test_cell<MAC_ANY>(a, ps, node, lane < ncell);
        // accepted cells -> list (there is room: fewer than FLUSH_AT entries at a batch's begin)
        const unsigned am = __ballot_sync(FULL, t.ok);
        if (t.ok) write_cell(t, lx + list_n + __popc(am & lt), SEG_CAP);
        list_n += __popc(am);
        // opened cells: their children join the queue as one entry per cell
        const unsigned om = __ballot_sync(FULL, t.nch != 0u);
        if (om) {
            if (t.nch) q[(tail + __popc(om & lt)) & qmask] = make_uint2(t.l0, t.nch);
            tail += __popc(om);
            if (8u * (tail - head) > (uint32_t)a.qcap) {  // more cells than the queue may hold?  count them
                __syncwarp();
                uint32_t live = 0;
                for (uint32_t e = head + lane; e < tail; e += 32) live += q[e & qmask].y;
                if (__reduce_add_sync(FULL, live) - off > (uint32_t)a.qcap) {
                    overflow = true;
                    break;
                }
            }
        }
        // opened leaves -> their particles
        const unsigned lm = __ballot_sync(FULL, t.lc != 0u);
        if (lm) {
            const uint32_t incl = warp_incl_scan(t.lc), tot = __shfl_sync(FULL, incl, 31);
            if (list_n + tot <= SEG_CAP) {
                write_particles(a, t, incl, lm, lx, SEG_CAP, list_n, 0u, tot);
                list_n += tot;
            } else if (__all_sync(FULL, t.lc < 2048u)) {  // in steps of 32 children and particles
                const uint32_t both = warp_incl_scan(t.nch + t.lc), first = both - t.lc;  // a lane has one or the other
                const uint32_t steps = (__shfl_sync(FULL, both, 31) + 31u) >> 5;
                uint32_t w0 = 0, w1 = 0;  // particles before this window, and before this step
                for (uint32_t r = 0; r < steps; r++) {
                    const uint32_t pm = particles_of_step(first, t.lc, r);
                    if (pm && list_n + (w1 - w0) + pm > SEG_CAP) {
                        write_particles(a, t, incl, lm, lx, SEG_CAP, list_n - w0, w0, w1);
                        list_n += w1 - w0;
                        flush();
                        w0 = w1;
                    }
                    w1 += pm;
                }
                write_particles(a, t, incl, lm, lx, SEG_CAP, list_n - w0, w0, w1);
                list_n += w1 - w0;
            } else {  // a leaf of 2048 or more particles (coincident particles chained to level 21)
                flush();
                for (uint32_t w0 = 0; w0 < tot;) {
                    const uint32_t w1 = min(tot, w0 + (SEG_CAP - list_n));
                    write_particles(a, t, incl, lm, lx, SEG_CAP, list_n - w0, w0, w1);
                    list_n += w1 - w0;
                    w0 = w1;
                    if (list_n == SEG_CAP) flush();
                }
            }
        }
        if (list_n >= FLUSH_AT) flush();
        __syncwarp();
    }
    if (!overflow) {
        flush();
    } else {
        if (lane == 0) gt_set_error(a.ctl, GT_EOVERFLOW, GTK_WALK);
        cp_async_wait_all();
        mem[2] = mem[3] = make_float4(NAN, NAN, NAN, NAN);
    }
    __syncwarp();
    // the range is read again: held over the traversal it would cost registers
    group_range(a, g, ngroups, a0, a1);
    (void)store_group<false, 1>(a, a0, a1, mem);
    __syncwarp();
}

// One group g of system a (Sec. 2.3) by one warp.  The interactions and MAC tests are added to stat[0] and
// stat[1].  lx: the warp's WARP_SM words of shared memory.
template <int MAC, bool LEVELS, bool PACK>
__device__ __forceinline__ void walk_group(const WalkArgs &a, uint32_t g, uint32_t ngroups, float *lx, uint2 *q,
                                           unsigned long long *stat) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t qmask = gt_queue_ring(a.qcap) - 1u;
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = lanemask_lt();
    float4 *mem = (float4 *)(lx + 4 * LIST_CAP) + lane;
    uint32_t a0, a1;
    group_range(a, g, ngroups, a0, a1);
    const bool two = a1 - a0 > 32u;
    Pseudo ps;
    if (!group_setup<false, 32>(a, a0, a1 - a0, mem, ps)) {
        if (lane == 0) gt_set_error(a.ctl, GT_EINVAL, GTK_WALK);
        return;
    }
    uint32_t list_n = 0, chunks = 0, tests = 0;  // entries in the list; chunks summed; this lane's MAC tests
    auto chunk = [&](uint32_t k0, uint32_t k1) {
        add_force(mem[64], chunk_force(lx, LIST_CAP, mem[0], a.eps2, k0, k1));
        if (two) add_force(mem[96], chunk_force(lx, LIST_CAP, mem[32], a.eps2, k0, k1));
    };
    // every full chunk of the list, then the rest moved to its front
    auto flush = [&]() {
        cp_async_wait_all();
        chunks += flush_chunks<CHUNK>(lx, LIST_CAP, list_n, Lanes{}, chunk);
    };
    uint32_t head = 0, tail = 1;
    if (lane == 0) q[0] = make_uint2(0u, 1u);  // the root
    __syncwarp();
    bool overflow = false;
    while (head != tail) {
        // breadth-first from the head while there is room, depth-first from the tail after
        uint32_t nb = min(tail - head, 4u), base = head;
        const bool newest = 8 * (int)(tail - head) > a.qcap - LIFO_ROOM;
        Take k;
        if (PACK && !newest) {
            k = take_packed(q, head, tail - head, qmask);
            head += k.nb;
        } else {
            if (newest) {
                tail -= nb;
                base = tail;
            } else {
                head += nb;
            }
            k = take_four(q[(base + (lane >> 3)) & qmask], nb);
        }
        const Batch t = test_batch<MAC>(a, ps, k, tests);
        // opened cells: their children join the queue as one entry per cell
        const unsigned om = __ballot_sync(FULL, t.nch != 0u);
        if (om) {
            if (t.nch) q[(tail + __popc(om & lt)) & qmask] = make_uint2(t.l0, t.nch);
            tail += __popc(om);
            if (8u * (tail - head) > (uint32_t)a.qcap) {  // more cells than the queue may hold?  count them
                __syncwarp();
                uint32_t live = 0;
                for (uint32_t e = head + lane; e < tail; e += 32) live += q[e & qmask].y;
                if (__reduce_add_sync(FULL, live) > (uint32_t)a.qcap) {
                    overflow = true;
                    break;
                }
            }
        }
        // accepted cells and opened leaves: entries of the list, in the cells' order
        const unsigned am = __ballot_sync(FULL, t.ok);
        const unsigned lm = __ballot_sync(FULL, t.mine != 0u) & ~am;
        if (!lm && list_n + 32u <= LIST_CAP) {
            if (t.ok) {
                float *e = lx + list_n + __popc(am & lt);
                e[0] = t.jp.x; e[LIST_CAP] = t.jp.y; e[2 * LIST_CAP] = t.jp.z; e[3 * LIST_CAP] = t.jp.w;
            }
            list_n += __popc(am);
        } else {
            const uint32_t incl = warp_incl_scan(t.mine);
            const uint32_t tot = __shfl_sync(FULL, incl, 31);
            // a window of the batch's entries at a time: what the list has room for
            for (uint32_t w0 = 0; w0 < tot;) {
                const uint32_t w1 = min(tot, w0 + (LIST_CAP - list_n));
                write_entries<PACK>(a, t, incl - t.mine, lm, lx, LIST_CAP, list_n - w0, w0, w1);
                list_n += w1 - w0;
                w0 = w1;
                if (w0 < tot) flush();
            }
        }
        if (list_n >= CHUNK) flush();
        __syncwarp();
    }
    if (!overflow) {
        flush();
        if (list_n) {  // the last, shorter chunk
            pad_list(lx, LIST_CAP, list_n);
            chunk(0, (list_n + 3) >> 2);
        }
    } else {
        if (lane == 0) gt_set_error(a.ctl, GT_EOVERFLOW, GTK_WALK);
        cp_async_wait_all();
        mem[64] = mem[96] = make_float4(NAN, NAN, NAN, NAN);
        list_n = chunks = 0;
    }
    __syncwarp();
    // the range is read again: held over the traversal it would cost registers
    group_range(a, g, ngroups, a0, a1);
    tests = __reduce_add_sync(FULL, tests);
    if (lane == 0) {
        stat[0] += ((unsigned long long)chunks * CHUNK + list_n) * (a1 - a0);
        stat[1] += tests;
    }
    const bool again = store_group<LEVELS, 32>(a, a0, a1, mem) && !overflow;
    __syncwarp();
    if (LEVELS && again) walk_group_ordered(a, g, ngroups, lx, q);
}

// The barrier of a team (a power of two of the block's warps).
__device__ __forceinline__ void team_sync(uint32_t team, uint32_t T) {
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1u), "r"(T * 32u) : "memory");
}

// One group by a team of T warps: every round tests up to 4 T queue entries, 4 per warp, and lists what they
// give in the order that one warp would (the queue is first in, first out, and entries and queue slots follow
// from scans over the team's warps); the team's warps sum different chunks, and their partial sums are added in
// the chunks' order.  So the result is the one warp's, bit for bit, whatever T is.  A queue that grows to
// where one warp may turn depth-first ends the attempt: false, and one warp walks the group.
// lx: T x WARP_SM words: four arrays of T LIST_CAP entries, the members and sums, T x 64 partial sums.
template <int MAC, bool LEVELS>
__device__ __forceinline__ bool team_group(const WalkArgs &a, uint32_t g, uint32_t ngroups, float *lx, uint2 *q,
                                           unsigned long long *stat, uint2 *counts, uint32_t team, uint32_t T) {
    const uint32_t lane = threadIdx.x & 31u, w = (threadIdx.x >> 5) & (T - 1u);
    const uint32_t qmask = gt_queue_ring(a.qcap) - 1u, cap = T * LIST_CAP;
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = lanemask_lt();
    float4 *mem = (float4 *)(lx + 4 * cap) + lane;
    float4 *part = mem + 128;  // of warp v: part[64 v], part[64 v + 32]
    uint32_t a0, a1;
    group_range(a, g, ngroups, a0, a1);
    const bool two = a1 - a0 > 32u;
    Pseudo ps;
    {   // every warp finds the same sphere; the first one's members are the team's
        float4 *own = w == 0 ? mem : part + 64 * (T - 2u) ;
        if (!group_setup<false, 32>(a, a0, a1 - a0, own, ps)) {
            if (w == 0 && lane == 0) gt_set_error(a.ctl, GT_EINVAL, GTK_WALK);
            return true;
        }
    }
    uint32_t list_n = 0, chunks = 0, tests = 0;
    // the list's full chunks (at the end: all of it), then the rest moved to its front
    auto flush = [&](bool last) {
        cp_async_wait_all();
        team_sync(team, T);
        const uint32_t full = list_n / CHUNK, todo = last ? (list_n + CHUNK - 1) / CHUNK : full;
        if (last && w == 0) pad_list(lx, cap, list_n);
        if (last) team_sync(team, T);
        for (uint32_t c0 = 0; c0 < todo; c0 += T) {
            const uint32_t c = c0 + w;
            if (c < todo) {
                const uint32_t k0 = c * (CHUNK / 4), k1 = c < full ? k0 + CHUNK / 4 : (list_n + 3) >> 2;
                part[64 * w] = chunk_force(lx, cap, mem[0], a.eps2, k0, k1);
                if (two) part[64 * w + 32] = chunk_force(lx, cap, mem[32], a.eps2, k0, k1);
            }
            team_sync(team, T);
            if (w == 0)
                for (uint32_t v = 0; v < min(T, todo - c0); v++) {
                    add_force(mem[64], part[64 * v]);
                    if (two) add_force(mem[96], part[64 * v + 32]);
                }
            if (c0 + T < todo) team_sync(team, T);
        }
        chunks += full;
        list_n -= full * CHUNK;
        if (!last) {
            if (full && w == T - 1u) move_rest(lx, cap, list_n, full * (CHUNK / 4));
            team_sync(team, T);
        }
    };
    uint32_t head = 0, tail = 1;
    if (w == 0 && lane == 0) q[0] = make_uint2(0u, 1u);
    team_sync(team, T);
    while (head != tail) {
        const uint32_t live = tail - head, nb = min(live, 4u * T), b0 = min(4u * w, nb);
        const Batch t = test_batch<MAC>(a, ps, take_four(q[(head + b0 + (lane >> 3)) & qmask], nb - b0), tests);
        head += nb;
        const unsigned om = __ballot_sync(FULL, t.nch != 0u), am = __ballot_sync(FULL, t.ok);
        const unsigned lm = __ballot_sync(FULL, t.mine != 0u) & ~am;
        const uint32_t incl = lm ? warp_incl_scan(t.mine) : (uint32_t)__popc(am & (lt | (1u << lane)));
        if (lane == 31) counts[w] = make_uint2(__popc(om), incl);
        team_sync(team, T);
        uint32_t push = 0, pushes = 0, first = 0, tot = 0;
        for (uint32_t v = 0; v < T; v++) {
            const uint2 c = counts[v];
            if (v == w) { push = pushes; first = tot; }
            pushes += c.x;
            tot += c.y;
        }
        if (8 * (int)(live + pushes) > a.qcap - LIFO_ROOM) {  // the same for every warp
            cp_async_wait_all();
            team_sync(team, T);
            return false;
        }
        if (t.nch) q[(tail + push + __popc(om & lt)) & qmask] = make_uint2(t.l0, t.nch);
        tail += pushes;
        const uint32_t excl = first + incl - t.mine;
        for (uint32_t w0 = 0; w0 < tot;) {
            const uint32_t w1 = min(tot, w0 + (cap - list_n));
            write_entries<false>(a, t, excl, lm, lx, cap, list_n - w0, w0, w1);
            list_n += w1 - w0;
            w0 = w1;
            if (w0 < tot) flush(false);
        }
        if (list_n >= T * CHUNK) flush(false);  // its last barrier ends the round
        else team_sync(team, T);
    }
    flush(true);
    tests = __reduce_add_sync(FULL, tests);
    group_range(a, g, ngroups, a0, a1);
    if (lane == 0) {
        if (w == 0) stat[0] += ((unsigned long long)chunks * CHUNK + list_n) * (a1 - a0);
        stat[1] += tests;
    }
    if (w == 0 && store_group<LEVELS, 32>(a, a0, a1, mem)) {
        __syncwarp();
        if (LEVELS) walk_group_ordered(a, g, ngroups, lx, q);
    }
    return true;
}

// Groups are taken one after another from a counter, by single warps or, when there are too few of them to
// keep the grid busy, by teams.  A team of T does a group in ~T / 1.2, T / 1.7, T / 2.7 (T = 2, 4, 8) of one
// warp's time (barriers, and batches that the first levels of the tree do not fill), so it pays where the
// longest groups, not their sum, set the time.  Whole calls in us with T = 1, 2, 4, 8 (3648 warps): 476 groups
// 704, 509, 399, 354; 4600 groups 370, 264, 214, 238; 6080 groups 412, 368, 365, 415; 11333 groups 272, 303,
// 380, 573; 115000 groups 2620, 3207, 4456, 7118.  (The 4600 would be faster by fours, and from 4600 to 6080 it makes no
// difference: the cut between fours and twos could lie higher.)
// FLAT: a team's batches are four entries of each warp, which on flat trees leaves half or more of its lanes idle, so
// teams end earlier.  Calls with T = 1, 2, 4, 8: lines, 373 groups 63, 78, 65, 56; 754 groups 70, 93, 69, 87; 1524 groups
// 76, 108, 113, -; sheets, 256 groups 62, 62, 50, 47; 1024 groups 75, 77, 68, -; 2386 groups 107, 113, 117, -.
// A queue that is depth-first from the start (qcap) has a team hand every group back to one warp, the others idle: no
// teams.  65536 particles of a Plummer sphere, 3618 groups, a queue of 4096: 162 with teams, 115 without.
__device__ __forceinline__ uint32_t team_of(bool flat, uint32_t ngroups, uint32_t warps, int qcap) {
    if (qcap <= LIFO_ROOM) return 1u;
    if (flat) return ngroups > warps / 3u ? 1u : (ngroups > warps / 8u ? 4u : 8u);
    return ngroups > 2u * warps ? 1u : (ngroups > warps ? 2u : (ngroups > warps / 4u ? 4u : 8u));
}

// groups of one system in a list of the systems' group counts: gprefix[s] is the first
// global group of system s, gprefix[nsys] the total
__device__ __forceinline__ int system_of(const uint32_t *gprefix, int nsys, uint32_t gg) {
    int lo = 0, hi = nsys - 1;  // the last s with gprefix[s] <= gg
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (gprefix[mid] <= gg) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// FLAT: for a system whose tree is flat; one of the two kernels walks it, the other ends at once.
template <int MAC, bool LEVELS, bool FLAT>
__global__ __launch_bounds__(WT, GT_WALK_MINB) void k_walk(const __grid_constant__ WalkArgs a) {
    gt_grid_ready();
    if ((a.ctl->flat != 0u) != FLAT) return;
    __shared__ __align__(16) float list_sm[NWARP][WARP_SM];
    __shared__ unsigned long long stat_sm[NWARP][2];
    __shared__ uint2 counts_sm[NWARP];
    __shared__ uint32_t g_sm[NWARP];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint32_t na = a.ctl->n_active;
    const uint32_t gmax = (uint32_t)a.gmax;
    const uint32_t ngroups = a.gstart ? a.ctl->n_groups : (na + gmax - 1) / gmax;
    const uint32_t T = team_of(FLAT, ngroups, gridDim.x * NWARP, a.qcap), team = warp / T, first = team * T;
    uint2 *q = (uint2 *)a.queue + (size_t)(blockIdx.x * NWARP + first) * gt_queue_ring(a.qcap);
    unsigned long long *stat = stat_sm[warp];
    if (lane < 2) stat[lane] = 0;
    __syncwarp();
    if (T == 1) {
        for (;;) {
            uint32_t g = 0;
            if (lane == 0) g = atomicAdd(&a.ctl->group_next, 1u);
            g = __shfl_sync(0xffffffffu, g, 0);
            if (g >= ngroups) break;
            walk_group<MAC, LEVELS, FLAT>(a, g, ngroups, list_sm[warp], q, stat);
        }
    } else {
        for (;;) {
            if (warp == first && lane == 0) g_sm[team] = atomicAdd(&a.ctl->group_next, 1u);
            team_sync(team, T);
            const uint32_t g = g_sm[team];
            if (g >= ngroups) break;
            if (!team_group<MAC, LEVELS>(a, g, ngroups, list_sm[first], q, stat, counts_sm + first, team, T) && warp == first)
                walk_group<MAC, LEVELS, FLAT>(a, g, ngroups, list_sm[first], q, stat);
            team_sync(team, T);
        }
    }
    __syncwarp();
    if (lane == 0) {
        if (stat[0]) atomicAdd(&a.ctl->interactions, stat[0]);
        if (stat[1]) atomicAdd(&a.ctl->mac_tests, stat[1]);
    }
}

// Many systems in one persistent launch: global group numbers run over the systems
// in order (gprefix), every warp or team takes the next one from one counter and walks it
// with that system's arguments (copied to shared memory).  mac >= 0 overrides every
// system's MAC (the opening-angle start-up pass).  FLAT: the groups of the systems whose trees are flat, or of the others
// (gprefix and group_next are this kind's).
template <int MAC, bool LEVELS, bool FLAT>
__global__ __launch_bounds__(WT, GT_WALK_MINB) void k_walk_batch(const WalkArgs *__restrict__ args, int nsys,
                                                                 const uint32_t *__restrict__ gprefix,
                                                                 unsigned int *group_next, uint32_t *queue, int qcap,
                                                                 int mac) {
    gt_grid_ready();
    __shared__ __align__(16) float list_sm[NWARP][WARP_SM];
    __shared__ WalkArgs sargs[NWARP];
    __shared__ unsigned long long stat_sm[NWARP][2];
    __shared__ uint2 counts_sm[NWARP];
    __shared__ uint32_t g_sm[NWARP];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint32_t total = gprefix[nsys];
    if (FLAT && !total) return;
    const uint32_t T = group_next[2], team = warp / T, first = team * T;  // (k_batch_prefix)
    uint2 *q = (uint2 *)queue + (size_t)(blockIdx.x * NWARP + first) * gt_queue_ring(qcap);
    unsigned long long *stat = stat_sm[warp];
    const WalkArgs &a = sargs[warp];
    // A warp's groups are in ascending order: it looks a system up, fetches its arguments and adds to its counters only
    // when the system changes (for every group: 64 systems of 2^12 to 2^18 particles 7225 us, now 7094).
    int sys = -1;
    uint32_t g0 = 0, g1 = 0;  // the system's first group and the next one's
    if (lane < 2) stat[lane] = 0;
    __syncwarp();
    auto count = [&]() {
        if (sys >= 0 && lane == 0) {
            if (stat[0]) atomicAdd(&a.ctl->interactions, stat[0]);
            if (stat[1]) atomicAdd(&a.ctl->mac_tests, stat[1]);
        }
        __syncwarp();
    };
    for (;;) {
        uint32_t gg = 0;
        if (T == 1) {
            if (lane == 0) gg = atomicAdd(group_next, 1u);
            gg = __shfl_sync(0xffffffffu, gg, 0);
        } else {
            if (warp == first && lane == 0) g_sm[team] = atomicAdd(group_next, 1u);
            team_sync(team, T);
            gg = g_sm[team];
        }
        if (gg >= total) break;
        if (gg >= g1) {
            count();
            if (lane == 0) sys = system_of(gprefix, nsys, gg);
            sys = __shfl_sync(0xffffffffu, sys, 0);
            g0 = gprefix[sys];
            g1 = gprefix[sys + 1];
            static_assert(sizeof(WalkArgs) % 4 == 0, "copied as words");
            const uint32_t *src = (const uint32_t *)&args[sys];
            uint32_t *dst = (uint32_t *)&sargs[warp];
            for (int w = lane; w < (int)(sizeof(WalkArgs) / 4); w += 32) dst[w] = src[w];
            if (lane < 2) stat[lane] = 0;
            __syncwarp();
            if (mac >= 0 && lane == 0) sargs[warp].mac = mac;
            __syncwarp();
        }
        // the batch queue replaces the system's own
        if (T == 1) {
            walk_group<MAC, LEVELS, FLAT>(a, gg - g0, g1 - g0, list_sm[warp], q, stat);
        } else {
            if (!team_group<MAC, LEVELS>(a, gg - g0, g1 - g0, list_sm[first], q, stat, counts_sm + first, team, T) &&
                warp == first)
                walk_group<MAC, LEVELS, FLAT>(a, gg - g0, g1 - g0, list_sm[first], q, stat);
            team_sync(team, T);
        }
    }
    __syncwarp();
    count();
}

// gprefix over the group counts of the systems whose trees aren't flat, and behind it over those of the others (a warp
// each; also resets the two counters and chooses the teams' sizes, behind them)
__global__ __launch_bounds__(64) void k_batch_prefix(DevCtl *const *__restrict__ ctls, const WalkArgs *__restrict__ args,
                                                     int nsys, uint32_t *gprefix, unsigned int *group_next,
                                                     uint32_t walk_warps) {
    gt_grid_ready();
    const int lane = threadIdx.x & 31, kind = threadIdx.x >> 5;
    gprefix += kind * (nsys + 1);
    uint32_t carry = 0;
    int qcap = INT_MAX;  // the smallest queue
    for (int s0 = 0; s0 < nsys; s0 += 32) {
        const int s = s0 + lane;
        uint32_t ng = 0;
        if (s < nsys) {
            const DevCtl *c = ctls[s];
            const uint32_t na = c->n_active;
            const uint32_t gm = (uint32_t)args[s].gmax;
            if ((c->flat != 0u) == (kind == 1)) ng = args[s].gstart ? c->n_groups : (na + gm - 1) / gm;
            if (ng) qcap = min(qcap, args[s].qcap);
        }
        const uint32_t incl = warp_incl_scan(ng);
        if (s < nsys) gprefix[s] = carry + incl - ng;
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    qcap = __reduce_min_sync(0xffffffffu, qcap);
    if (lane == 0) {
        gprefix[nsys] = carry;
        group_next[kind] = 0u;
        group_next[2 + kind] = team_of(kind == 1, carry, walk_warps, qcap);
    }
}

}  // namespace

int gt_walk_blocks(int nsm) {
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_walk<MAC_ANY, true, false>, WT, 0);
    if (per < 1) per = 1;
    return per * nsm;
}

int gt_walk_warps_per_block() { return NWARP; }

void gt_launch_walk(const WalkArgs &a, int nblocks, cudaStream_t st) {
    constexpr int ACC = GT_MAC_ACCELERATION;
    const bool acc = a.mac == ACC, levels = a.inv_c2 > 0.0f;
    auto launch = [&](auto kernel) { gt_launch(kernel, nblocks, WT, 0, st, a); };
    if (levels) launch(acc ? k_walk<ACC, true, false> : k_walk<MAC_ANY, true, false>);
    else launch(acc ? k_walk<ACC, false, false> : k_walk<MAC_ANY, false, false>);
    launch(levels ? k_walk<MAC_ANY, true, true> : k_walk<MAC_ANY, false, true>);
    gt_note_launches(2);
}

void gt_launch_walk_batch(DevCtl *const *ctls, const WalkArgs *args, int nsys, uint32_t *gprefix,
                          unsigned int *group_next, uint32_t *queue, int qcap, int mac, bool all_acc, bool levels,
                          int nblocks, cudaStream_t st) {
    if (nsys <= 0) return;
    { k_batch_prefix<<<1, 64, 0, st>>>(ctls, args, nsys, gprefix, group_next, (uint32_t)(nblocks * NWARP)); gt_note_launches(1); }
    constexpr int ACC = GT_MAC_ACCELERATION;
    const bool acc = all_acc && mac < 0;
    auto launch = [&](auto kernel, int kind) {
        gt_launch(kernel, nblocks, WT, 0, st, args, nsys, gprefix + kind * (nsys + 1), group_next + kind, queue, qcap, mac);
    };
    if (levels) launch(acc ? k_walk_batch<ACC, true, false> : k_walk_batch<MAC_ANY, true, false>, 0);
    else launch(acc ? k_walk_batch<ACC, false, false> : k_walk_batch<MAC_ANY, false, false>, 0);
    launch(levels ? k_walk_batch<MAC_ANY, true, true> : k_walk_batch<MAC_ANY, false, true>, 1);
    gt_note_launches(2);
}
