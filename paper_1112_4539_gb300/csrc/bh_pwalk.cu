// bh_pwalk.cu -- the paper's own per-particle walk (Sec. 4.4, Fig. 5,
// Appendix A) on the device tree.
//
// Every node gets the two links of Fig. 5: "more" (its first child, the
// breadth-first child range's start) and "next" (the node that follows its
// subtree in depth-first order: the next sibling, else the parent's next).
// A particle's walk follows them without a stack: an accepted cell (Eq. 2,
// d^2 > S_eff with d = |x_i - COM|, the node not holding i) or a rejected leaf
// is applied and the walk goes on at next; a rejected internal node continues
// at more.  A node holding a single particle is a particle-particle term.
// bh_pwalk_kernel reaches the same nodes with the same decisions for every
// particle, 32 particles at a time (below); the links are still derived, for
// export.
//
// Accumulation: FP32 terms summed in tiles of 32, each tile added to the
// totals with Kahan compensation (as the group walk's tiles).  With
// BH_PWALK_UNSOFTENED_CELLS the particle-cell term uses eps = 0, as the
// Appendix A kernel does; particle-particle terms are always softened.
#include <algorithm>

#include "bh_walk.cuh"

namespace bh {

constexpr int kLinkDepthCap = 32;  // > the 22 levels of a 63-bit key tree

// parent of every node; roots (level 0, one per system) get -1
__global__ void bh_parent_kernel(const int4* __restrict__ rec, int32_t* __restrict__ parent,
                                 const bh_dev_ctrl* __restrict__ c)
{
    bh_let_next_start();
    bh_after_previous(rec, parent, c);
    const int nn = (int)c->n_nodes, n_roots = (int)c->level_offset[1];
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nn; v += gridDim.x * blockDim.x) {
        const int4 r = rec[v];
        if (v < n_roots) parent[v] = -1;
        for (int k = 0; k < r.w; k++) parent[r.z + k] = v;
    }
}

// next link: climb while the node is its parent's last child
__global__ void bh_next_kernel(const int4* __restrict__ rec, const int32_t* __restrict__ parent,
                               int32_t* __restrict__ next, bh_dev_ctrl* __restrict__ c)
{
    bh_let_next_start();
    bh_after_previous(rec, parent, next, c);
    const int nn = (int)c->n_nodes;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nn; v += gridDim.x * blockDim.x) {
        int u = v, nx = -1, d = 0;
        for (; d < kLinkDepthCap; d++) {
            const int p = parent[u];
            if (p < 0) break;
            const int4 rp = rec[p];
            if (u < rp.z + rp.w - 1) {
                nx = u + 1;
                break;
            }
            u = p;
        }
        if (d == kLinkDepthCap) bh_set_error(c, BH_ERR_CAPACITY);
        next[v] = nx;
    }
}

struct PWalkParams {
    const float* soft_h;     // individual softening: eps_i^2 / 2 per particle (key order)
    const float* soft_hbar;  //   and the mass-weighted mean of it per node
    bool soft_cells;         //   cells softened (not BH_PWALK_UNSOFTENED_CELLS)
    const float4* pos_s;
    const uint32_t* perm;
    const int4* rec;
    const float4* com_m;
    const float* seff;
    const float4* quad;
    float4* out;
    bh_dev_ctrl* ctrl;
    int n;
    float eps2;   // particle-particle softening
    float eps2c;  // particle-cell softening (0 when unsoftened)
};

// ------------------------------------------------------------ walk
// One warp walks for 32 particles that are neighbours in key order, lane i
// holding the i-th.  A stack entry is a range of siblings with the mask of the
// particles that reach it.  Nodes are tested 32 at a time, one per lane,
// against the particles' bounding box: farther than S_eff from the whole box,
// every particle accepts; nearer than S_eff to its farthest corner, every one
// rejects; only in between do the lanes test their own particles.  The box
// tests use the operations of the particle's test on distances that bound its
// own, and rounding keeps order, so each particle's list is exactly the one
// that its own walk gives.  Sources carry the mask of the particles they
// apply to (bits cleared by setting 1/r to zero) and are evaluated in tiles.
//
// Bound by the FP32 pipe in the tile loops; about two thirds of the evaluated
// lanes hold a particle that the source applies to.  A thread per particle,
// walking by the links, was bound by its chain of dependent node loads and by
// divergence (7% of the FP32 peak).  One launch on GB300, a thread per particle
// -> this kernel, the same interaction counts: Plummer 2^20 quadrupole theta
// 0.554 15.26 -> 4.63 ms (139 -> 460 Ginteractions/s), clumpy 2^20 14.39 ->
// 3.99 ms, clumpy 262147 with individual softening 5.00 -> 1.16 ms, uniform
// 20000 438 -> 119 us, Plummer 3000 952 -> 125 us.  Tiles of 32 with 5 blocks per
// SM against tiles of 64 with 4 (Plummer 2^20): 4.63 and 4.72 ms; 4 and 6
// blocks with tiles of 32: 4.76 and 4.69 ms.
constexpr int kPTile = 32;  // sources per tile (one Kahan-compensated addition each)
constexpr int kPRing = 2 * kPTile;
constexpr int kPThreads = 128;

template <int ORDER, bool IND>
struct PSmem {
    int2 leafq[32];         // pending leaves: first, count
    uint32_t leafm[32];     //   and the particles that opened them
    float4 nodes[32];       // nodes between the box tests: centre of mass, S_eff
    int2 range[32];         //   first particle, end
    float4 pa[kPRing / 2], pb[kPRing / 2], pc[kPRing / 2];  // points: (-x, -x', -y, -y') (-z, -z', -m, -m') (softening, softening', mask, mask')
    float4 ca[kPRing / 2], cb[kPRing / 2], cf[kPRing / 2];  // cells, as the points
    float4 cc[ORDER >= 2 ? kPRing / 2 : 1], cd[ORDER >= 2 ? kPRing / 2 : 1], ce[ORDER >= 2 ? kPRing / 2 : 1];  // quadrupole, as WarpQuad
    float2 ct[ORDER >= 2 ? kPRing / 2 : 1];  // (-T, -T') (IND) or (-T eps^2, ...)
};

// Sums of one particle: totals with Kahan compensations.
struct PAcc {
    float x, y, z, p, cx, cy, cz, cp;
};

// 1 / sqrt(a) of the lanes whose bit is set in the masks (as float bits), else 0.
template <bool NORMAL>
__device__ __forceinline__ f2 bh_rsqrt_masked(f2 a, f2 mask, unsigned int bit)
{
    const float u = bh_rsqrt_of<NORMAL>(a.x), v = bh_rsqrt_of<NORMAL>(a.y);
    return make_float2((__float_as_uint(mask.x) & bit) ? u : 0.0f, (__float_as_uint(mask.y) & bit) ? v : 0.0f);
}

// Pairs [p0, p0 + np) of point sources (or monopole cells) on the lane's
// particle; arithmetic as bh_pp2 with the pair's own softening.
template <bool IND, bool NORMAL>
__device__ __forceinline__ void bh_p_points(const float4* __restrict__ a, const float4* __restrict__ b,
                                            const float4* __restrict__ c, int p0, int np, f2 h, unsigned int bit, f2 x,
                                            f2 y, f2 z, PAcc& A)
{
    f2 ax = make_float2(0.f, 0.f), ay = ax, az = ax, ap = ax;
#pragma unroll 4
    for (int j = p0; j < p0 + np; j++) {
        const float4 sa = a[j], sb = b[j], sc = c[j];
        const f2 dx = bh_add2(x, bh_lo(sa)), dy = bh_add2(y, bh_hi(sa)), dz = bh_add2(z, bh_lo(sb));
        const f2 e2 = IND ? bh_add2(h, bh_lo(sc)) : bh_lo(sc);
        const f2 r2 = bh_fma2(dz, dz, bh_fma2(dy, dy, bh_fma2(dx, dx, e2)));
        const f2 ri = bh_rsqrt_masked<NORMAL>(r2, bh_hi(sc), bit);
        const f2 mr = bh_mul2(bh_hi(sb), ri);
        const f2 mr3 = bh_mul2(mr, bh_mul2(ri, ri));
        ax = bh_fma2(mr3, dx, ax);
        ay = bh_fma2(mr3, dy, ay);
        az = bh_fma2(mr3, dz, az);
        ap = bh_add2(ap, mr);
    }
    bh_kahan(A.x, A.cx, ax.x + ax.y);
    bh_kahan(A.y, A.cy, ay.x + ay.y);
    bh_kahan(A.z, A.cz, az.x + az.y);
    bh_kahan(A.p, A.cp, ap.x + ap.y);
}

// Pairs of quadrupole cells; arithmetic as bh_pq2.
template <bool IND, bool NORMAL, class S>
__device__ __forceinline__ void bh_p_quads(const S& Q, int p0, int np, f2 h, float eps2c, unsigned int bit, f2 x, f2 y,
                                           f2 z, PAcc& A)
{
    f2 ax = make_float2(0.f, 0.f), ay = ax, az = ax, ap = ax, aq = ax;
#pragma unroll 2
    for (int j = p0; j < p0 + np; j++) {
        const float4 ca = Q.ca[j], cb = Q.cb[j], cc = Q.cc[j], cd = Q.cd[j], ce = Q.ce[j], cf = Q.cf[j];
        const float2 ct = Q.ct[j];
        const f2 rx = bh_add2(x, bh_lo(ca)), ry = bh_add2(y, bh_hi(ca)), rz = bh_add2(z, bh_lo(cb));
        const f2 e2 = IND ? bh_add2(h, bh_lo(cf)) : make_float2(eps2c, eps2c);
        const f2 te = IND ? bh_mul2(ct, e2) : ct;
        const f2 h2 = bh_fma2(rz, rz, bh_fma2(ry, ry, bh_fma2(rx, rx, e2)));
        const f2 g1 = bh_rsqrt_masked<NORMAL>(h2, bh_hi(cf), bit);
        const f2 g2 = bh_mul2(g1, g1);
        const f2 g3 = bh_mul2(g1, g2);
        const f2 g5 = bh_mul2(g3, g2);
        const f2 mneg = bh_hi(cb);
        const f2 u0 = bh_fma2(bh_hi(cd), ry, bh_fma2(bh_lo(ce), rz, bh_mul2(bh_lo(cc), rx)));
        const f2 u1 = bh_fma2(bh_hi(cd), rx, bh_fma2(bh_hi(ce), rz, bh_mul2(bh_hi(cc), ry)));
        const f2 u2 = bh_fma2(bh_lo(ce), rx, bh_fma2(bh_hi(ce), ry, bh_mul2(bh_lo(cd), rz)));
        const f2 sq = bh_fma2(rx, u0, bh_fma2(ry, u1, bh_fma2(rz, u2, te)));
        const f2 w = bh_mul2(bh_mul2(sq, make_float2(-2.5f, -2.5f)), g2);
        const f2 k = bh_fma2(g5, w, bh_mul2(mneg, g3));
        ax = bh_fma2(g5, u0, bh_fma2(k, rx, ax));
        ay = bh_fma2(g5, u1, bh_fma2(k, ry, ay));
        az = bh_fma2(g5, u2, bh_fma2(k, rz, az));
        ap = bh_fma2(mneg, g1, ap);
        aq = bh_fma2(sq, g5, aq);
    }
    bh_kahan(A.x, A.cx, ax.x + ax.y);
    bh_kahan(A.y, A.cy, ay.x + ay.y);
    bh_kahan(A.z, A.cz, az.x + az.y);
    bh_kahan(A.p, A.cp, fmaf(-0.5f, aq.x + aq.y, ap.x + ap.y));
}

// Store source v (softening e, mask m) as ring entry r.
__device__ __forceinline__ void bh_p_put(float4* a, float4* b, float4* c, int r, float4 v, float e, uint32_t m)
{
    bh_put_point(a, b, r, v);
    float* f = reinterpret_cast<float*>(&c[r >> 1]) + (r & 1);
    f[0] = e;
    f[2] = __uint_as_float(m);
}

// IND: individual softening (symmetrized): a particle term softens with
// h_i + h_j, a cell term with h_i + hbar_c (h = eps^2 / 2), instead of eps^2.
// NORMAL: every softened distance is at least eps^2, a normal number.
template <int ORDER, bool IND, bool NORMAL>
__global__ void __launch_bounds__(kPThreads, 5) bh_pwalk_kernel(PWalkParams P, int stack_cap)
{
    bh_let_next_start();
    bh_after_previous();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef PSmem<ORDER, IND> Smem;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    Smem& S = reinterpret_cast<Smem*>(smem_raw)[wib];
    uint32_t* stack = reinterpret_cast<uint32_t*>(smem_raw + (kPThreads / 32) * sizeof(Smem)) + wib * 2 * stack_cap;
    uint32_t* smask = stack + stack_cap;
    bh_dev_ctrl* ctrl = P.ctrl;
    const unsigned int lt = bh_lanemask_lt(), bit = 1u << lane;
    const int nchunk = (P.n + 31) / 32;
    unsigned long long cnt_pp = 0ull, cnt_pc = 0ull;
    for (;;) {
        int g = 0;
        if (lane == 0) g = (int)atomicAdd(&ctrl->group_ctr, 1u);
        g = __shfl_sync(BH_FULL_MASK, g, 0);
        if (g >= nchunk) break;
        const int gb = g * 32, ge = min(gb + 32, P.n);
        const int i = min(gb + lane, P.n - 1);  // lanes past the end: the last particle, in no mask
        const float4 xi = P.pos_s[i];
        const float hi = IND ? P.soft_h[i] : 0.0f;
        const float bx0 = bh_ord2f(__reduce_min_sync(BH_FULL_MASK, bh_f2ord(xi.x)));
        const float by0 = bh_ord2f(__reduce_min_sync(BH_FULL_MASK, bh_f2ord(xi.y)));
        const float bz0 = bh_ord2f(__reduce_min_sync(BH_FULL_MASK, bh_f2ord(xi.z)));
        const float bx1 = bh_ord2f(__reduce_max_sync(BH_FULL_MASK, bh_f2ord(xi.x)));
        const float by1 = bh_ord2f(__reduce_max_sync(BH_FULL_MASK, bh_f2ord(xi.y)));
        const float bz1 = bh_ord2f(__reduce_max_sync(BH_FULL_MASK, bh_f2ord(xi.z)));
        const f2 x = make_float2(xi.x, xi.x), y = make_float2(xi.y, xi.y), z = make_float2(xi.z, xi.z);
        const f2 hp = make_float2(hi, hi);
        const float hcs = P.soft_cells ? hi : 0.0f;
        const f2 hc = make_float2(hcs, hcs);
        PAcc A;
        A.x = A.y = A.z = A.p = A.cx = A.cy = A.cz = A.cp = 0.0f;
        int sp = 1, p_head = 0, p_cnt = 0, c_head = 0, c_cnt = 0;
        if (lane == 0) {
            stack[0] = 0u;
            smask[0] = ge - gb == 32 ? BH_FULL_MASK : (1u << (ge - gb)) - 1u;
        }
        __syncwarp();
        bool overflow = false;
        while (sp > 0) {
            // ---- pop the top 32 nodes with their masks
            int v, row;
            const int top = sp;
            const int npop = bh_pop_nodes(stack, sp, lt, v, row);
            const bool has = lane < npop;
            const uint32_t M = has ? smask[top - 1 - row] : 0u;
            float4 cm = make_float4(0.f, 0.f, 0.f, 0.f);
            float se = 0.f;
            int4 r = make_int4(0, 1, -1, 0);
            if (has) {
                cm = P.com_m[v];
                se = P.seff[v];
                r = P.rec[v];
            }
            // ---- who accepts: the box tests, then the lanes' own where they leave it open
            const bool cell = has && r.y > 1;  // a node of one particle is a particle term
            const float qx = cm.x - bx0, qy = cm.y - by0, qz = cm.z - bz0;
            const float wx = bx1 - cm.x, wy = by1 - cm.y, wz = bz1 - cm.z;
            const float near2 = bh_dist2(fmaxf(fmaxf(-qx, -wx), 0.0f), fmaxf(fmaxf(-qy, -wy), 0.0f), fmaxf(fmaxf(-qz, -wz), 0.0f));
            const float far2 = bh_dist2(fmaxf(fabsf(qx), fabsf(wx)), fmaxf(fabsf(qy), fabsf(wy)), fmaxf(fabsf(qz), fabsf(wz)));
            const int re = r.x + r.y;
            const bool holds = r.x < ge && re > gb;  // a particle of the chunk
            const bool all = cell && near2 > se && !holds;
            const bool open = cell && !all && !(far2 <= se);
            uint32_t acc = all ? M : 0u;
            const unsigned int om = __ballot_sync(BH_FULL_MASK, open);
            if (om) {
                const int at = __popc(om & lt), no = __popc(om);
                if (open) {
                    S.nodes[at] = make_float4(cm.x, cm.y, cm.z, se);
                    S.range[at] = make_int2(r.x, re);
                }
                __syncwarp();
                uint32_t mine = 0u;
#pragma unroll 2
                for (int k = 0; k < no; k++) {
                    const float4 q = S.nodes[k];
                    const int2 h = S.range[k];
                    const float d2 = bh_dist2(q.x - xi.x, q.y - xi.y, q.z - xi.z);
                    const unsigned int yes = __ballot_sync(BH_FULL_MASK, d2 > q.w && !(h.x <= i && i < h.y));
                    if (at == k) mine = yes;
                }
                if (open) acc = M & mine;
                __syncwarp();
            }
            const uint32_t rej = M & ~acc;
            // ---- open: push child ranges with the particles that rejected
            const bool opn = cell && rej != 0u && r.z >= 0;
            const unsigned int pm = __ballot_sync(BH_FULL_MASK, opn);
            if (sp + __popc(pm) > stack_cap) {
                overflow = true;
                break;
            }
            if (opn) {
                const int at = sp + __popc(pm & lt);
                stack[at] = ((uint32_t)r.z << 3) | (uint32_t)(r.w - 1);
                smask[at] = rej;
            }
            sp += __popc(pm);
            // ---- accept: cell sources
            const unsigned int am = __ballot_sync(BH_FULL_MASK, acc != 0u);
            if (acc != 0u) {
                cnt_pc += (unsigned long long)__popc(acc);
                const int s = (c_head + c_cnt + __popc(am & lt)) & (kPRing - 1);
                const float e = IND ? (P.soft_cells ? P.soft_hbar[v] : 0.0f) : P.eps2c;
                bh_p_put(S.ca, S.cb, S.cf, s, cm, e, acc);
                if (ORDER >= 2) {
                    const float4 qb = P.quad[2 * (size_t)v], qc = P.quad[2 * (size_t)v + 1];
                    const int p = s >> 1, o = s & 1;
                    float* c = reinterpret_cast<float*>(&S.cc[p]) + o;
                    float* d = reinterpret_cast<float*>(&S.cd[p]) + o;
                    float* f = reinterpret_cast<float*>(&S.ce[p]) + o;
                    const float T = 2.0f * qc.w;  // exact
                    c[0] = __fmaf_rn(3.0f, qb.x, -T); c[2] = __fmaf_rn(3.0f, qb.y, -T);
                    d[0] = __fmaf_rn(3.0f, qb.z, -T); d[2] = 3.0f * qb.w;
                    f[0] = 3.0f * qc.x; f[2] = 3.0f * qc.y;
                    reinterpret_cast<float*>(&S.ct[p])[o] = IND ? -T : -T * P.eps2c;
                }
            }
            c_cnt += __popc(am);
            // ---- rejected leaves: their particles
            const bool leaf = has && rej != 0u && r.z < 0;
            const unsigned int lm = __ballot_sync(BH_FULL_MASK, leaf);
            const int lq_n = __popc(lm);
            if (leaf) {
                const int at = __popc(lm & lt);
                S.leafq[at] = make_int2(r.x, r.y);
                S.leafm[at] = rej;
                // terms: each opener with each particle but itself
                const int o0 = max(r.x, gb) - gb, o1 = min(re, ge) - gb;
                const uint32_t own = o1 > o0 ? (BH_FULL_MASK >> (32 - (o1 - o0))) << o0 : 0u;
                cnt_pp += (unsigned long long)__popc(rej) * (unsigned long long)r.y - (unsigned long long)__popc(rej & own);
            }
            __syncwarp();
            // ---- drain
            while (c_cnt >= kPTile) {
                if (ORDER >= 2) bh_p_quads<IND, NORMAL>(S, c_head >> 1, kPTile / 2, hc, P.eps2c, bit, x, y, z, A);
                else bh_p_points<IND, NORMAL>(S.ca, S.cb, S.cf, c_head >> 1, kPTile / 2, hc, bit, x, y, z, A);
                c_head ^= kPTile;
                c_cnt -= kPTile;
            }
            int lq_pos = 0;
            for (;;) {
                if (p_cnt >= kPTile) {
                    bh_p_points<IND, NORMAL>(S.pa, S.pb, S.pc, p_head >> 1, kPTile / 2, hp, bit, x, y, z, A);
                    p_head ^= kPTile;
                    p_cnt -= kPTile;
                    continue;
                }
                if (lq_pos >= lq_n) break;
                int k, at;
                const int q0 = lq_pos;
                const int nfill = bh_take_particles(S.leafq, lq_pos, lq_n, lt, k, at);
                if (lane < nfill) {
                    uint32_t m = S.leafm[q0 + at];
                    if (k >= gb && k < ge) m &= ~(1u << (k - gb));  // not on itself
                    bh_p_put(S.pa, S.pb, S.pc, (p_head + p_cnt + lane) & (kPRing - 1), P.pos_s[k],
                             IND ? P.soft_h[k] : P.eps2, m);
                }
                p_cnt += nfill;
                __syncwarp();
            }
        }
        if (overflow) {
            if (lane == 0) bh_set_error(ctrl, BH_ERR_CAPACITY);
            break;
        }
        // ---- the partial tiles, filled up with sources that apply to no lane
        if (c_cnt > 0) {
            for (int k = lane; k < kPTile; k += 32)
                if (k >= c_cnt) {
                    const int s = c_head + k, p = s >> 1, o = s & 1;
                    bh_p_put(S.ca, S.cb, S.cf, s, bh_pad_source(), 0.0f, 0u);
                    if (ORDER >= 2) {
                        float* c = reinterpret_cast<float*>(&S.cc[p]) + o;
                        float* d = reinterpret_cast<float*>(&S.cd[p]) + o;
                        float* f = reinterpret_cast<float*>(&S.ce[p]) + o;
                        c[0] = c[2] = d[0] = d[2] = f[0] = f[2] = 0.0f;
                        reinterpret_cast<float*>(&S.ct[p])[o] = 0.0f;
                    }
                }
            __syncwarp();
            if (ORDER >= 2) bh_p_quads<IND, NORMAL>(S, c_head >> 1, (c_cnt + 1) >> 1, hc, P.eps2c, bit, x, y, z, A);
            else bh_p_points<IND, NORMAL>(S.ca, S.cb, S.cf, c_head >> 1, (c_cnt + 1) >> 1, hc, bit, x, y, z, A);
        }
        if (p_cnt > 0) {
            for (int k = lane; k < kPTile; k += 32)
                if (k >= p_cnt) bh_p_put(S.pa, S.pb, S.pc, p_head + k, bh_pad_source(), 0.0f, 0u);
            __syncwarp();
            bh_p_points<IND, NORMAL>(S.pa, S.pb, S.pc, p_head >> 1, (p_cnt + 1) >> 1, hp, bit, x, y, z, A);
        }
        __syncwarp();
        if (gb + lane < ge) P.out[P.perm[i]] = make_float4(A.x - A.cx, A.y - A.cy, A.z - A.cz, A.p - A.cp);
    }
    // interaction counters: one atomic per warp
    for (int o = 16; o > 0; o >>= 1) {
        cnt_pp += __shfl_down_sync(BH_FULL_MASK, cnt_pp, o);
        cnt_pc += __shfl_down_sync(BH_FULL_MASK, cnt_pc, o);
    }
    if (lane == 0) {
        atomicAdd(&ctrl->n_pp, cnt_pp);
        atomicAdd(&ctrl->n_pc, cnt_pc);
        atomicAdd(&ctrl->cum_pp, cnt_pp);
        atomicAdd(&ctrl->cum_pc, cnt_pc);
    }
}

__global__ void bh_pwalk_reset_kernel(bh_dev_ctrl* c)
{
    bh_let_next_start();
    bh_after_previous();
    c->group_ctr = 0u;
    c->n_pp = 0ull;
    c->n_pc = 0ull;
}

// Individual softening, step 1: h = eps^2 / 2 of every particle in key order
// (a negative or non-finite length is reported as BH_ERR_NONFINITE).
__global__ void __launch_bounds__(256) bh_soft_gather_kernel(const float* __restrict__ eps,
                                                             const uint32_t* __restrict__ perm, int n,
                                                             float* __restrict__ h, bh_dev_ctrl* c)
{
    bh_let_next_start();
    bh_after_previous(eps, perm, h);
    bool bad = false;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const float e = eps[perm[k]];
        bad |= !(e >= 0.0f && isfinite(e));
        h[k] = 0.5f * (e * e);
    }
    if (__any_sync(BH_FULL_MASK, bad) && (threadIdx.x & 31) == 0) atomicCAS(&c->status, 0u, (unsigned int)(-BH_ERR_NONFINITE));
}

// Step 2, one level (deepest first): per node the FP64 sums (sum m, sum m h)
// over its particles (leaves) or its children, and hbar = sum m h / sum m.
__global__ void __launch_bounds__(256) bh_soft_level_kernel(const float4* __restrict__ pos_s,
                                                            const float* __restrict__ h, bh_nodes nd, int lev,
                                                            double2* __restrict__ sums, float* __restrict__ hbar,
                                                            const bh_dev_ctrl* __restrict__ c)
{
    bh_let_next_start();
    bh_after_previous(pos_s, h, sums, hbar, c);
    if (c->n_nodes == 0u) return;
    const int v0 = (int)c->level_offset[lev], v1 = (int)c->level_offset[lev + 1];
    for (int v = v0 + blockIdx.x * blockDim.x + threadIdx.x; v < v1; v += gridDim.x * blockDim.x) {
        const int4 r = nd.rec[v];
        double sm = 0.0, se = 0.0;
        if (r.z < 0) {
            for (int j = r.x; j < r.x + r.y; j++) {
                const double m = pos_s[j].w;
                sm += m;
                se += m * (double)h[j];
            }
        } else {
            for (int k = 0; k < r.w; k++) {
                const double2 t = sums[r.z + k];
                sm += t.x;
                se += t.y;
            }
        }
        sums[v] = make_double2(sm, se);
        hbar[v] = sm != 0.0 ? (float)(se / sm) : 0.0f;
    }
}

void launch_softening(const float* eps, const uint32_t* perm, const float4* pos_s, const bh_nodes& nd, int n,
                      bool deep, const bh_soft& soft, bh_dev_ctrl* ctrl, int grid, cudaStream_t s)
{
    bh_launch_after(bh_soft_gather_kernel, grid, 256, 0, s, eps, perm, n, soft.h, ctrl);
    for (int lev = deep ? BH_MAX_LEVEL_DEEP : BH_MAX_LEVEL; lev >= 0; lev--)
        bh_launch_after(bh_soft_level_kernel, grid, 256, 0, s, pos_s, soft.h, nd, lev, soft.sums, soft.hbar, ctrl);
}

// persistent warps, as many blocks per SM as registers and shared memory allow;
// the stack holds at most 33 ranges per level (as the group walk's)
template <int ORDER, bool IND, bool NORMAL>
static int bh_pwalk_launch(const PWalkParams& P, bool deep, int sm_count, cudaStream_t s)
{
    const int cap = 33 * (deep ? BH_MAX_LEVEL_DEEP : BH_MAX_LEVEL) + 2;
    const size_t smem = (kPThreads / 32) * (sizeof(PSmem<ORDER, IND>) + 2 * cap * sizeof(uint32_t));
    auto kern = bh_pwalk_kernel<ORDER, IND, NORMAL>;
    int bps = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, kPThreads, smem) != cudaSuccess || bps < 1)
        return BH_ERR_CUDA;
    const int warps = (P.n + 31) / 32, blocks = (warps + kPThreads / 32 - 1) / (kPThreads / 32);
    bh_launch_after(kern, std::min(blocks, sm_count * bps), kPThreads, smem, s, P, cap);
    return BH_OK;
}

int launch_pwalk(const float4* pos_s, const uint32_t* perm, const bh_nodes& nd, int32_t* parent, int32_t* next,
                 int order, bool deep, int n, int node_cap, float eps, bool unsoftened_cells, float4* out, bh_dev_ctrl* ctrl,
                 int sm_count, cudaStream_t s, const bh_soft* soft)
{
    const int link_grid = std::max(1, std::min((node_cap + 255) / 256, sm_count * 16));
    bh_launch_after(bh_parent_kernel, link_grid, 256, 0, s, nd.rec, parent, ctrl);
    bh_launch_after(bh_next_kernel, link_grid, 256, 0, s, nd.rec, parent, next, ctrl);
    bh_launch_after(bh_pwalk_reset_kernel, 1, 1, 0, s, ctrl);
    PWalkParams P;
    P.pos_s = pos_s;
    P.perm = perm;
    P.rec = nd.rec;
    P.com_m = nd.com_m;
    P.seff = nd.seff;
    P.quad = nd.quad;
    P.out = out;
    P.ctrl = ctrl;
    P.n = n;
    P.eps2 = eps * eps;
    P.eps2c = unsoftened_cells ? 0.0f : eps * eps;
    P.soft_h = soft ? soft->h : nullptr;
    P.soft_hbar = soft ? soft->hbar : nullptr;
    P.soft_cells = !unsoftened_cells;
    // without individual softening every softened distance is at least the
    // smaller eps^2: a normal number needs no scaling before its square root
    const bool normal = !soft && std::min(P.eps2, P.eps2c) >= 1.17549435e-38f;
    if (soft) return order >= 2 ? bh_pwalk_launch<2, true, false>(P, deep, sm_count, s)
                                : bh_pwalk_launch<1, true, false>(P, deep, sm_count, s);
    if (normal) return order >= 2 ? bh_pwalk_launch<2, false, true>(P, deep, sm_count, s)
                                  : bh_pwalk_launch<1, false, true>(P, deep, sm_count, s);
    return order >= 2 ? bh_pwalk_launch<2, false, false>(P, deep, sm_count, s)
                      : bh_pwalk_launch<1, false, false>(P, deep, sm_count, s);
}

}  // namespace bh
