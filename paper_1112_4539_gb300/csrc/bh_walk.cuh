// bh_walk.cuh -- device code shared by the group-walk kernels (bh_walk.cu: one
// warp per group, warp pairs, TMA staging; bh_walk_team.cu: a block per group):
// the shared-memory staging of sources, the tile arithmetic on packed source
// pairs, the layout of a group's targets on a warp, and bounded mbarrier waits.
#pragma once

#include "bh_mlp.cuh"
#include "bh_wait.h"

namespace bh {

constexpr int kStackCap = 704;      // see the stack bound in bh_walk.cu (21 levels)
constexpr int kStackCapFlat = 336;  // the same bound for 10 levels (30-bit keys)
constexpr int kTile = 64;              // sources per tile (one Kahan-compensated addition per tile)
constexpr int kTilePairs = kTile / 2;  // a tile as even/odd source pairs
constexpr int kRing = 2 * kTile;       // sources per ring (two tiles), stored as even/odd pairs
// unroll factors of the per-tile pair loops (tuning constants, measured:
// larger factors overflow the instruction cache, as every T-slot variant of
// the loops is live at once across the SM's warps)
#ifndef BH_POINT_UNROLL
#define BH_POINT_UNROLL 4
#endif
#ifndef BH_POINT_UNROLL_LEARNED
#define BH_POINT_UNROLL_LEARNED 4
#endif
#ifndef BH_QUAD_UNROLL
#define BH_QUAD_UNROLL 2           // one-warp kernel (the paired and TMA kernels keep 1)
#endif
#ifndef BH_QUAD_UNROLL_LEARNED
#define BH_QUAD_UNROLL_LEARNED 1    // the learned walk (more registers for the network)
#endif
constexpr int kPointUnroll = BH_POINT_UNROLL;
constexpr int kPointUnrollLearned = BH_POINT_UNROLL_LEARNED;
constexpr int kPointUnrollPaired = 2;
constexpr int kQuadUnroll = BH_QUAD_UNROLL;
constexpr int kQuadUnrollLearned = BH_QUAD_UNROLL_LEARNED;
constexpr int kQuadUnrollPaired = 1;
constexpr int kQuadUnrollTma = 1;

// Quadrupole-pair unroll of the one-warp kernel: 2 up to 3 slots per lane;
// the 4-slot and learned kernels, with more registers live, keep 1.
template <int T, bool LEARNED>
__host__ __device__ constexpr int bh_quad_unroll() { return LEARNED ? kQuadUnrollLearned : (T <= 3 ? kQuadUnroll : 1); }

// Sources are staged negated and as pairs (ring positions 2p, 2p+1 side by
// side) so that the interaction arithmetic runs on packed f32x2 operations:
// one instruction computes the same step for two sources.
template <int CAP>
struct WarpSmemOf {
    float gbox[8];              // the group's box: xmin, ymin, zmin, radius, xmax, ymax, zmax, -
    unsigned long long tot[2];  // interactions so far: particle-particle, particle-cell
    uint32_t stack[CAP];        // (first node << 3) | (count - 1)
    uint32_t staging[32];
    int2 leafq[64];             // pending particle ranges (first, count)
    float4 ra[kRing / 2];       // point sources: (-x, -x', -y, -y')
    float4 rb[kRing / 2];       //                (-z, -z', -m, -m')
};
typedef WarpSmemOf<kStackCap> WarpSmem;
struct WarpQuad {               // quadrupole cells, pairs as above; Q = 3 I - T 1 (traceless), T = tr I
    float4 a[kRing / 2];        // (-x, -x', -y, -y')      centre of mass
    float4 b[kRing / 2];        // (-z, -z', -M, -M')
    float4 c[kRing / 2];        // (Qxx, Qxx', Qyy, Qyy')
    float4 d[kRing / 2];        // (Qzz, Qzz', Qxy, Qxy')
    float4 e[kRing / 2];        // (Qxz, Qxz', Qyz, Qyz')
    float4 f[kRing / 2];        // (-T eps^2, -T' eps^2, -, -)
};

__device__ __forceinline__ void bh_put_point(float4* ra, float4* rb, int r, float4 v)
{
    float* a = reinterpret_cast<float*>(&ra[r >> 1]) + (r & 1);
    float* b = reinterpret_cast<float*>(&rb[r >> 1]) + (r & 1);
    a[0] = -v.x; a[2] = -v.y;
    b[0] = -v.z; b[2] = -v.w;
}
template <int CAP>
__device__ __forceinline__ void bh_put_point(WarpSmemOf<CAP>& S, int r, float4 v)
{
    bh_put_point(S.ra, S.rb, r, v);
}
// cell with centre/mass cm and stored moments qb = (Ixx, Iyy, Izz, Ixy),
// qc = (Ixz, Iyz, 1.5 T, 0.5 T): staged as the traceless Q = 3 I - T 1 and
// -T eps^2 (see bh_pq2)
template <class QC>
__device__ __forceinline__ void bh_put_quad(QC& Q, int r, float4 cm, float4 qb, float4 qc, float eps2)
{
    const int p = r >> 1, h = r & 1;
    float* a = reinterpret_cast<float*>(&Q.a[p]) + h;
    float* b = reinterpret_cast<float*>(&Q.b[p]) + h;
    float* c = reinterpret_cast<float*>(&Q.c[p]) + h;
    float* d = reinterpret_cast<float*>(&Q.d[p]) + h;
    float* e = reinterpret_cast<float*>(&Q.e[p]) + h;
    float* f = reinterpret_cast<float*>(&Q.f[p]) + h;
    const float T = 2.0f * qc.w;  // exact
    a[0] = -cm.x; a[2] = -cm.y;
    b[0] = -cm.z; b[2] = -cm.w;
    c[0] = __fmaf_rn(3.0f, qb.x, -T); c[2] = __fmaf_rn(3.0f, qb.y, -T);
    d[0] = __fmaf_rn(3.0f, qb.z, -T); d[2] = 3.0f * qb.w;
    e[0] = 3.0f * qc.x; e[2] = 3.0f * qc.y;
    f[0] = -T * eps2;
}

struct WalkParams {
    const float4* pos_s;
    const uint32_t* perm;
    const int32_t* g_first;
    const int32_t* g_count;
    const int32_t* g_order;  // the groups by falling cost (nullptr: in their own order)
    const int4* rec;
    const float4* com_m;
    const float* seff;
    const float4* quad;
    float4* out;
    bh_dev_ctrl* ctrl;
    float eps2;
    // learned criterion
    const float4* mfeat;     // node-constant features
    const bh_mlp_dev* mlp;   // network (global copy)
    float theta_guard;       // theta of the S_eff in use (the guard)
    const float4* wrec;      // walk records (TMA-staged walk)
    int sm_count;
};

// Running totals of a lane's T targets with their Kahan compensations, the
// latter either in registers or in shared memory (this lane's column of a
// per-warp [4T][32] array: touched once per tile, they need no register).
#ifndef BH_KAHAN_SMEM
#define BH_KAHAN_SMEM 1
#endif
template <int T>
struct Acc {
    float x[T], y[T], z[T], p[T];
#if BH_KAHAN_SMEM
    float* kc;
    __device__ __forceinline__ float& c(int t, int k) { return kc[(4 * t + k) * 32]; }
#else
    float cc[4][T];
    __device__ __forceinline__ float& c(int t, int k) { return cc[k][t]; }
#endif
};
template <int T>
__host__ __device__ constexpr size_t bh_kahan_smem_bytes()
{
    return BH_KAHAN_SMEM ? (size_t)T * 4 * 32 * sizeof(float) : 0;
}

// Squared distance of a node's centre of mass from the group's box, as
// explicit round-to-nearest operations: every walk kernel takes the same
// opening decisions bit for bit (an expression left to the compiler may be
// contracted into FMAs differently in each kernel, which flips near ties).
__device__ __forceinline__ float bh_dist2(float dx, float dy, float dz)
{
    return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// Target layout of a group of gc particles on the warp's T slots per lane
// (warp-uniform).  Slots 0..nf-1 hold targets t*32 + lane.  When the last
// slot would hold at most kSplitMax targets (k = gc - 32*nf) it is "split":
// lane l holds target nf*32 + (l mod m), m = 2^lg >= k, and evaluates only
// the 2m sources of each tile in its phase (l / m); the phases' partial sums
// are added across lanes once, when the group ends.  A slot with 4 targets
// then costs 8 evaluations per tile instead of 64.
#ifndef BH_SPLIT_MAX
#define BH_SPLIT_MAX 16
#endif
constexpr int kSplitMax = BH_SPLIT_MAX;
struct Layout {
    int nf;      // full slots
    bool split;  // slot nf is split
    int lg;      // log2 of the targets per phase in the split slot
};

__device__ __forceinline__ void bh_kahan(float& s, float& c, float v)
{
    const float y = __fsub_rn(v, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
}

typedef float2 f2;
__device__ __forceinline__ f2 bh_add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 bh_mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 bh_fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 bh_rsqrt2(f2 a) { return make_float2(rsqrtf(a.x), rsqrtf(a.y)); }
// 1 / sqrt(a).  NORMAL: a is known to be no denormal, which saves rsqrtf's scaling.
template <bool NORMAL>
__device__ __forceinline__ float bh_rsqrt_of(float a)
{
    if (!NORMAL) return rsqrtf(a);
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ f2 bh_lo(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ f2 bh_hi(float4 v) { return make_float2(v.z, v.w); }

// Per-slot partial sums of one tile, two lanes of a pair each.
template <int T>
struct Part {
    f2 x[T], y[T], z[T], p[T], q[T];
};

// Adds the tile's pair sums of slots 0..TN-1 to the running totals.
template <int T, int TN, class AC>
__device__ __forceinline__ void bh_add_tile(AC& A, const Part<T>& P, bool with_q)
{
#pragma unroll
    for (int t = 0; t < TN; t++) {
        float pt = P.p[t].x + P.p[t].y;
        if (with_q) pt = fmaf(-0.5f, P.q[t].x + P.q[t].y, pt);
        bh_kahan(A.x[t], A.c(t, 0), P.x[t].x + P.x[t].y);
        bh_kahan(A.y[t], A.c(t, 1), P.y[t].x + P.y[t].y);
        bh_kahan(A.z[t], A.c(t, 2), P.z[t].x + P.z[t].y);
        bh_kahan(A.p[t], A.c(t, 3), pt);
    }
}

// A pair of point sources (negated, as staged) on one target held twice in
// (x, y, z); Eq. 1:  a += m (s - x_i) / r^3,  phi -= m / r.
__device__ __forceinline__ void bh_pp2(float4 sa, float4 sb, f2 eps2, f2 x, f2 y, f2 z, f2& ax, f2& ay, f2& az,
                                       f2& ap)
{
    const f2 dx = bh_add2(x, bh_lo(sa)), dy = bh_add2(y, bh_hi(sa)), dz = bh_add2(z, bh_lo(sb));  // x_i - s
    const f2 r2 = bh_fma2(dz, dz, bh_fma2(dy, dy, bh_fma2(dx, dx, eps2)));
    const f2 ri = bh_rsqrt2(r2);
    const f2 mr = bh_mul2(bh_hi(sb), ri);          // -m / r
    const f2 mr3 = bh_mul2(mr, bh_mul2(ri, ri));   // -m / r^3
    ax = bh_fma2(mr3, dx, ax);
    ay = bh_fma2(mr3, dy, ay);
    az = bh_fma2(mr3, dz, az);
    ap = bh_add2(ap, mr);
}

// A pair of quadrupole cells on one target.  With r = x_i - c, h^2 = r^2 +
// eps^2, g_n = h^-n, the traceless Q = 3 I - T 1, u = Q r and
// s = r.u - T eps^2, the second-order term of the softened kernel is
//   a   += g5 u + k r,   k = -M g3 - 2.5 g5 g2 s
//   phi += -M g1 - 0.5 s g5
// (the same as  a += 3 g5 I r + (1.5 T g5 - 7.5 q g7) r,
// phi -= 0.5 (3 q g5 - T g3) with q = r.I.r, since 3 q = r.Q.r + T r^2 and
// r^2 = h^2 - eps^2); the last term accumulated apart (aq) and scaled once
// per tile.  33 FP32 operations per source (21 FMA, 9 mul, 3 add).
__device__ __forceinline__ void bh_pq2(float4 ca, float4 cb, float4 cc, float4 cd, float4 ce, float4 cf, f2 eps2,
                                       f2 x, f2 y, f2 z, f2& ax, f2& ay, f2& az, f2& ap, f2& aq)
{
    const f2 rx = bh_add2(x, bh_lo(ca)), ry = bh_add2(y, bh_hi(ca)), rz = bh_add2(z, bh_lo(cb));
    const f2 h2 = bh_fma2(rz, rz, bh_fma2(ry, ry, bh_fma2(rx, rx, eps2)));
    const f2 g1 = bh_rsqrt2(h2);
    const f2 g2 = bh_mul2(g1, g1);
    const f2 g3 = bh_mul2(g1, g2);
    const f2 g5 = bh_mul2(g3, g2);
    const f2 mneg = bh_hi(cb);
    const f2 u0 = bh_fma2(bh_hi(cd), ry, bh_fma2(bh_lo(ce), rz, bh_mul2(bh_lo(cc), rx)));
    const f2 u1 = bh_fma2(bh_hi(cd), rx, bh_fma2(bh_hi(ce), rz, bh_mul2(bh_hi(cc), ry)));
    const f2 u2 = bh_fma2(bh_lo(ce), rx, bh_fma2(bh_hi(ce), ry, bh_mul2(bh_lo(cd), rz)));
    const f2 sq = bh_fma2(rx, u0, bh_fma2(ry, u1, bh_fma2(rz, u2, bh_lo(cf))));
    const f2 w = bh_mul2(bh_mul2(sq, make_float2(-2.5f, -2.5f)), g2);
    const f2 k = bh_fma2(g5, w, bh_mul2(mneg, g3));
    ax = bh_fma2(g5, u0, bh_fma2(k, rx, ax));
    ay = bh_fma2(g5, u1, bh_fma2(k, ry, ay));
    az = bh_fma2(g5, u2, bh_fma2(k, rz, az));
    ap = bh_fma2(mneg, g1, ap);
    aq = bh_fma2(sq, g5, aq);
}

// Targets of a lane: slot t holds (x, x), (y, y), (z, z).
template <int T>
struct Tgt {
    f2 x[T], y[T], z[T];
};

// One tile (np <= kTilePairs pairs) of point sources on the first NF slots of every lane,
// the pair loop unrolled PU times.
template <int T, int NF, int PU, class AC>
__device__ __forceinline__ void bh_eval_points(const float4* __restrict__ ra, const float4* __restrict__ rb,
                                               f2 eps2, const Tgt<T>& X, AC& A, int np)
{
    Part<T> P;
#pragma unroll
    for (int t = 0; t < NF; t++) P.x[t] = P.y[t] = P.z[t] = P.p[t] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int j0 = 0; j0 < np; j0 += PU) {
#pragma unroll
        for (int j = j0; j < j0 + PU; j++) {
            const float4 sa = ra[j], sb = rb[j];
#pragma unroll
            for (int t = 0; t < NF; t++)
                bh_pp2(sa, sb, eps2, X.x[t], X.y[t], X.z[t], P.x[t], P.y[t], P.z[t], P.p[t]);
        }
    }
    bh_add_tile<T, NF>(A, P, false);
}

// One tile (np <= kTilePairs pairs) of quadrupole cells on the first NF slots of every lane.
// QC: any staging with the six pair arrays a..f of WarpQuad (pairs p0..p0+15).
template <int T, int NF, class QC, int QU, class AC>
__device__ __forceinline__ void bh_eval_quads(const QC& Q, int p0, f2 eps2, const Tgt<T>& X, AC& A, int np)
{
    Part<T> P;
#pragma unroll
    for (int t = 0; t < NF; t++) P.x[t] = P.y[t] = P.z[t] = P.p[t] = P.q[t] = make_float2(0.f, 0.f);
#pragma unroll QU
    for (int j = p0; j < p0 + np; j++) {
        const float4 ca = Q.a[j], cb = Q.b[j], cc = Q.c[j], cd = Q.d[j], ce = Q.e[j], cf = Q.f[j];
#pragma unroll
        for (int t = 0; t < NF; t++)
            bh_pq2(ca, cb, cc, cd, ce, cf, eps2, X.x[t], X.y[t], X.z[t], P.x[t], P.y[t], P.z[t], P.p[t], P.q[t]);
    }
    bh_add_tile<T, NF>(A, P, true);
}

// The split slot: its target, and the m = 2^lg sources of the lane's phase
// (pairs from p; with m = 1 the pair holding the lane's source, one half kept).
template <int T>
__device__ __forceinline__ void bh_split_target(const Layout& L, const Tgt<T>& X, f2& x, f2& y, f2& z)
{
    x = X.x[0]; y = X.y[0]; z = X.z[0];
#pragma unroll
    for (int t = 1; t < T; t++)
        if (t == L.nf) { x = X.x[t]; y = X.y[t]; z = X.z[t]; }
}
// With kTilePairs = 32 pairs per tile and 32 / m phases, a phase (and each
// of its lanes) takes m whole pairs: pairs (l / m) * m .. + m - 1.
static_assert(kTilePairs == 32, "split phases assume 32 pairs per tile");
__device__ __forceinline__ float bh_split_sum(const Layout&, f2 v) { return v.x + v.y; }
template <int T, class AC>
__device__ __forceinline__ void bh_split_add(const Layout& L, AC& A, float ax, float ay, float az, float ap)
{
#pragma unroll
    for (int t = 0; t < T; t++)
        if (t == L.nf) {
            bh_kahan(A.x[t], A.c(t, 0), ax);
            bh_kahan(A.y[t], A.c(t, 1), ay);
            bh_kahan(A.z[t], A.c(t, 2), az);
            bh_kahan(A.p[t], A.c(t, 3), ap);
        }
}
template <int T, class AC>
__device__ __forceinline__ void bh_split_points(const Layout& L, const float4* __restrict__ ra,
                                                const float4* __restrict__ rb, f2 eps2, const Tgt<T>& X, AC& A)
{
    f2 x, y, z, ax = make_float2(0.f, 0.f), ay = ax, az = ax, ap = ax;
    bh_split_target<T>(L, X, x, y, z);
    const int p = ((threadIdx.x & 31) >> L.lg) << L.lg, np = 1 << L.lg;
    for (int i = p; i < p + np; i++) bh_pp2(ra[i], rb[i], eps2, x, y, z, ax, ay, az, ap);
    bh_split_add<T>(L, A, bh_split_sum(L, ax), bh_split_sum(L, ay), bh_split_sum(L, az), bh_split_sum(L, ap));
}
template <int T, class QC, class AC>
__device__ __forceinline__ void bh_split_quads(const Layout& L, const QC& Q, int p0, f2 eps2, const Tgt<T>& X,
                                               AC& A)
{
    f2 x, y, z, ax = make_float2(0.f, 0.f), ay = ax, az = ax, ap = ax, aq = ax;
    bh_split_target<T>(L, X, x, y, z);
    const int p = p0 + (((threadIdx.x & 31) >> L.lg) << L.lg), np = 1 << L.lg;
    for (int i = p; i < p + np; i++)
        bh_pq2(Q.a[i], Q.b[i], Q.c[i], Q.d[i], Q.e[i], Q.f[i], eps2, x, y, z, ax, ay, az, ap, aq);
    bh_split_add<T>(L, A, bh_split_sum(L, ax), bh_split_sum(L, ay), bh_split_sum(L, az),
                    fmaf(-0.5f, bh_split_sum(L, aq), bh_split_sum(L, ap)));
}

// Dispatch on the warp-uniform layout.  Every bh_eval_* instance is reached
// from one call site only (they are inlined: a second site would double the
// code of the hottest loop).
template <int T, int PU = kPointUnroll, class AC>
// A point tile; np: pairs evaluated on the full slots (kTilePairs, or fewer
// for a group's last, partly padded tile: the padding pairs add exact zeros),
// a multiple of PU.  The split slot always takes the whole tile.
__device__ __forceinline__ void bh_points(const Layout& L, const float4* __restrict__ ra,
                                          const float4* __restrict__ rb, f2 eps2, const Tgt<T>& X, AC& A,
                                          int np = kTilePairs)
{
    if (T > 1 && L.nf == 1) bh_eval_points<T, 1, PU>(ra, rb, eps2, X, A, np);
    else if (T > 2 && L.nf == 2) bh_eval_points<T, (T > 2 ? 2 : T), PU>(ra, rb, eps2, X, A, np);
    else if (T > 3 && L.nf == 3) bh_eval_points<T, (T > 3 ? 3 : T), PU>(ra, rb, eps2, X, A, np);
    else if (T > 4 && L.nf == 4) bh_eval_points<T, (T > 4 ? 4 : T), PU>(ra, rb, eps2, X, A, np);
    else if (L.nf > 0) bh_eval_points<T, T, PU>(ra, rb, eps2, X, A, np);
    if (L.split) bh_split_points<T>(L, ra, rb, eps2, X, A);
}
// A quadrupole tile (pairs p0 ..); np as for bh_points (any count); QU: the
// unroll factor of the pair loop.
template <int T, class QC, int QU = kQuadUnroll, class AC>
__device__ __forceinline__ void bh_quads(const Layout& L, const QC& Q, int p0, f2 eps2, const Tgt<T>& X,
                                         AC& A, int np = kTilePairs)
{
    if (T > 1 && L.nf == 1) bh_eval_quads<T, 1, QC, QU>(Q, p0, eps2, X, A, np);
    else if (T > 2 && L.nf == 2) bh_eval_quads<T, (T > 2 ? 2 : T), QC, QU>(Q, p0, eps2, X, A, np);
    else if (T > 3 && L.nf == 3) bh_eval_quads<T, (T > 3 ? 3 : T), QC, QU>(Q, p0, eps2, X, A, np);
    else if (T > 4 && L.nf == 4) bh_eval_quads<T, (T > 4 ? 4 : T), QC, QU>(Q, p0, eps2, X, A, np);
    else if (L.nf > 0) bh_eval_quads<T, T, QC, QU>(Q, p0, eps2, X, A, np);
    if (L.split) bh_split_quads<T, QC>(L, Q, p0, eps2, X, A);
}

// The group's own particles on its members, target itself masked.
// With a split slot, only its phase-0 lanes (lane < m) keep their sums: the
// other phases hold copies of the same targets.
template <int T, class AC>
__device__ __forceinline__ void bh_eval_self(int gc, const Layout& L, float eps2, const float (&xi)[T],
                                             const float (&yi)[T], const float (&zi)[T], const float (&mi)[T],
                                             AC& A)
{
    const int lane = threadIdx.x & 31;
    float tx[T], ty[T], tz[T], tp[T];
#pragma unroll
    for (int t = 0; t < T; t++) tx[t] = ty[t] = tz[t] = tp[t] = 0.0f;
#pragma unroll
    for (int t2 = 0; t2 < T; t2++) {
        for (int j = 0; j < 32; j++) {
            if (t2 * 32 + j >= gc) break;
            const float sx = __shfl_sync(BH_FULL_MASK, xi[t2], j);
            const float sy = __shfl_sync(BH_FULL_MASK, yi[t2], j);
            const float sz = __shfl_sync(BH_FULL_MASK, zi[t2], j);
            const float sm = __shfl_sync(BH_FULL_MASK, mi[t2], j);
#pragma unroll
            for (int t = 0; t < T; t++) {
                const bool self = (t == t2) && (lane == j);
                const float dx = sx - xi[t], dy = sy - yi[t], dz = sz - zi[t];
                float r2 = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, eps2)));
                r2 = self ? 1.0f : r2;
                const float ri = rsqrtf(r2);
                const float mr = __fmul_rn(self ? 0.0f : sm, ri);
                const float mr3 = __fmul_rn(__fmul_rn(mr, ri), ri);
                tx[t] = fmaf(mr3, dx, tx[t]);
                ty[t] = fmaf(mr3, dy, ty[t]);
                tz[t] = fmaf(mr3, dz, tz[t]);
                tp[t] = __fsub_rn(tp[t], mr);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < T; t++)
        if (L.split && t == L.nf && (lane >> L.lg) != 0) tx[t] = ty[t] = tz[t] = tp[t] = 0.0f;
#pragma unroll
    for (int t = 0; t < T; t++) {
        bh_kahan(A.x[t], A.c(t, 0), tx[t]);
        bh_kahan(A.y[t], A.c(t, 1), ty[t]);
        bh_kahan(A.z[t], A.c(t, 2), tz[t]);
        bh_kahan(A.p[t], A.c(t, 3), tp[t]);
    }
}

__device__ __forceinline__ float4 bh_pad_source() { return make_float4(1e18f, 1e18f, 1e18f, 0.0f); }

// The group box is read from shared memory at every batch of node tests
// rather than held in six registers across the walk: the tile loops of the
// three-slot kernel are at the register limit.  The load is explicit so that
// the compiler does not hoist it back into registers.
__device__ __forceinline__ float4 bh_lds4(const float* p)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(static_cast<unsigned int>(__cvta_generic_to_shared(p))));
    return v;
}

struct WsTile {  // kTile sources as pairs, laid out as WarpSmem (points: a, b) and WarpQuad (cells: a..f)
    float4 a[kTilePairs], b[kTilePairs], c[kTilePairs], d[kTilePairs], e[kTilePairs], f[kTilePairs];
};

// ------------------------------------------------------------ bounded mbarrier waits
__device__ __forceinline__ unsigned int bh_smem_addr(const void* p)
{
    return static_cast<unsigned int>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void bh_mbar_init(unsigned long long* b, unsigned int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bh_smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void bh_mbar_arrive(unsigned long long* b)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(bh_smem_addr(b))
                 : "memory");
}
__device__ __forceinline__ bool bh_mbar_try_wait(unsigned long long* b, unsigned int parity)
{
    unsigned int ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bh_smem_addr(b)), "r"(parity)
        : "memory");
    return ok != 0u;
}
// Wait for the phase of the given parity to complete.  False (with the error
// recorded) some polls after a second has passed (WaitLimit) or after
// kWsSpinLimit polls, whichever comes first; false at once when another warp
// has aborted.
__device__ __forceinline__ unsigned long long bh_globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool bh_mbar_wait(unsigned long long* b, unsigned int parity, bh_dev_ctrl* c)
{
    if (bh_mbar_try_wait(b, parity)) return true;
    WaitLimit lim(bh_globaltimer());
    for (int i = 0; i < lim.end; i++) {
        if (bh_mbar_try_wait(b, parity)) return true;
        if ((i & 63) == 63) {
            if (*(volatile unsigned int*)&c->abort) return false;
            lim.look(i, bh_globaltimer());
        }
    }
    bh_set_error(c, BH_ERR_DEVICE_TIMEOUT);
    return false;
}

// ------------------------------------------------------------ dealing ranges to lanes
// Lanes hold ranges (start, count) in lane order; lane l gets element l of
// their concatenation: the lane of its range is the rank of l among the bits
// that mark where the ranges begin.  Four to seven ballots, one reduction and one
// shuffle, where a shuffle scan and a staging array in shared memory took ten
// dependent shuffles and additions, up to eight stores and two barriers.

// Pop: up to 32 nodes from the top of a stack of sibling ranges (first << 3 |
// count - 1), sp > 0 entries.  Sets v to the lane's node (lanes below the
// returned count) and row to its range's place below the top, updates the
// stack in place.
__device__ __forceinline__ int bh_pop_nodes(uint32_t* stack, int& sp, unsigned int lt, int& v, int& row)
{
    const int lane = threadIdx.x & 31;
    const bool in = lane < sp;
    uint32_t e = 0u;
    if (in) e = stack[sp - 1 - lane];
    const unsigned int b0 = __ballot_sync(BH_FULL_MASK, e & 1u), b1 = __ballot_sync(BH_FULL_MASK, e & 2u),
                       b2 = __ballot_sync(BH_FULL_MASK, e & 4u);
    const int rows = min(sp, 32);
    const int c = (int)(e & 7u) + 1;
    const int excl = min(lane, rows) + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt);
    const int npop = min(rows + __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2), 32);
    const int st = (int)(e >> 3);
    const bool begins = in && excl < 32;
    const unsigned int marks = __reduce_or_sync(BH_FULL_MASK, begins ? 1u << (excl & 31) : 0u);
    const int nfull = __popc(__ballot_sync(BH_FULL_MASK, in && excl + c <= 32));
    row = __popc(marks & (lt | (1u << lane))) - 1;
    v = __shfl_sync(BH_FULL_MASK, st - excl, row) + lane;
    if (begins && lane == nfull) {  // taken in part: the rest stays
        const int take = 32 - excl;
        stack[sp - 1 - lane] = ((uint32_t)(st + take) << 3) | (uint32_t)(c - take - 1);
    }
    sp -= nfull;
    return npop;
}

// Up to 32 particles from the pending ranges q[pos ..] (n in all).  Returns
// how many, the lane's particle in k and its range's place after pos in row;
// advances pos, shortens the range that was taken in part.
__device__ __forceinline__ int bh_take_particles(int2* q, int& pos, int n, unsigned int lt, int& k, int& row)
{
    const int lane = threadIdx.x & 31;
    const bool in = pos + lane < n;
    int2 r = make_int2(0, 0);
    if (in) r = q[pos + lane];
    const unsigned int c = (unsigned int)min(r.y, 32);
    int excl = 0, total = 0;
#pragma unroll
    for (int b = 0; b < 6; b++) {
        const unsigned int m = __ballot_sync(BH_FULL_MASK, c & (1u << b));
        excl += __popc(m & lt) << b;
        total += __popc(m) << b;
    }
    const bool begins = in && excl < 32;
    const unsigned int marks = __reduce_or_sync(BH_FULL_MASK, begins ? 1u << (excl & 31) : 0u);
    const int nfull = __popc(__ballot_sync(BH_FULL_MASK, in && excl + r.y <= 32));
    row = __popc(marks & (lt | (1u << lane))) - 1;
    k = __shfl_sync(BH_FULL_MASK, r.x - excl, row) + lane;
    if (begins && lane == nfull) q[pos + lane] = make_int2(r.x + (32 - excl), r.y - (32 - excl));
    pos += nfull;
    return min(total, 32);
}

// A block of warps per group (bh_walk_team.cu), for few enough groups of at most
// kTeamMaxGroup targets: a BH_* code, or 1 when the set is not for it.
int launch_walk_team(const WalkParams& P, int order, int G, const WalkSet& set, int sm_count, cudaStream_t s);

}  // namespace bh
