// bh_sph.cu -- neighbour search and SPH density: the short-range application
// of the general tree walk (Sec. 4.3, Fig. 4).
//
// Fig. 4's walk calls distance_test on each cell and, for a neighbour search,
// skips a cell that lies farther than the search radius (its proc_cell does
// nothing) and descends otherwise; proc_particle tests one pair.  Here, as in
// the gravity walk, one warp walks the tree for a whole group of up to 32*T
// particles: a node is skipped when its particles' bounding box lies farther
// than the group's largest radius from the group's bounding box (with a
// 1e-5 relative allowance, so FP32 rounding of the box gap can never skip a
// neighbour), a leaf is taken when its box is also within reach of at least one
// target of the warp (each with its own radius), other nodes are opened.  The
// particles of a taken leaf that lie within the largest radius of the group's
// box become candidates; they go through a 64-entry ring in shared memory, as
// pairs, and are tested 32 at a time against each lane's T targets.
//
// Bound by instruction issue: about 6 candidates are tested per neighbour found,
// and some lane has a hit at nearly every one.  Against the form that took
// every particle of a leaf, one at a time, with a test for the target itself
// (GB300, build and search, Plummer, 64 neighbours): 2^20, G = 32 1.42 -> 1.08 ms
// (510 -> 395 M candidate pairs), 2^20, G = 64 1.61 -> 1.24 ms, 2^24, G = 32
// 28.1 -> 15.8 ms (21.9 -> 8.1 G pairs).
//
// Pair rule (identical to the oracle's): d = x_j - x_i per axis in FP32,
// r2 = fma(dz, dz, fma(dy, dy, dx * dx)), j != i is a neighbour iff
// r2 < h_i * h_i.  Density rho_i = sum over i and its neighbours of
// m_j W(sqrt(r2), h_i) with the cubic spline of support h (Monaghan &
// Lattanzio 1985), FP32.
#include <algorithm>

#include "bh_walk.cuh"

namespace bh {

constexpr int kSphStackCap = kStackCap;  // ranges of <= 8 siblings; same bound as the gravity walk
#ifndef BH_SPH_TEAM_STACK
#define BH_SPH_TEAM_STACK kSphStackCap   // smaller only to see a block of warps report an overflow
#endif
constexpr int kSphRing = 64;             // candidates per ring (two tiles of 32)

struct SphParams {
    const float4* pos_s;
    const uint32_t* perm;
    const int32_t* g_first;
    const int32_t* g_count;
    const int4* rec;
    const float4* blo;
    const float4* bhi;
    const float* h;      // per particle, caller order (nullptr: h_const)
    float h_const;
    int32_t* count;      // caller order (nullptr: not written)
    float* rho;          // caller order (nullptr: not written)
    bh_dev_ctrl* ctrl;
    int32_t* heavy;      // groups left to the second launch (tile_ctr[0] of them)
    int max_level;
};

// What a group at large costs: candidates at the density of its box, n at most,
// added up over 1024 groups spread over the list (whole numbers, so that the sum
// is the same in any order).  Groups of few particles say little about their density.
constexpr int kSphSamples = 1024;
constexpr int kSphSampleLevel = 6;  // (the deepest is 10 or 21)
__device__ __forceinline__ void bh_sph_sample(const SphParams& P, int n)
{
    const int lane = threadIdx.x & 31, ng = (int)P.ctrl->n_groups;
    if (ng <= kSphSamples) return;
    for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < kSphSamples; w += (gridDim.x * blockDim.x) >> 5) {
        const int g = (int)((long long)ng * w / kSphSamples), gb = P.g_first[g], gc = P.g_count[g];
        if (gc < 8) continue;
        float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY}, h = 0.0f;
        for (int o = lane; o < gc; o += 32) {
            const float4 q = P.pos_s[gb + o];
            h = fmaxf(h, P.h ? P.h[P.perm[gb + o]] : P.h_const);
            lo[0] = fminf(lo[0], q.x); lo[1] = fminf(lo[1], q.y); lo[2] = fminf(lo[2], q.z);
            hi[0] = fmaxf(hi[0], q.x); hi[1] = fmaxf(hi[1], q.y); hi[2] = fmaxf(hi[2], q.z);
        }
        h = bh_ord2f(__reduce_max_sync(BH_FULL_MASK, bh_f2ord(h)));
        float side = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; k++)
            side = fmaxf(side, bh_ord2f(__reduce_max_sync(BH_FULL_MASK, bh_f2ord(hi[k]))) -
                                   bh_ord2f(__reduce_min_sync(BH_FULL_MASK, bh_f2ord(lo[k]))));
        const float r = 1.0f + 2.0f * h / side;
        if (lane == 0) {
            atomicAdd(&P.ctrl->sph_like, (unsigned long long)fminf((float)gc * (r * r * r), (float)n));
            atomicAdd(&P.ctrl->sph_samples, 1u);
        }
    }
}

// ------------------------------------------------------------ node boxes
// Tight bounding box of every node's particles, bottom-up by level: a leaf
// scans its particles, an internal node combines its children (one level
// deeper, already done).  Min/max are exact.  The first launch clears the search's
// counters; that of a level with many nodes samples the groups beside them.
__global__ void __launch_bounds__(256)
bh_node_box_kernel(const float4* __restrict__ pos_s, const int4* __restrict__ rec, float4* __restrict__ lo,
                   float4* __restrict__ hi, int lev, SphParams P, int n)
{
    bh_let_next_start();
    bh_after_previous(pos_s, rec, lo, hi);
    bh_dev_ctrl* c = P.ctrl;
    if (lev == P.max_level && blockIdx.x == 0 && threadIdx.x == 0) {  // the search's counters
        c->group_ctr = 0u;
        c->tile_ctr[0] = 0u;  // groups listed as heavy (the sort's tickets are free after the build)
        c->tile_ctr[1] = 0u;  // and taken
        c->sph_like = 0ull;
        c->sph_samples = 0u;
        c->n_pp = 0ull;
        c->n_pc = 0ull;
    }
    const int v0 = (int)c->level_offset[lev], v1 = (int)c->level_offset[lev + 1];
    for (int v = v0 + blockIdx.x * blockDim.x + threadIdx.x; v < v1; v += gridDim.x * blockDim.x) {
        const int4 r = rec[v];
        float4 a = make_float4(INFINITY, INFINITY, INFINITY, 0.f), b = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
        // loads in batches: the pass waits for little else
        if (r.z < 0) {
            for (int k = 0; k < r.y; k += 8) {
                float4 p[8];
#pragma unroll
                for (int u = 0; u < 8; u++) p[u] = pos_s[r.x + min(k + u, r.y - 1)];  // (repeats change no bound)
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    a.x = fminf(a.x, p[u].x); a.y = fminf(a.y, p[u].y); a.z = fminf(a.z, p[u].z);
                    b.x = fmaxf(b.x, p[u].x); b.y = fmaxf(b.y, p[u].y); b.z = fmaxf(b.z, p[u].z);
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < 8; k += 4) {
                float4 l[4], h[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    l[u] = lo[r.z + min(k + u, r.w - 1)];
                    h[u] = hi[r.z + min(k + u, r.w - 1)];
                }
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    a.x = fminf(a.x, l[u].x); a.y = fminf(a.y, l[u].y); a.z = fminf(a.z, l[u].z);
                    b.x = fmaxf(b.x, h[u].x); b.y = fmaxf(b.y, h[u].y); b.z = fmaxf(b.z, h[u].z);
                }
            }
        }
        lo[v] = a;
        hi[v] = b;
    }
    if (lev == kSphSampleLevel) bh_sph_sample(P, n);
}

// ------------------------------------------------------------ walk
struct SphSmem {
    uint32_t stack[kSphStackCap];
    int2 leafq[32];
    float4 blo[32], bhi[32];                      // boxes of the pop's near leaves
    float4 ra[kSphRing / 2], rb[kSphRing / 2];    // candidates as pairs: (x, x', y, y') (z, z', m, m')
};

// cubic spline with support h (normalised to unit integral), FP32
__device__ __forceinline__ float bh_w3(float r, float hinv, float c)
{
    const float q = r * hinv;
    const float u = 1.0f - q;
    const float inner = fmaf(6.0f * q * q, q - 1.0f, 1.0f);  // 1 - 6 q^2 + 6 q^3
    return c * (q <= 0.5f ? inner : (q <= 1.0f ? 2.0f * u * u * u : 0.0f));
}

// np pairs of candidates against the lane's targets; (nx, ny, nz): minus the
// target, held twice.  The target itself is among the candidates once, at r2 =
// 0 (the caller starts its count at -1); one without a finite place has no pair,
// not even its own, and its count of -1 is written as 0.
template <int T>
__device__ __forceinline__ void bh_sph_tile(const float4* __restrict__ ra, const float4* __restrict__ rb, int np,
                                            const f2 (&nx)[T], const f2 (&ny)[T], const f2 (&nz)[T],
                                            const float (&h2)[T], const float (&hinv)[T], const float (&cw)[T], int tn,
                                            int (&cnt)[T], float (&rho)[T])
{
#pragma unroll 4
    for (int j = 0; j < np; j++) {
        const float4 sa = ra[j], sb = rb[j];
#pragma unroll
        for (int t = 0; t < T; t++) {
            if (t < tn) {
                const f2 dx = bh_add2(bh_lo(sa), nx[t]), dy = bh_add2(bh_hi(sa), ny[t]), dz = bh_add2(bh_lo(sb), nz[t]);
                const f2 r2 = bh_fma2(dz, dz, bh_fma2(dy, dy, bh_mul2(dx, dx)));
                if (r2.x < h2[t]) {
                    cnt[t]++;
                    rho[t] = fmaf(sb.z, bh_w3(sqrtf(r2.x), hinv[t], cw[t]), rho[t]);
                }
                if (r2.y < h2[t]) {
                    cnt[t]++;
                    rho[t] = fmaf(sb.w, bh_w3(sqrtf(r2.y), hinv[t], cw[t]), rho[t]);
                }
            }
        }
    }
}

// NW = 1: a warp per group, which gives up a group after `most` candidates or one
// batch of nodes per 16 of them and lists it.  NW > 1: a block of NW warps per
// listed group, which share its subtrees; their counts and densities are added
// in warp order.  A group's work varies with its radii (in a Plummer sphere's
// outskirts the radius that holds 64 neighbours reaches into the core), and the
// few long ones were the whole tail of the launch.
//
// A listed group is walked again from the start, so the limit must leave alone
// what is no exception.  While every warp has a group at most, idle warps are
// plenty and it is kSphHeavy; with more groups it is at least twice what a
// group at large costs (bh_sph_sample), and a quarter of a warp's share.  All of
// this is the same on every run, and so are the densities' bits.  The block's
// warps share the subtrees of about half the search radius: from one level
// (4) on a dense knot's neighbourhood was a single subtree, of one warp.
// ms, a warp per group | 1024 throughout, level 4 | this: clumpy 2^20, 500
// neighbours, G = 32 6.96 | 17.1 | 5.4, 32 neighbours 2.01 | 3.21 | 1.75;
// uniform 2^20, 500, G = 64 3.80 | 5.29 | 3.05; Plummer 250000, 32, G = 64 10.5 | 2.16 |
// 2.17.
//
// GB300, build and search, a warp per group throughout -> this (the same counts):
// Plummer 131072, G = 32 1.56 -> 0.77 ms, 4000 particles 580 -> 477 us, 2^20
// unchanged.  Limits of 32 / 64 / 128 batches: 2^20 1.17 / 1.09 / 1.09 ms, 131072
// 0.72 / 0.77 / 0.90 ms; of 512 / 1024 / 2048 candidates at 2^20 1.17 / 1.10 / 1.10.
constexpr int kSphHeavy = 1024;
constexpr int kSphPops = 64;
constexpr int kSphSplit = 4;  // the least level whose subtrees are shared out
template <int T>
constexpr int bh_sph_team() { return T <= 3 ? 8 : 4; }  // (shared memory)
template <int T, int NW>
__global__ void __launch_bounds__(NW == 1 ? 128 : NW * 32) bh_sph_kernel(SphParams P)
{
    bh_let_next_start();
    bh_after_previous();
    __shared__ SphSmem smem[NW == 1 ? 4 : NW];
    __shared__ int s_group;
    __shared__ volatile int s_most;  // NW = 1: candidates after which a group is given up (volatile: in no register)
    __shared__ float s_rho[NW == 1 ? 1 : NW * T * 32];
    __shared__ int s_cnt[NW == 1 ? 1 : NW * T * 32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    SphSmem& S = smem[wib];
    const unsigned int lt = bh_lanemask_lt();
    bh_dev_ctrl* ctrl = P.ctrl;
    const int ng = (int)ctrl->n_groups;
    const int n_roots = (int)ctrl->level_offset[1];
    unsigned long long tested = 0ull;
    if (NW == 1) {
        if (threadIdx.x == 0) {
            const float load = (float)ng / (4.0f * (float)gridDim.x);  // groups per warp
            float most = (float)kSphHeavy;
            if (load > 1.0f && ctrl->sph_samples)
                most = fmaxf(most, fmaxf(2.0f, 0.25f * load) * ((float)ctrl->sph_like / (float)ctrl->sph_samples));
            s_most = (int)fminf(most, 1e9f);
        }
        __syncthreads();
    }

    for (;;) {
        int g = 0;
        if (NW == 1) {
            if (lane == 0) {
                g = (int)atomicAdd(&ctrl->group_ctr, 1u);
                if (*(volatile unsigned int*)&ctrl->abort) g = ng;
            }
            g = __shfl_sync(BH_FULL_MASK, g, 0);
            if (g >= ng) break;
        } else {
            __syncthreads();  // the last group's sums have been read
            if (threadIdx.x == 0) {
                const unsigned int k = atomicAdd(&ctrl->tile_ctr[1], 1u);
                s_group = (k < ctrl->tile_ctr[0] && !*(volatile unsigned int*)&ctrl->abort) ? P.heavy[k] : -1;
            }
            __syncthreads();
            g = s_group;
            if (g < 0) break;
        }
        const int gb = P.g_first[g], gc = P.g_count[g];
        const int tn = (gc + 31) >> 5;

        float xi[T], yi[T], zi[T], h2[T], hinv[T], cw[T], rho[T];
        f2 nx[T], ny[T], nz[T];
        int cnt[T];
        float bx0 = INFINITY, by0 = INFINITY, bz0 = INFINITY, bx1 = -INFINITY, by1 = -INFINITY, bz1 = -INFINITY;
        float hmax = 0.0f;
        bool bad = false;
#pragma unroll
        for (int t = 0; t < T; t++) {
            const int o = t * 32 + lane;
            float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
            float h = 1.0f;
            if (o < gc) {
                q = P.pos_s[gb + o];
                h = P.h ? P.h[P.perm[gb + o]] : P.h_const;
                bad = bad || !(h > 0.0f && h < INFINITY);
                bx0 = fminf(bx0, q.x); by0 = fminf(by0, q.y); bz0 = fminf(bz0, q.z);
                bx1 = fmaxf(bx1, q.x); by1 = fmaxf(by1, q.y); bz1 = fmaxf(bz1, q.z);
                hmax = fmaxf(hmax, h);
            }
            xi[t] = q.x; yi[t] = q.y; zi[t] = q.z;
            h2[t] = __fmul_rn(h, h);
            hinv[t] = 1.0f / h;
            cw[t] = 8.0f / (3.14159265358979f * h * h * h);
            nx[t] = make_float2(-q.x, -q.x); ny[t] = make_float2(-q.y, -q.y); nz[t] = make_float2(-q.z, -q.z);
            // the target's own pair has r2 = 0, below h^2 unless that underflows
            const bool own = h2[t] > 0.0f, first = NW == 1 || wib == 0;
            cnt[t] = own && first ? -1 : 0;
            rho[t] = own || !first ? 0.0f : q.w * bh_w3(0.0f, hinv[t], cw[t]);
        }
        if (__any_sync(BH_FULL_MASK, bad)) {
            if (lane == 0) bh_set_error(ctrl, BH_ERR_NONFINITE);
            break;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            bx0 = fminf(bx0, __shfl_xor_sync(BH_FULL_MASK, bx0, o));
            by0 = fminf(by0, __shfl_xor_sync(BH_FULL_MASK, by0, o));
            bz0 = fminf(bz0, __shfl_xor_sync(BH_FULL_MASK, bz0, o));
            bx1 = fmaxf(bx1, __shfl_xor_sync(BH_FULL_MASK, bx1, o));
            by1 = fmaxf(by1, __shfl_xor_sync(BH_FULL_MASK, by1, o));
            bz1 = fmaxf(bz1, __shfl_xor_sync(BH_FULL_MASK, bz1, o));
            hmax = fmaxf(hmax, __shfl_xor_sync(BH_FULL_MASK, hmax, o));
        }
        const float reach2 = hmax * hmax * (1.0f + 1e-5f);
        // each target's own reach for the leaf filter (-1: no target in the slot)
        float reach_t[T];
#pragma unroll
        for (int t = 0; t < T; t++) reach_t[t] = (t * 32 + lane < gc) ? h2[t] * (1.0f + 1e-5f) : -1.0f;

        // root of the group's system
        int root = 0;
        for (int hi = n_roots; hi - root > 1;) {
            const int mid = (root + hi) >> 1;
            if (P.rec[mid].x <= gb) root = mid;
            else hi = mid;
        }
        // NW > 1: the first node and the end of the level whose subtrees are shared out
        int split = 0, below = 0;
        if (NW > 1) {
            const int lev = ilogbf(fminf(fmaxf(ctrl->box[3] / hmax, 1.0f), 1e9f)) + 1;
            split = (int)ctrl->level_offset[max(kSphSplit, min(lev, P.max_level))];
            below = (int)ctrl->level_offset[max(kSphSplit, min(lev, P.max_level)) + 1];
        }
        int sp = 1, ring_head = 0, ring_cnt = 0, pops = 0, taken = 0;
        if (lane == 0) S.stack[0] = (uint32_t)root << 3;
        __syncwarp();
        bool overflow = false, heavy = false;
        while (sp > 0) {
            if (NW == 1 && max(taken, kSphHeavy / kSphPops * pops++) >= s_most) {
                heavy = true;
                break;
            }
            // pop the top 32 nodes
            int v, row;
            const int npop = bh_pop_nodes(S.stack, sp, lt, v, row);
            const bool has = lane < npop;
            __syncwarp();

            // distance_test: the node's box against the group's box
            int4 r = make_int4(0, 0, -1, 0);
            bool near = false;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (has) {
                r = P.rec[v];
                a = P.blo[v];
                b = P.bhi[v];
                const float gx = fmaxf(fmaxf(a.x - bx1, bx0 - b.x), 0.0f);
                const float gy = fmaxf(fmaxf(a.y - by1, by0 - b.y), 0.0f);
                const float gz = fmaxf(fmaxf(a.z - bz1, bz0 - b.z), 0.0f);
                near = gx * gx + gy * gy + gz * gz <= reach2;
            }
            // a block's warps walk the top of the tree alike and share out its
            // leaves and the subtrees from the split level down by node index
            if (NW > 1 && v < below && (v >= split || r.z < 0)) near = near && v % NW == wib;
            bool leaf = near && r.z < 0;
            const bool opn = near && r.z >= 0;
            // per-target filter: a leaf near the group's box is kept only when
            // its box lies within reach of at least one target of the warp
            {
                const unsigned int lm0 = __ballot_sync(BH_FULL_MASK, leaf);
                const int at = __popc(lm0 & lt), nl = __popc(lm0);
                if (leaf) {
                    S.blo[at] = a;
                    S.bhi[at] = b;
                }
                __syncwarp();
                unsigned int keep = 0u;  // by place in the list
                for (int q = 0; q < nl; q++) {
                    const float4 l = S.blo[q], u = S.bhi[q];
                    bool hit = false;
#pragma unroll
                    for (int t = 0; t < T; t++) {
                        const float dx = fmaxf(fmaxf(l.x - xi[t], xi[t] - u.x), 0.0f);
                        const float dy = fmaxf(fmaxf(l.y - yi[t], yi[t] - u.y), 0.0f);
                        const float dz = fmaxf(fmaxf(l.z - zi[t], zi[t] - u.z), 0.0f);
                        hit = hit || (dx * dx + dy * dy + dz * dz <= reach_t[t]);
                    }
                    if (__any_sync(BH_FULL_MASK, hit)) keep |= 1u << q;
                }
                leaf = leaf && ((keep >> at) & 1u);
            }
            const unsigned int om = __ballot_sync(BH_FULL_MASK, opn);
            if (sp + __popc(om) > (NW == 1 ? kSphStackCap : BH_SPH_TEAM_STACK)) {
                overflow = true;
                break;
            }
            if (opn) S.stack[sp + __popc(om & lt)] = ((uint32_t)r.z << 3) | (uint32_t)(r.w - 1);
            sp += __popc(om);

            // leaves: their particle ranges become candidates
            const unsigned int lm = __ballot_sync(BH_FULL_MASK, leaf);
            const int lq_n = __popc(lm);
            if (leaf) S.leafq[__popc(lm & lt)] = make_int2(r.x, r.y);
            __syncwarp();
            int lq_pos = 0;
            for (;;) {
                if (ring_cnt >= 32) {
                    bh_sph_tile<T>(S.ra + (ring_head >> 1), S.rb + (ring_head >> 1), 16, nx, ny, nz, h2, hinv, cw, tn,
                                   cnt, rho);
                    taken += 32;
                    ring_head ^= 32;
                    ring_cnt -= 32;
                    __syncwarp();
                    continue;
                }
                if (lq_pos >= lq_n) break;
                // candidates: the leaves' particles within the largest radius of the group's box
                int k;
                const int nfill = bh_take_particles(S.leafq, lq_pos, lq_n, lt, k, row);
                bool in = false;
                float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
                if (lane < nfill) {
                    p = P.pos_s[k];
                    const float gx = fmaxf(fmaxf(p.x - bx1, bx0 - p.x), 0.0f);
                    const float gy = fmaxf(fmaxf(p.y - by1, by0 - p.y), 0.0f);
                    const float gz = fmaxf(fmaxf(p.z - bz1, bz0 - p.z), 0.0f);
                    in = gx * gx + gy * gy + gz * gz <= reach2;
                }
                const unsigned int im = __ballot_sync(BH_FULL_MASK, in);
                if (in) {
                    const int slot = (ring_head + ring_cnt + __popc(im & lt)) & (kSphRing - 1);
                    float* fa = reinterpret_cast<float*>(&S.ra[slot >> 1]) + (slot & 1);
                    float* fb = reinterpret_cast<float*>(&S.rb[slot >> 1]) + (slot & 1);
                    fa[0] = p.x; fa[2] = p.y;
                    fb[0] = p.z; fb[2] = p.w;
                }
                ring_cnt += __popc(im);
                __syncwarp();
            }
        }
        // (a block's warps leave together, at the next group, which thread 0 does
        // not take once the error is set: if it left here, the others would find
        // its last group for ever)
        if (overflow) {
            if (lane == 0) bh_set_error(ctrl, BH_ERR_CAPACITY);
            if (NW == 1) break;
        }
        if (heavy) {
            if (lane == 0) P.heavy[atomicAdd(&ctrl->tile_ctr[0], 1u)] = g;
            continue;
        }
        if (ring_cnt > 0) {
            // an odd last candidate gets a far one beside it, which is nobody's neighbour
            if (lane == 0 && (ring_cnt & 1)) {
                const int slot = ring_head + ring_cnt;
                float* fa = reinterpret_cast<float*>(&S.ra[slot >> 1]) + 1;
                float* fb = reinterpret_cast<float*>(&S.rb[slot >> 1]) + 1;
                fa[0] = fa[2] = fb[0] = INFINITY;
                fb[2] = 0.0f;
            }
            __syncwarp();
            bh_sph_tile<T>(S.ra + (ring_head >> 1), S.rb + (ring_head >> 1), (ring_cnt + 1) >> 1, nx, ny, nz, h2, hinv,
                           cw, tn, cnt, rho);
            taken += ring_cnt;
        }
        tested += (unsigned long long)taken * (unsigned long long)gc;
        __syncwarp();
        if (NW > 1) {
#pragma unroll
            for (int t = 0; t < T; t++) {
                s_cnt[(wib * T + t) * 32 + lane] = cnt[t];
                s_rho[(wib * T + t) * 32 + lane] = rho[t];
            }
            __syncthreads();
            for (int t = wib; t < T; t += NW) {
                int c = 0;
                float d = 0.0f;
                for (int w = 0; w < NW; w++) {
                    c += s_cnt[(w * T + t) * 32 + lane];
                    d += s_rho[(w * T + t) * 32 + lane];
                }
                const int o = t * 32 + lane;
                if (o < gc) {
                    const uint32_t dst = P.perm[gb + o];
                    if (P.count) P.count[dst] = max(c, 0);
                    if (P.rho) P.rho[dst] = d;
                }
            }
            continue;
        }
#pragma unroll
        for (int t = 0; t < T; t++) {
            const int o = t * 32 + lane;
            if (o < gc) {
                const uint32_t dst = P.perm[gb + o];
                if (P.count) P.count[dst] = max(cnt[t], 0);
                if (P.rho) P.rho[dst] = rho[t];
            }
        }
    }
    if (lane == 0) {
        atomicAdd(&ctrl->n_pp, tested);
        atomicAdd(&ctrl->cum_pp, tested);
    }
}

// persistent grid: as many blocks per SM as the registers and shared memory allow
template <int T, int NW>
static void bh_sph_launch_nw(const SphParams& P, int sm_count, cudaStream_t s)
{
    constexpr int threads = NW == 1 ? 128 : NW * 32;
    int bps = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, bh_sph_kernel<T, NW>, threads, 0) != cudaSuccess || bps < 1) {
        cudaGetLastError();
        bps = 1;
    }
    bh_launch_after(bh_sph_kernel<T, NW>, sm_count * bps, threads, 0, s, P);
}
template <int T>
static int bh_sph_launch(const SphParams& P, int sm_count, cudaStream_t s)
{
    bh_sph_launch_nw<T, 1>(P, sm_count, s);
    bh_sph_launch_nw<T, bh_sph_team<T>()>(P, sm_count, s);
    return BH_OK;
}

int launch_sph(const float4* pos_s, const uint32_t* perm, const int32_t* g_first, const int32_t* g_count,
               const bh_nodes& nd, float4* blo, float4* bhi, int G, const float* h, float h_const, int32_t* count,
               float* rho, int32_t* heavy, int n, bh_dev_ctrl* ctrl, int sm_count, int grid, int max_level, cudaStream_t s)
{
    SphParams P;
    P.pos_s = pos_s;
    P.perm = perm;
    P.g_first = g_first;
    P.g_count = g_count;
    P.rec = nd.rec;
    P.blo = blo;
    P.bhi = bhi;
    P.h = h;
    P.h_const = h_const;
    P.count = count;
    P.rho = rho;
    P.ctrl = ctrl;
    P.heavy = heavy;
    P.max_level = max_level;
    for (int lev = max_level; lev >= 0; lev--)
        bh_launch_after(bh_node_box_kernel, grid, 256, 0, s, pos_s, nd.rec, blo, bhi, lev, P, n);
    const int T = G <= 32 ? 1 : G <= 64 ? 2 : G <= 96 ? 3 : G <= 128 ? 4 : 8;
    switch (T) {
        case 1: return bh_sph_launch<1>(P, sm_count, s);
        case 2: return bh_sph_launch<2>(P, sm_count, s);
        case 3: return bh_sph_launch<3>(P, sm_count, s);
        case 4: return bh_sph_launch<4>(P, sm_count, s);
        default: return bh_sph_launch<8>(P, sm_count, s);
    }
}

}  // namespace bh
