// bh_walk_team.cu -- the group walk with a block of warps per group.
//
// bh_walk_kernel gives each group to one warp.  A set of a few thousand to a
// few hundred thousand particles has fewer groups than the GPU holds warps, so
// its time is the latency of the longest single warp's walk: 195 us for 71
// groups, most of the GPU idle.  Here a block of kTeamWarps warps shares one
// group: warp 0 walks the tree and cuts the source lists into tiles (node or
// particle indices only, it loads no source), the other warps take the tiles
// as they come, stage their sources and evaluate them.
//
// Same bits as bh_walk_kernel: the walk pops, tests and appends in its order,
// a tile holds the same 64 sources, its partial sums are computed by the same
// device functions, and the tiles' sums are added to the group's totals (in
// shared memory, Kahan compensated) in tile order: an evaluator waits for its
// tile's turn.  Tiles of one group are evaluated at once; only these additions
// (a few dozen instructions per tile) are serial.
#include <algorithm>

#include "bh_walk.cuh"

namespace bh {

constexpr int kTeamSlots = 16;                 // tiles handed over and not yet read
constexpr int kTeamRing = 1024;                // pending point sources (indices)
constexpr uint32_t kTeamCell = 0x80000000u;    // index of a node (monopole cell), not of a particle
enum : int { kTeamSelf = 0, kTeamPoints = 1, kTeamQuads = 2, kTeamEnd = 3 };

struct TeamSmem {
    uint32_t stack[kStackCap];
    int2 leafq[64];
    uint32_t qring[kRing];
    uint32_t pring[kTeamRing];
    uint32_t idx[kTeamSlots][kTile];
    int meta[kTeamSlots];  // kind << 8 | sources
    unsigned long long full[kTeamSlots], empty[kTeamSlots];
    int group;             // the block's group, -1: done
    int claim;             // next tile to be taken
    volatile int turn;     // next tile to be added to the totals
    volatile int dead;     // a wait gave up
};

// One tile's sums: the running-total interface of Acc with nothing before it
// (the compensation of 0 + v is 0).
template <int T>
struct TileSum {
    float x[T], y[T], z[T], p[T], cc[4 * T];
    __device__ __forceinline__ float& c(int t, int k) { return cc[4 * t + k]; }
};

// Wait for tile i's turn (bounded like bh_mbar_wait).
__device__ __forceinline__ bool bh_turn_wait(const volatile int* turn, int i, bh_dev_ctrl* c)
{
    if (*turn == i) return true;
    WaitLimit lim(bh_globaltimer());
    for (int k = 0; k < lim.end; k++) {
        if (*turn == i) return true;
        __nanosleep(20);
        if ((k & 63) == 63) {
            if (*(volatile unsigned int*)&c->abort) return false;
            lim.look(k, bh_globaltimer());
        }
    }
    bh_set_error(c, BH_ERR_DEVICE_TIMEOUT);
    return false;
}

// Walker side: hand `cnt` indices (fill(k) = k-th) over as the next tile.
template <class Fill>
__device__ __forceinline__ bool bh_team_send(TeamSmem& S, int& item, int kind, int cnt, bh_dev_ctrl* ctrl, Fill fill)
{
    const int lane = threadIdx.x & 31, s = item % kTeamSlots;
    const bool ok = bh_mbar_wait(&S.empty[s], ((unsigned int)(item / kTeamSlots) & 1u) ^ 1u, ctrl);
    if (__any_sync(BH_FULL_MASK, !ok)) return false;
    for (int k = lane; k < cnt; k += 32) S.idx[s][k] = fill(k);
    if (lane == 0) S.meta[s] = (kind << 8) | cnt;
    __syncwarp();
    if (lane == 0) bh_mbar_arrive(&S.full[s]);
    item++;
    return true;
}

template <int T, int NW>
__host__ __device__ constexpr size_t bh_team_smem_bytes()
{
    return sizeof(TeamSmem) + 2 * 4 * T * 32 * sizeof(float) + (NW - 1) * sizeof(WsTile);
}

// NW: warps per block, one walker and NW - 1 evaluators
template <int T, int ORDER, int NW>
__global__ void __launch_bounds__(NW * 32, (T <= 3 ? 16 : 8) / NW) bh_walk_team_kernel(WalkParams P)
{
    bh_let_next_start();
    bh_after_previous();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // A block's warps sit on the SM's schedulers in turn; the walker, which
    // issues little, is another warp in each of the blocks that share an SM.
    const int lane = threadIdx.x & 31;
    const int wib = (int)(threadIdx.x / 32 + blockIdx.x / P.sm_count) % NW;  // 0: walker
    WsTile* tiles = reinterpret_cast<WsTile*>(smem_raw);
    float* tot = reinterpret_cast<float*>(smem_raw + (NW - 1) * sizeof(WsTile));  // [4T][32] sums
    float* comp = tot + 4 * T * 32;                                                // [4T][32] compensations
    TeamSmem& S = *reinterpret_cast<TeamSmem*>(comp + 4 * T * 32);
    bh_dev_ctrl* ctrl = P.ctrl;
    const int ng = (int)ctrl->n_groups, n_roots = (int)ctrl->level_offset[1];
    const float eps2 = P.eps2;
    const f2 eps2v = make_float2(eps2, eps2);
    const unsigned int lt = bh_lanemask_lt();
    if (threadIdx.x < kTeamSlots) {
        bh_mbar_init(&S.full[threadIdx.x], 1u);
        bh_mbar_init(&S.empty[threadIdx.x], 1u);
    }
    if (threadIdx.x == 0) {
        S.claim = 0;
        S.turn = 0;
        S.dead = 0;
    }
    int item = 0, next = 0;  // walker: next tile; lane 0: next group of the block
    unsigned long long cnt_pp = 0ull, cnt_pc = 0ull;
    const bool lead = wib == 0 && lane == 0;
    if (lead) next = (int)atomicAdd(&ctrl->group_ctr, 1u);
    for (;;) {
        if (lead) {
            S.group = (next < ng && !*(volatile unsigned int*)&ctrl->abort) ? next : -1;
            if (next < ng) next = (int)atomicAdd(&ctrl->group_ctr, 1u);
        }
        __syncthreads();
        if (S.group < 0) break;
        const int g = P.g_order ? P.g_order[S.group] : S.group;
        const int gb = P.g_first[g], gc = P.g_count[g], ge = gb + gc;
        Layout L;
        {
            const int tn = (gc + 31) >> 5, kl = gc - 32 * (tn - 1);
            L.split = (T <= 4) && (kl <= kSplitMax);
            L.nf = L.split ? tn - 1 : tn;
            L.lg = L.split ? (kl > 1 ? 32 - __clz(kl - 1) : 0) : 5;
        }
        if (wib == 0) {
            // ---------------------------------------------------- walker
            bool alive = bh_team_send(S, item, kTeamSelf, 0, ctrl, [](int) { return 0u; });
            unsigned int lo0 = 0xffffffffu, lo1 = 0xffffffffu, lo2 = 0xffffffffu, hi0 = 0u, hi1 = 0u, hi2 = 0u;
            for (int o = lane; o < gc; o += 32) {
                const float4 q = P.pos_s[gb + o];
                lo0 = min(lo0, bh_f2ord(q.x)); lo1 = min(lo1, bh_f2ord(q.y)); lo2 = min(lo2, bh_f2ord(q.z));
                hi0 = max(hi0, bh_f2ord(q.x)); hi1 = max(hi1, bh_f2ord(q.y)); hi2 = max(hi2, bh_f2ord(q.z));
            }
            const float bx0 = bh_ord2f(__reduce_min_sync(BH_FULL_MASK, lo0));
            const float by0 = bh_ord2f(__reduce_min_sync(BH_FULL_MASK, lo1));
            const float bz0 = bh_ord2f(__reduce_min_sync(BH_FULL_MASK, lo2));
            const float bx1 = bh_ord2f(__reduce_max_sync(BH_FULL_MASK, hi0));
            const float by1 = bh_ord2f(__reduce_max_sync(BH_FULL_MASK, hi1));
            const float bz1 = bh_ord2f(__reduce_max_sync(BH_FULL_MASK, hi2));
            cnt_pp += (unsigned long long)gc * (unsigned long long)(gc - 1);
            int root = 0;  // the group's system: the last level-0 node starting at or before gb
            for (int hi = n_roots; hi - root > 1;) {
                const int mid = (root + hi) >> 1;
                if (P.rec[mid].x <= gb) root = mid;
                else hi = mid;
            }
            int sp = 1, p_head = 0, p_cnt = 0, q_head = 0, q_cnt = 0;
            if (lane == 0) S.stack[0] = (uint32_t)root << 3;
            __syncwarp();
            bool overflow = false;
            // Pop the top 32 nodes (ranges of siblings), issue the loads of their
            // records and return how many there are.  The next pop is taken as
            // soon as a pop's children are pushed, so that its records arrive
            // while the pop's tiles are handed over.
            int v = 0;
            float4 cm;
            float se;
            int4 r;
            auto pop = [&]() -> int {
                if (sp == 0) return 0;
                int row;
                const int npop = bh_pop_nodes(S.stack, sp, lt, v, row);
                cm = make_float4(0.f, 0.f, 0.f, 0.f);
                se = 0.f;
                r = make_int4(0, 0, -1, 0);
                if (lane < npop) {
                    cm = P.com_m[v];
                    se = P.seff[v];
                    r = P.rec[v];
                }
                __syncwarp();
                return npop;
            };
            int npop = pop();
            while (npop > 0 && alive) {
                // ---- test the nodes
                const bool has = lane < npop;
                const float dx = fmaxf(fmaxf(bx0 - cm.x, cm.x - bx1), 0.0f);
                const float dy = fmaxf(fmaxf(by0 - cm.y, cm.y - by1), 0.0f);
                const float dz = fmaxf(fmaxf(bz0 - cm.z, cm.z - bz1), 0.0f);
                const float d2 = bh_dist2(dx, dy, dz);
                const bool member = (r.x < ge) && (r.x + r.y > gb);
                const bool acc = has && (d2 > se) && !member;
                const bool leaf = has && !acc && (r.z < 0);
                const bool opn = has && !acc && (r.z >= 0);

                // ---- open: push child ranges
                const unsigned int om = __ballot_sync(BH_FULL_MASK, opn);
                const int npush = __popc(om);
                if (sp + npush > kStackCap) {
                    overflow = true;
                    break;
                }
                if (opn) S.stack[sp + __popc(om & lt)] = ((uint32_t)r.z << 3) | (uint32_t)(r.w - 1);
                sp += npush;

                // ---- accept: cell sources
                const unsigned int am = __ballot_sync(BH_FULL_MASK, acc);
                const int nacc = __popc(am);
                cnt_pc += (unsigned long long)nacc * (unsigned long long)gc;
                if (ORDER >= 2) {
                    if (acc) S.qring[(q_head + q_cnt + __popc(am & lt)) & (kRing - 1)] = (uint32_t)v;
                    q_cnt += nacc;
                } else {
                    if (acc) S.pring[(p_head + p_cnt + __popc(am & lt)) & (kTeamRing - 1)] = (uint32_t)v | kTeamCell;
                    p_cnt += nacc;
                }

                // ---- rejected leaves: particle ranges outside the group
                const int a0 = r.x, a1 = r.x + r.y;
                const bool pa = leaf && (a0 < gb);
                const bool pb = leaf && (a1 > ge);
                const int pa_n = pa ? (min(a1, gb) - a0) : 0;
                const int pb_s = max(a0, ge);
                const int pb_n = pb ? (a1 - pb_s) : 0;
                const unsigned int ma = __ballot_sync(BH_FULL_MASK, pa), mb = __ballot_sync(BH_FULL_MASK, pb);
                const int lq_n = __popc(ma) + __popc(mb);
                if (pa) S.leafq[__popc(ma & lt)] = make_int2(a0, pa_n);
                if (pb) S.leafq[__popc(ma) + __popc(mb & lt)] = make_int2(pb_s, pb_n);
                cnt_pp += (unsigned long long)__reduce_add_sync(BH_FULL_MASK, (unsigned int)(pa_n + pb_n)) *
                          (unsigned long long)gc;
                __syncwarp();
                npop = pop();

                // ---- hand over: quadrupole tiles, then point tiles
                while (ORDER >= 2 && q_cnt >= kTile && alive) {
                    alive = bh_team_send(S, item, kTeamQuads, kTile, ctrl,
                                         [&](int k) { return S.qring[(q_head + k) & (kRing - 1)]; });
                    q_head = (q_head + kTile) & (kRing - 1);
                    q_cnt -= kTile;
                }
                int lq_pos = 0;
                while (alive) {
                    if (p_cnt >= kTile) {
                        alive = bh_team_send(S, item, kTeamPoints, kTile, ctrl,
                                             [&](int k) { return S.pring[(p_head + k) & (kTeamRing - 1)]; });
                        p_head = (p_head + kTile) & (kTeamRing - 1);
                        p_cnt -= kTile;
                        continue;
                    }
                    if (lq_pos >= lq_n) break;
                    // a round: up to kTeamRing - kTile particles of the pending ranges, each
                    // lane writing its range's indices at its place in the ring
                    int c2 = 0;
                    int2 q = make_int2(0, 0);
                    if (lq_pos + lane < lq_n) {
                        q = S.leafq[lq_pos + lane];
                        c2 = q.y;
                    }
                    const int inc2 = bh_warp_incl_scan(c2);
                    const int ex2 = inc2 - c2;
                    const int take2 = max(0, min(c2, kTeamRing - kTile - ex2));
#pragma unroll 4
                    for (int t = 0; t < take2; t++)
                        S.pring[(p_head + p_cnt + ex2 + t) & (kTeamRing - 1)] = (uint32_t)(q.x + t);
                    const bool full2 = (lq_pos + lane < lq_n) && (take2 == c2);
                    const int nf2 = __popc(__ballot_sync(BH_FULL_MASK, full2));
                    const int nround = min(__shfl_sync(BH_FULL_MASK, inc2, 31), kTeamRing - kTile);
                    __syncwarp();
                    if (lane == nf2 && lq_pos + lane < lq_n && take2 > 0)
                        S.leafq[lq_pos + lane] = make_int2(q.x + take2, c2 - take2);
                    lq_pos += nf2;
                    p_cnt += nround;
                    __syncwarp();
                }
            }
            if (overflow && lane == 0) {
                bh_set_error(ctrl, BH_ERR_CAPACITY);
                S.dead = 1;
            }
            // ---- the partial tiles, then one end mark per evaluator
            if (ORDER >= 2 && q_cnt > 0 && alive)
                alive = bh_team_send(S, item, kTeamQuads, q_cnt, ctrl,
                                     [&](int k) { return S.qring[(q_head + k) & (kRing - 1)]; });
            if (p_cnt > 0 && alive)
                alive = bh_team_send(S, item, kTeamPoints, p_cnt, ctrl,
                                     [&](int k) { return S.pring[(p_head + k) & (kTeamRing - 1)]; });
            for (int k = 0; k < NW - 1 && alive; k++)
                alive = bh_team_send(S, item, kTeamEnd, 0, ctrl, [](int) { return 0u; });
            if (!alive && lane == 0) S.dead = 1;
        } else {
            // ---------------------------------------------------- evaluator
            WsTile& W = tiles[wib - 1];
            const int lmask = (1 << L.lg) - 1;
            Tgt<T> X;
#pragma unroll
            for (int t = 0; t < T; t++) {
                const int o = t * 32 + ((L.split && t == L.nf) ? (lane & lmask) : lane);
                float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                if (o < gc) q = P.pos_s[gb + o];
                X.x[t] = make_float2(q.x, q.x);
                X.y[t] = make_float2(q.y, q.y);
                X.z[t] = make_float2(q.z, q.z);
            }
            for (;;) {
                int i = 0;
                if (lane == 0) i = atomicAdd(&S.claim, 1);
                i = __shfl_sync(BH_FULL_MASK, i, 0);
                const int s = i % kTeamSlots;
                bool ok = bh_mbar_wait(&S.full[s], (unsigned int)(i / kTeamSlots) & 1u, ctrl);
                if (__any_sync(BH_FULL_MASK, !ok)) {
                    S.dead = 1;
                    break;
                }
                const int kind = S.meta[s] >> 8, cnt = S.meta[s] & 0xff;
                const uint32_t j0 = S.idx[s][lane], j1 = S.idx[s][lane + 32];
                __syncwarp();
                if (lane == 0) bh_mbar_arrive(&S.empty[s]);  // read: the walker may reuse the slot
                if (kind == kTeamEnd) break;
                TileSum<T> V;
#pragma unroll
                for (int t = 0; t < T; t++) V.x[t] = V.y[t] = V.z[t] = V.p[t] = 0.0f;
#pragma unroll
                for (int k = 0; k < 4 * T; k++) V.cc[k] = 0.0f;
                if (kind == kTeamSelf) {
                    float xi[T], yi[T], zi[T], mi[T];
#pragma unroll
                    for (int t = 0; t < T; t++) {
                        const int o = t * 32 + ((L.split && t == L.nf) ? (lane & lmask) : lane);
                        xi[t] = X.x[t].x; yi[t] = X.y[t].x; zi[t] = X.z[t].x;
                        mi[t] = o < gc ? P.pos_s[gb + o].w : 0.0f;
                    }
                    bh_eval_self<T>(gc, L, eps2, xi, yi, zi, mi, V);
                } else if (ORDER >= 2 && kind == kTeamQuads) {
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int k = lane + 32 * h;
                        const uint32_t v = h ? j1 : j0;
                        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (k < cnt) bh_put_quad(W, k, P.com_m[v], P.quad[2 * (size_t)v], P.quad[2 * (size_t)v + 1], eps2);
                        else bh_put_quad(W, k, bh_pad_source(), z4, z4, eps2);
                    }
                    __syncwarp();
                    bh_quads<T, WsTile, bh_quad_unroll<T, false>()>(L, W, 0, eps2v, X, V, (cnt + 1) >> 1);
                } else if (kind == kTeamPoints) {
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int k = lane + 32 * h;
                        const uint32_t j = h ? j1 : j0;
                        float4 q = bh_pad_source();
                        if (k < cnt) q = (j & kTeamCell) ? P.com_m[j & ~kTeamCell] : P.pos_s[j];
                        bh_put_point(W.a, W.b, k, q);
                    }
                    __syncwarp();
                    bh_points<T, kPointUnroll>(L, W.a, W.b, eps2v, X, V,
                                               (((cnt + 1) >> 1) + kPointUnroll - 1) / kPointUnroll * kPointUnroll);
                }
                // ---- in tile order: add to the group's totals (the self tile, the first, starts them)
                ok = bh_turn_wait(&S.turn, i, ctrl);
                if (__any_sync(BH_FULL_MASK, !ok)) {
                    S.dead = 1;
                    break;
                }
                __threadfence_block();
#pragma unroll
                for (int t = 0; t < T; t++) {
                    const float w[4] = {V.x[t], V.y[t], V.z[t], V.p[t]};
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const int o = (4 * t + k) * 32 + lane;
                        float sum = kind == kTeamSelf ? 0.0f : tot[o], cmp = kind == kTeamSelf ? 0.0f : comp[o];
                        bh_kahan(sum, cmp, w[k]);
                        tot[o] = sum;
                        comp[o] = cmp;
                    }
                }
                __threadfence_block();
                __syncwarp();
                if (lane == 0) S.turn = i + 1;
            }
        }
        __syncthreads();
        if (S.dead) break;
        if (lead) S.turn = item;  // past the end marks, which are not added
        // ---- write (ax, ay, az, phi) in the caller's order, a slot per warp; a
        // split slot first adds its phases' sums
        for (int t = wib; t < T; t += NW) {
            float4 f;
            {
                const int o = 4 * t * 32 + lane;
                f.x = tot[o] - comp[o];
                f.y = tot[o + 32] - comp[o + 32];
                f.z = tot[o + 64] - comp[o + 64];
                f.w = tot[o + 96] - comp[o + 96];
            }
            if (L.split && t == L.nf) {
                for (int off = 1 << L.lg; off < 32; off <<= 1) {
                    f.x += __shfl_xor_sync(BH_FULL_MASK, f.x, off);
                    f.y += __shfl_xor_sync(BH_FULL_MASK, f.y, off);
                    f.z += __shfl_xor_sync(BH_FULL_MASK, f.z, off);
                    f.w += __shfl_xor_sync(BH_FULL_MASK, f.w, off);
                }
            }
            const int o = t * 32 + lane;
            if (o < gc) P.out[P.perm[gb + o]] = f;
        }
    }
    if (lead && (cnt_pp | cnt_pc) != 0ull) {
        atomicAdd(&ctrl->n_pp, cnt_pp);
        atomicAdd(&ctrl->n_pc, cnt_pc);
        atomicAdd(&ctrl->cum_pp, cnt_pp);
        atomicAdd(&ctrl->cum_pc, cnt_pc);
    }
}

template <int T, int ORDER, int NW>
static int bh_team_launch(const WalkParams& P, int n, int sm_count, cudaStream_t s)
{
    constexpr size_t smem = bh_team_smem_bytes<T, NW>();
    auto kern = bh_walk_team_kernel<T, ORDER, NW>;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return BH_ERR_CUDA;
    int bps = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, NW * 32, smem) != cudaSuccess || bps < 1)
        return BH_ERR_CUDA;
    bh_launch_after(kern, std::min(sm_count * bps, n), NW * 32, smem, s, P);  // at most a group per particle
    return BH_OK;
}

template <int NW>
static int bh_team_dispatch(const WalkParams& P, int order, int G, int n, int sm_count, cudaStream_t s)
{
    const int T = (G + 31) / 32;
    if (order >= 2) {
        switch (T) {
            case 1: return bh_team_launch<1, 2, NW>(P, n, sm_count, s);
            case 2: return bh_team_launch<2, 2, NW>(P, n, sm_count, s);
            case 3: return bh_team_launch<3, 2, NW>(P, n, sm_count, s);
            default: return bh_team_launch<4, 2, NW>(P, n, sm_count, s);
        }
    }
    switch (T) {
        case 1: return bh_team_launch<1, 1, NW>(P, n, sm_count, s);
        case 2: return bh_team_launch<2, 1, NW>(P, n, sm_count, s);
        case 3: return bh_team_launch<3, 1, NW>(P, n, sm_count, s);
        default: return bh_team_launch<4, 1, NW>(P, n, sm_count, s);
    }
}

// (How many warps a set gets: bh_team_warps in bh_internal.cuh.)
int launch_walk_team(const WalkParams& P, int order, int G, const WalkSet& set, int sm_count, cudaStream_t s)
{
    switch (bh_team_warps(set, G, sm_count)) {
        case 8: return bh_team_dispatch<8>(P, order, G, set.n, sm_count, s);
        case 4: return bh_team_dispatch<4>(P, order, G, set.n, sm_count, s);
        default: return 1;
    }
}

}  // namespace bh
