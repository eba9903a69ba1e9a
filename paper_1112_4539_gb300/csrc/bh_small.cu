// bh_small.cu -- the whole build of a small set in one block.
//
// The 14 launches of a small set's build (18 with 63-bit keys) are a chain of
// short kernels with a few blocks each: about 5 us of latency apiece, 72 us for
// 4096 particles, for work that fits one SM's shared memory.  Here a
// block of 1024 threads does it all: bounds, keys, the stable radix sort (keys
// and indices stay in shared memory between its passes), the gather, node
// levels, node arrays and walk groups, with the same arithmetic and orders as
// bh_sort.cu and bh_tree.cu, so every array is the same.
//
// Bound by the latency of its phases up to about 1000 particles, then by one
// SM's issue slots (6 us per 1024 particles).  Build on GB300, leaf 8, the chain
// of launches -> this: 30-bit keys 1000 59 -> 30 us, 4096 72 -> 37, 8192 78 -> 62,
// 16384 87 -> 122; 63-bit keys 1000 80 -> 48, 4096 97 -> 60, 8192 100 -> 106.  Hence
// the limits in bh_small_set, 8192 and 4096 particles.
#include <algorithm>

#include "bh_internal.cuh"

namespace bh {

constexpr int kST = 1024;        // threads
constexpr int kSW = kST / 32;    // warps

struct SmallParams {
    const float4* pos;
    int n, n_leaf, G;
    long long node_cap;
    bh_nodes nd;
    void* keys;
    uint32_t* vals;
    float4* pos_s;
    int32_t* g_first;
    int32_t* g_count;
    bh_dev_ctrl* ctrl;
};

// Shared memory: sorted keys, 16-bit words per particle (indices, then d and
// lambda of each position), and bytes per particle that first hold the warps'
// digit counts, then window levels, then group flags.
template <typename K, int IT>
struct SmallSmem {
    K key[kST * IT];
    uint16_t val[kST * IT];
    union {
        uint16_t hist[kSW][256];
        int8_t win[kST * IT];
        uint8_t flag[kST * IT];
    };
    unsigned int start[256];
    unsigned int wtot[11][kSW];
    unsigned int red[kSW][8];
    int next[kSW + 1];
    unsigned int off[BH_LEVEL_SLOTS];
    float box[4];
    float inv;
    int nodes;
};

template <int CURVE, typename K, int IT>
__global__ void __launch_bounds__(kST) bh_small_build_kernel(SmallParams P)
{
    bh_let_next_start();
    bh_after_previous();
    constexpr int L = bh_key_traits<K>::kMaxLevel, NP = bh_key_traits<K>::kPasses;
    constexpr unsigned int CMAX = (1u << L) - 1u;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem<K, IT>& S = *reinterpret_cast<SmallSmem<K, IT>*>(smem_raw);
    bh_dev_ctrl* c = P.ctrl;
    const int n = P.n, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int i0 = w * (32 * IT) + lane;  // item k of the thread: position i0 + 32 k

    // ---- bounds (as bh_bbox_kernel) and the control block (as bh_init_kernel)
    {
        unsigned int lo0 = 0xffffffffu, lo1 = 0xffffffffu, lo2 = 0xffffffffu, hi0 = 0u, hi1 = 0u, hi2 = 0u;
        bool bad = false;
#pragma unroll
        for (int k = 0; k < IT; k++)
            if (i0 + 32 * k < n) {
                const float4 p = P.pos[i0 + 32 * k];
                bad |= !(isfinite(p.x) && isfinite(p.y) && isfinite(p.z) && isfinite(p.w));
                const unsigned int ox = bh_f2ord(p.x), oy = bh_f2ord(p.y), oz = bh_f2ord(p.z);
                lo0 = min(lo0, ox); lo1 = min(lo1, oy); lo2 = min(lo2, oz);
                hi0 = max(hi0, ox); hi1 = max(hi1, oy); hi2 = max(hi2, oz);
            }
        lo0 = __reduce_min_sync(BH_FULL_MASK, lo0); lo1 = __reduce_min_sync(BH_FULL_MASK, lo1);
        lo2 = __reduce_min_sync(BH_FULL_MASK, lo2); hi0 = __reduce_max_sync(BH_FULL_MASK, hi0);
        hi1 = __reduce_max_sync(BH_FULL_MASK, hi1); hi2 = __reduce_max_sync(BH_FULL_MASK, hi2);
        const unsigned int nb = __any_sync(BH_FULL_MASK, bad) ? 1u : 0u;
        if (lane == 0) {
            S.red[w][0] = lo0; S.red[w][1] = lo1; S.red[w][2] = lo2;
            S.red[w][3] = hi0; S.red[w][4] = hi1; S.red[w][5] = hi2;
            S.red[w][6] = nb;
        }
        __syncthreads();
        if (w == 0) {
            unsigned int mm[6];
#pragma unroll
            for (int k = 0; k < 3; k++) mm[k] = __reduce_min_sync(BH_FULL_MASK, S.red[lane][k]);
#pragma unroll
            for (int k = 3; k < 6; k++) mm[k] = __reduce_max_sync(BH_FULL_MASK, S.red[lane][k]);
            const unsigned int any = __reduce_or_sync(BH_FULL_MASK, S.red[lane][6]);
            if (lane == 0) {
                bh_box_from_minmax(mm, S.box, &S.inv);
                for (int k = 0; k < 6; k++) c->minmax[k] = mm[k];
                for (int k = 0; k < 4; k++) c->box[k] = S.box[k];
                c->inv = S.inv;
                c->status = any ? (unsigned int)(-BH_ERR_NONFINITE) : 0u;
                c->abort = 0u;
                c->group_ctr = 0u;
                c->n_pp = 0ull;
                c->n_pc = 0ull;
                c->build_seq += 1u;
            }
        }
        __syncthreads();
    }

    // ---- keys (as bh_keys_kernel)
    K key[IT];
    uint16_t val[IT], rank[IT];
    {
        const float x0 = S.box[0], y0 = S.box[1], z0 = S.box[2], inv = __fmul_rn(S.inv, (float)(1u << (L - 10)));
#pragma unroll
        for (int k = 0; k < IT; k++) {
            const int i = i0 + 32 * k;
            key[k] = 0;
            val[k] = (uint16_t)i;
            if (i < n) {
                const float4 p = P.pos[i];
                const unsigned int cx = min(__float2uint_rz(__fmul_rn(__fsub_rn(p.x, x0), inv)), CMAX);
                const unsigned int cy = min(__float2uint_rz(__fmul_rn(__fsub_rn(p.y, y0), inv)), CMAX);
                const unsigned int cz = min(__float2uint_rz(__fmul_rn(__fsub_rn(p.z, z0), inv)), CMAX);
                key[k] = bh_key_of<CURVE, K>(cx, cy, cz);
            }
        }
    }

    // ---- stable 8-bit passes from the lowest bits
    const unsigned int lt = bh_lanemask_lt();
#pragma unroll 1
    for (int pass = 0; pass < NP; pass++) {
        const int shift = 8 * pass;
        reinterpret_cast<uint4*>(&S.hist[0][0])[tid] = make_uint4(0u, 0u, 0u, 0u);  // 16 KB
        __syncthreads();
#pragma unroll
        for (int k = 0; k < IT; k++) {
            const bool ok = i0 + 32 * k < n;
            const unsigned int d = (unsigned int)(key[k] >> shift) & 255u;
            const unsigned int peers = bh_match_digit(d, ok);
            unsigned int prior = 0u;
            if (ok) prior = S.hist[w][d];
            __syncwarp();
            if (ok && lane == __ffs(peers) - 1) S.hist[w][d] = (uint16_t)(prior + __popc(peers));
            __syncwarp();
            rank[k] = (uint16_t)(prior + __popc(peers & lt));
        }
        __syncthreads();
        // per digit, exclusive over the warps: four threads each, eight warps apiece
        {
            const int d = tid >> 2, q = tid & 3;
            unsigned int cnt[8], sum = 0u;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                cnt[i] = S.hist[8 * q + i][d];
                sum += cnt[i];
            }
            unsigned int incl = sum;
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                const unsigned int t = __shfl_up_sync(BH_FULL_MASK, incl, o, 4);
                if (q >= o) incl += t;
            }
            unsigned int run = incl - sum;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                S.hist[8 * q + i][d] = (uint16_t)run;
                run += cnt[i];
            }
            if (q == 3) S.start[d] = run;  // the digit's count
        }
        __syncthreads();
        // exclusive over the digits
        unsigned int mine = 0u, incl = 0u;
        if (tid < 256) {
            mine = S.start[tid];
            incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int t = __shfl_up_sync(BH_FULL_MASK, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) S.red[w][0] = incl;
        }
        __syncthreads();
        if (tid < 256) {
            unsigned int before = incl - mine;
            for (int i = 0; i < w; i++) before += S.red[i][0];
            S.start[tid] = before;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < IT; k++)
            if (i0 + 32 * k < n) {
                const unsigned int d = (unsigned int)(key[k] >> shift) & 255u;
                const unsigned int at = S.start[d] + S.hist[w][d] + rank[k];
                S.key[at] = key[k];
                S.val[at] = val[k];
            }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < IT; k++)
            if (i0 + 32 * k < n) {
                key[k] = S.key[i0 + 32 * k];
                val[k] = S.val[i0 + 32 * k];
            }
    }
    // ---- sorted keys, indices, particles
#pragma unroll
    for (int k = 0; k < IT; k++) {
        const int i = i0 + 32 * k;
        if (i < n) {
            reinterpret_cast<K*>(P.keys)[i] = key[k];
            P.vals[i] = val[k];
            P.pos_s[i] = P.pos[val[k]];
        }
    }
    __syncthreads();  // (val is read; hist is done with)

    // ---- node levels (as bh_levels_kernel)
    for (int j = tid; j < n; j += kST)
        S.win[j] = j + P.n_leaf < n ? (int8_t)bh_common_level(S.key[j], S.key[j + P.n_leaf]) : (int8_t)-1;
    __syncthreads();
    for (int k = tid; k < kST * IT; k += kST) {
        uint16_t dl = (uint16_t)(L + 1);  // past the end: d + 1 = L + 1 > lambda = 0, no node
        if (k < n) {
            const int d = k == 0 ? -1 : bh_common_level(S.key[k - 1], S.key[k]);
            int W = -1;
            for (int j = max(0, k - P.n_leaf); j <= k; j++) W = max(W, (int)S.win[j]);
            dl = (uint16_t)((d + 1) | (min(L, W + 1) << 5));
        }
        S.val[k] = dl;
    }
    __syncthreads();
    // ---- node indices: per level, the nodes of the positions before the thread's
    const int k0 = tid * IT;  // the thread's IT consecutive positions
    constexpr int NQ = (L + 2) / 2;  // two levels per word, 16 bits each
    unsigned int run[NQ];
    {
        unsigned int cnt[NQ];
#pragma unroll
        for (int q = 0; q < NQ; q++) cnt[q] = 0u;
#pragma unroll 1
        for (int r = 0; r < IT; r++) {
            const unsigned int dl = S.val[k0 + r];
            const int d1 = (int)(dl & 31u), lam = (int)(dl >> 5);  // nodes of levels d1 .. lam
#pragma unroll
            for (int l = 0; l <= L; l++) cnt[l >> 1] += (l >= d1 && l <= lam) ? 1u << (16 * (l & 1)) : 0u;
        }
#pragma unroll
        for (int q = 0; q < NQ; q++) {
            unsigned int incl = cnt[q];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int t = __shfl_up_sync(BH_FULL_MASK, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) S.wtot[q][w] = incl;
            run[q] = incl - cnt[q];
        }
        __syncthreads();
        if (w < NQ) {  // exclusive over the warps; the total of the pair of levels in the end
            const unsigned int x = S.wtot[w][lane];
            unsigned int incl = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int t = __shfl_up_sync(BH_FULL_MASK, incl, o);
                if (lane >= o) incl += t;
            }
            S.wtot[w][lane] = incl - x;
            if (lane == 31) {
                S.off[2 * w] = incl & 0xffffu;
                if (2 * w + 1 <= L) S.off[2 * w + 1] = incl >> 16;
            }
        }
        __syncthreads();
        if (tid == 0) {
            unsigned int total = 0u;
            for (int l = 0; l <= L; l++) {
                const unsigned int t = S.off[l];
                c->level_total[l] = t;
                S.off[l] = total;
                total += t;
            }
            if ((long long)total > P.node_cap) {
                bh_set_error(c, BH_ERR_CAPACITY);
                total = 0u;  // later kernels see an empty tree
                for (int l = 0; l <= L; l++) S.off[l] = 0u;
            }
            for (int l = L + 1; l < BH_LEVEL_SLOTS; l++) S.off[l] = total;
            S.nodes = (int)total;
            c->n_nodes = total;
        }
        __syncthreads();
        if (tid < BH_LEVEL_SLOTS) c->level_offset[tid] = S.off[tid];
#pragma unroll
        for (int q = 0; q < NQ; q++) run[q] += S.wtot[q][w];
    }
    const int nn = S.nodes;
    // ---- node arrays (as bh_node_write_kernel)
    if (nn > 0) {
#pragma unroll 1
        for (int r = 0; r < IT; r++) {
            const unsigned int dl = S.val[k0 + r];
            const int d1 = (int)(dl & 31u), lam = (int)(dl >> 5);
            int below = -1;  // index of node (k, l + 1)
#pragma unroll
            for (int l = L; l >= 0; l--)
                if (l >= d1 && l <= lam) {
                    const int idx = (int)(S.off[l] + ((run[l >> 1] >> (16 * (l & 1))) & 0xffffu));
                    run[l >> 1] += 1u << (16 * (l & 1));
                    P.nd.first[idx] = k0 + r;
                    P.nd.level[idx] = (uint8_t)l;
                    P.nd.child[idx] = l < lam ? below : -1;
                    below = idx;
                }
        }
    }
    __syncthreads();
    // ---- counts, children, walk records (as bh_node_finalize_kernel)
    {
        unsigned int leaves = 0u, maxleaf = 0u;
        for (int v = tid; v < nn; v += kST) {
            const int l = P.nd.level[v], k = P.nd.first[v], ch = P.nd.child[v];
            int end = n;
            if (l > 0) {
                const int sh = 3 * (L - l);
                const K target = ((S.key[k] >> sh) + (K)1) << sh;
                int lo = k, hi = k + 1, step = 1;
                while (hi < n && S.key[hi] < target) {
                    lo = hi;
                    step <<= 1;
                    hi = k + step;
                }
                if (hi > n) hi = n;
                while (hi - lo > 1) {
                    const int mid = lo + ((hi - lo) >> 1);
                    if (S.key[mid] < target) lo = mid;
                    else hi = mid;
                }
                end = hi;
            }
            int nch = 0;
            if (ch >= 0) {
                const int lim = (int)S.off[l + 2];
                nch = 1;
#pragma unroll
                for (int i = 1; i < 8; i++)  // (children are consecutive: the count of those that start before the end)
                    if (ch + i < lim && P.nd.first[ch + i] < end) nch++;
            } else {
                leaves++;
                maxleaf = max(maxleaf, (unsigned int)(end - k));
            }
            P.nd.count[v] = end - k;
            P.nd.nchild[v] = nch;
            P.nd.rec[v] = make_int4(k, end - k, ch, nch);
        }
        leaves = __reduce_add_sync(BH_FULL_MASK, leaves);
        maxleaf = __reduce_max_sync(BH_FULL_MASK, maxleaf);
        if (lane == 0) {
            S.red[w][0] = leaves;
            S.red[w][1] = maxleaf;
        }
    }
    for (int j = tid; j < kST * IT / 4; j += kST) reinterpret_cast<uint32_t*>(S.flag)[j] = 0u;
    __syncthreads();
    if (w == 0) {
        const unsigned int leaves = __reduce_add_sync(BH_FULL_MASK, S.red[lane][0]);
        const unsigned int maxleaf = __reduce_max_sync(BH_FULL_MASK, S.red[lane][1]);
        if (lane == 0) {
            c->n_leaves = leaves;
            c->max_leaf = maxleaf;
        }
    }
    // ---- group flags (as bh_group_mark_kernel; one root)
    for (int v = tid; v < nn; v += kST) {
        const int4 r = P.nd.rec[v];
        if (v == 0) {
            if (r.y <= P.G) S.flag[0] = 1;
            else if (r.z < 0)
                for (int j = 0; j < r.y; j += P.G) S.flag[j] = 1;
        }
        if (r.z < 0 || r.y <= P.G) continue;
        int run_first = -1, in_run = 0;
        for (int ci = 0; ci < r.w; ci++) {
            const int4 q = P.nd.rec[r.z + ci];
            if (q.y <= P.G) {
                if (run_first >= 0 && in_run + q.y <= P.G) {
                    in_run += q.y;
                } else {
                    if (run_first >= 0) S.flag[run_first] = 1;
                    run_first = q.x;
                    in_run = q.y;
                }
            } else {
                if (run_first >= 0) S.flag[run_first] = 1;
                run_first = -1;
                in_run = 0;
                if (q.z < 0)
                    for (int j = 0; j < q.y; j += P.G) S.flag[q.x + j] = 1;
            }
        }
        if (run_first >= 0) S.flag[run_first] = 1;
    }
    __syncthreads();
    // ---- groups (as bh_flag_write_kernel)
    {
        unsigned int s = 0u;
        int first = n;  // the thread's first flag
#pragma unroll 1
        for (int i = IT - 1; i >= 0; i--)
            if (S.flag[k0 + i]) {
                s++;
                first = k0 + i;
            }
        unsigned int incl = s;
        int next = first;  // first flag of this or a later lane
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int t = __shfl_up_sync(BH_FULL_MASK, incl, o);
            if (lane >= o) incl += t;
            const int u = __shfl_down_sync(BH_FULL_MASK, next, o);
            if (lane + o < 32) next = min(next, u);
        }
        if (lane == 31) S.wtot[0][w] = incl;
        if (lane == 0) S.next[w] = next;
        next = __shfl_down_sync(BH_FULL_MASK, next, 1);
        if (lane == 31) next = n;
        __syncthreads();
        unsigned int idx = incl;
        for (int i = 0; i < w; i++) idx += S.wtot[0][i];
        for (int i = w + 1; i < kSW; i++) next = min(next, S.next[i]);
        if (tid == kST - 1) c->n_groups = idx;
#pragma unroll 1
        for (int i = IT - 1; i >= 0; i--)
            if (S.flag[k0 + i]) {
                idx--;
                P.g_first[idx] = k0 + i;
                P.g_count[idx] = next - (k0 + i);
                next = k0 + i;
            }
    }
}

template <int CURVE, typename K, int IT>
static bool bh_small_launch(const SmallParams& P, cudaStream_t s)
{
    auto kern = bh_small_build_kernel<CURVE, K, IT>;
    constexpr size_t smem = sizeof(SmallSmem<K, IT>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
    return bh_launch_after(kern, 1, kST, smem, s, P) == cudaSuccess;
}
template <int CURVE>
static bool bh_small_dispatch(const SmallParams& P, bool deep, cudaStream_t s)
{
    if (deep) return bh_small_launch<CURVE, bh_key64, 4>(P, s);
    return P.n <= 4 * kST ? bh_small_launch<CURVE, uint32_t, 4>(P, s) : bh_small_launch<CURVE, uint32_t, 8>(P, s);
}

bool launch_small_build(const float4* pos, int n, int n_leaf, int G, int curve, bool deep, const bh_nodes& nd,
                        int64_t node_cap, void* keys, uint32_t* vals, float4* pos_s, int32_t* g_first, int32_t* g_count,
                        bh_dev_ctrl* ctrl, cudaStream_t s)
{
    SmallParams P;
    P.pos = pos;
    P.n = n;
    P.n_leaf = n_leaf;
    P.G = G;
    P.node_cap = (long long)node_cap;
    P.nd = nd;
    P.keys = keys;
    P.vals = vals;
    P.pos_s = pos_s;
    P.g_first = g_first;
    P.g_count = g_count;
    P.ctrl = ctrl;
    return curve == BH_CURVE_HILBERT ? bh_small_dispatch<BH_CURVE_HILBERT>(P, deep, s)
                                     : bh_small_dispatch<BH_CURVE_MORTON>(P, deep, s);
}

}  // namespace bh
