// bh_internal.cuh -- device-side layout shared by the kernels of libbhtree.
//
// Everything here belongs to the CUDA library; nothing is shared with the CPU
// oracle.  Tree conventions (Sec. 4.1, Sec. 5 of the paper, with this
// library's readings):
//   * keys of 10 bits per axis (30-bit, uint32) or 21 bits per axis (63-bit,
//     uint64), x in the high bit of each triple, Morton or Peano-Hilbert order;
//   * node = non-empty cell of the 2^l grid (l = 0..L, L = 10 or 21) whose
//     parent cell holds more than n_leaf particles; leaf = holds <= n_leaf
//     particles or l == L;
//   * nodes are stored breadth first (sorted by level, then first particle),
//     so the children of a node are contiguous.
#pragma once

#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/bhtree.h"

#define BH_MAX_LEVEL 10        // deepest level of 30-bit keys
#define BH_MAX_LEVEL_DEEP 21   // deepest level of 63-bit keys
#define BH_LEVEL_SLOTS 23      // level-indexed arrays: levels 0..21 and the total
#define BH_FULL_MASK 0xffffffffu

// ------------------------------------------------------------------ control
// One control block per context, in device memory.  Reset at every
// tree_build by bh_init_kernel (tree_force resets its own counters).
struct bh_dev_ctrl {
    unsigned int minmax[6];      // ordered-uint encoded min x,y,z then max x,y,z
    float box[4];                // xmin, ymin, zmin, L  (written by the keys kernel)
    float inv;                   // 1024 / L
    unsigned int status;         // first device-side error, as -BH_ERR_* (0 = ok)
    unsigned int abort;          // set with status: waiting kernels give up early
    unsigned int hist[8][256];   // upfront digit histograms of the sort passes (4 or 8)
    unsigned int tile_ctr[8];    // onesweep tile tickets, one per pass
    unsigned int level_total[BH_LEVEL_SLOTS];
    unsigned int level_offset[BH_LEVEL_SLOTS];  // first node of each level; entries past the
                                                // deepest level hold the node count
    unsigned int n_nodes;        // node count of the last build
    unsigned int n_leaves;
    unsigned int max_leaf;
    unsigned int n_groups;
    unsigned int group_ctr;      // walk work queue
    unsigned long long n_pp;
    unsigned long long n_pc;
    unsigned long long cum_pp;   // since context creation (never reset)
    unsigned long long cum_pc;
    unsigned int build_seq;      // builds since the block was zeroed (never reset): the sort
                                 // passes of build b use look-back epochs 8 b + 1 .. 8 b + 8
    unsigned int scan_done;      // level-scan blocks finished (the last one writes the offsets)
    unsigned int cost_count[16]; // groups of each cost class (bh_group_order_kernel)
    unsigned int cost_taken[16];
    unsigned long long sph_like; // neighbour search: candidates that its sample of groups expects
    unsigned int sph_samples;
    unsigned int pad[3];
};

// Record a device-side error (first one wins) and raise the abort flag.
__device__ __forceinline__ void bh_set_error(bh_dev_ctrl* c, int code)
{
    atomicCAS(&c->status, 0u, (unsigned int)(-code));
    atomicExch(&c->abort, 1u);
}

// Order-preserving map float -> uint (for atomicMin/Max on floats).
__device__ __forceinline__ unsigned int bh_f2ord(float f)
{
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float bh_ord2f(unsigned int u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Key width: 30-bit keys (10 levels, 4 sort passes of 8 bits) or 63-bit keys
// (21 levels, 8 passes).
template <typename K>
struct bh_key_traits;
template <>
struct bh_key_traits<uint32_t> {
    static constexpr int kMaxLevel = BH_MAX_LEVEL;
    static constexpr int kPasses = 4;
};
template <>
struct bh_key_traits<unsigned long long> {
    static constexpr int kMaxLevel = BH_MAX_LEVEL_DEEP;
    static constexpr int kPasses = 8;
};
typedef unsigned long long bh_key64;

// Spread the low 10 bits of v to every third bit (bit k -> bit 3k).
__device__ __forceinline__ unsigned int bh_spread3(unsigned int v)
{
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}
// Inverse of bh_spread3.
__device__ __forceinline__ unsigned int bh_compact3(unsigned int v)
{
    v &= 0x09249249u;
    v = (v | (v >> 2)) & 0x030c30c3u;
    v = (v | (v >> 4)) & 0x0300f00fu;
    v = (v | (v >> 8)) & 0x030000ffu;
    v = (v | (v >> 16)) & 0x000003ffu;
    return v;
}
// 21-bit versions for 63-bit keys: the same doubling steps on 64-bit words.
__device__ __forceinline__ unsigned long long bh_spread3_21(unsigned int v32)
{
    unsigned long long v = v32 & 0x1fffffu;
    v = (v | (v << 32)) & 0x001f00000000ffffull;
    v = (v | (v << 16)) & 0x001f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}
__device__ __forceinline__ unsigned int bh_compact3_21(unsigned long long v)
{
    v &= 0x1249249249249249ull;
    v = (v | (v >> 2)) & 0x10c30c30c30c30c3ull;
    v = (v | (v >> 4)) & 0x100f00f00f00f00full;
    v = (v | (v >> 8)) & 0x001f0000ff0000ffull;
    v = (v | (v >> 16)) & 0x001f00000000ffffull;
    v = (v | (v >> 32)) & 0x00000000001fffffull;
    return (unsigned int)v;
}
__device__ __forceinline__ uint32_t bh_spread3_k(unsigned int v, uint32_t) { return bh_spread3(v); }
__device__ __forceinline__ bh_key64 bh_spread3_k(unsigned int v, bh_key64) { return bh_spread3_21(v); }
__device__ __forceinline__ unsigned int bh_compact3_k(uint32_t v) { return bh_compact3(v); }
__device__ __forceinline__ unsigned int bh_compact3_k(bh_key64 v) { return bh_compact3_21(v); }

// Peano-Hilbert index of a cell (B = 10 or 21 bits per axis), the ordering
// Sec. 5 names as better than Morton's.  Skilling's construction
// ("Programming the Hilbert curve", 2004): from the top level down, the bits
// below the level are reflected in x when an axis has the level's bit set,
// else exchanged between x and that axis; the three words are then
// Gray-coded and interleaved as a Morton key (x in the high bit of each triple).
template <typename K>
__device__ __forceinline__ K bh_hilbert3(unsigned int x, unsigned int y, unsigned int z)
{
    constexpr int B = bh_key_traits<K>::kMaxLevel;
#pragma unroll
    for (int lv = B - 1; lv >= 1; lv--) {
        const unsigned int bit = 1u << lv, below = bit - 1u;
        if (x & bit) x ^= below;
        if (y & bit) {
            x ^= below;
        } else {
            const unsigned int d = (x ^ y) & below;
            x ^= d;
            y ^= d;
        }
        if (z & bit) {
            x ^= below;
        } else {
            const unsigned int d = (x ^ z) & below;
            x ^= d;
            z ^= d;
        }
    }
    y ^= x;
    z ^= y;
    unsigned int g = 0u;
#pragma unroll
    for (int lv = B - 1; lv >= 1; lv--)
        if (z & (1u << lv)) g ^= (1u << lv) - 1u;
    x ^= g;
    y ^= g;
    z ^= g;
    return (bh_spread3_k(x, K()) << 2) | (bh_spread3_k(y, K()) << 1) | bh_spread3_k(z, K());
}
// Cell of a Peano-Hilbert index (inverse of bh_hilbert3).
template <typename K>
__device__ __forceinline__ void bh_hilbert3_cell(K h, unsigned int& x, unsigned int& y, unsigned int& z)
{
    constexpr int B = bh_key_traits<K>::kMaxLevel;
    x = bh_compact3_k((K)(h >> 2));
    y = bh_compact3_k((K)(h >> 1));
    z = bh_compact3_k(h);
    const unsigned int g = z >> 1;
    z ^= y;
    y ^= x;
    x ^= g;
#pragma unroll
    for (int lv = 1; lv <= B - 1; lv++) {
        const unsigned int bit = 1u << lv, below = bit - 1u;
        if (z & bit) {
            x ^= below;
        } else {
            const unsigned int d = (x ^ z) & below;
            x ^= d;
            z ^= d;
        }
        if (y & bit) {
            x ^= below;
        } else {
            const unsigned int d = (x ^ y) & below;
            x ^= d;
            y ^= d;
        }
        if (x & bit) x ^= below;
    }
}
// Key of a cell, and cell of a key, for the context's order.
template <int CURVE, typename K>
__device__ __forceinline__ K bh_key_of(unsigned int x, unsigned int y, unsigned int z)
{
    return CURVE == BH_CURVE_HILBERT ? bh_hilbert3<K>(x, y, z)
                                     : (bh_spread3_k(x, K()) << 2) | (bh_spread3_k(y, K()) << 1) |
                                           bh_spread3_k(z, K());
}
template <typename K>
__device__ __forceinline__ void bh_cell_of(K key, int curve, unsigned int& x, unsigned int& y, unsigned int& z)
{
    if (curve == BH_CURVE_HILBERT) {
        bh_hilbert3_cell<K>(key, x, y, z);
    } else {
        x = bh_compact3_k((K)(key >> 2));
        y = bh_compact3_k((K)(key >> 1));
        z = bh_compact3_k(key);
    }
}

// Deepest level whose cell holds both keys (0..L); keys of one cell share
// their top 3*l bits.
__device__ __forceinline__ int bh_common_level(unsigned int a, unsigned int b)
{
    const unsigned int x = a ^ b;
    if (x == 0u) return BH_MAX_LEVEL;
    return (BH_MAX_LEVEL - 1) - (31 - __clz((int)x)) / 3;
}
__device__ __forceinline__ int bh_common_level(unsigned long long a, unsigned long long b)
{
    const unsigned long long x = a ^ b;
    if (x == 0ull) return BH_MAX_LEVEL_DEEP;
    return (BH_MAX_LEVEL_DEEP - 1) - (63 - __clzll((long long)x)) / 3;
}



// Root cube from the reduced bounds (same rule as the build's first kernel).
__device__ __forceinline__ void bh_box_from_minmax(const unsigned int* mm, float* box, float* inv)
{
    const float lo0 = bh_ord2f(mm[0]), lo1 = bh_ord2f(mm[1]), lo2 = bh_ord2f(mm[2]);
    const float hi0 = bh_ord2f(mm[3]), hi1 = bh_ord2f(mm[4]), hi2 = bh_ord2f(mm[5]);
    float L = __fsub_rn(hi0, lo0);
    const float L1 = __fsub_rn(hi1, lo1), L2 = __fsub_rn(hi2, lo2);
    if (L1 > L) L = L1;
    if (L2 > L) L = L2;
    float iv = __fdiv_rn(1024.0f, L);
    if (!(L > 0.0f) || !isfinite(iv)) {
        L = 1.0f;
        iv = 1024.0f;
    }
    box[0] = lo0;
    box[1] = lo1;
    box[2] = lo2;
    box[3] = L;
    *inv = iv;
}

// ---------------------------------------------------------- warp helpers
__device__ __forceinline__ unsigned int bh_lanemask_lt()
{
    unsigned int m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Lanes whose 8-bit digit d equals this lane's, among the lanes with ok.
// Eight ballots; a match instruction on the digit was slower (build of 2^24
// particles 1280 -> 1229 us, of 2^21 with 63-bit keys 428 -> 406 us on GB300).
__device__ __forceinline__ unsigned int bh_match_digit(unsigned int d, bool ok)
{
    unsigned int peers = __ballot_sync(BH_FULL_MASK, ok);
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const unsigned int set = __ballot_sync(BH_FULL_MASK, d & (1u << b));
        peers &= (d & (1u << b)) ? set : ~set;
    }
    return peers;
}

// Barrier of all threads of a cluster; what each wrote before it is visible to all after it.
__device__ __forceinline__ void bh_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ int bh_warp_incl_scan(int v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(BH_FULL_MASK, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// 32-byte FP64 vector (x, y, z, w)
struct __align__(32) bh_double4 {
    double x, y, z, w;
};

// ------------------------------------------------------------- node arrays
// Node record read by the walk: first particle, count, first child (-1 for
// leaves), number of children.
struct bh_nodes {
    int32_t* first;
    int32_t* count;
    int32_t* child;
    int32_t* nchild;
    uint8_t* level;
    int4* rec;        // (first, count, child, nchild) packed for the walk
    float4* com_m;    // centre of mass, mass
    float* seff;      // S_eff of Eq. (2)
    float4* quad;     // 2 per node: (xx, yy, zz, xy), (xz, yz, 1.5 T, 0.5 T)
    bh_double4* com64;   // FP64 centre of mass + mass (nodes above the FP64 threshold)
    double* quad64;   // 6 per node (FP64 nodes, order 2)
    // walk records for the TMA-staged walk (nullptr: not kept): one contiguous
    // record per node, so a range of siblings is one bulk copy.  float4 0 =
    // (centre of mass, M); float4 1 = (first, count, child << 3 | (nchild - 1)
    // or -1 for a leaf, S_eff) as bits; order 2 adds the two quad float4s;
    // one float4 of padding makes the record an odd number of float4s, so
    // that 8 lanes reading records i..i+7 from shared memory hit 8 distinct
    // bank quads (no conflicts).
    float4* wrec = nullptr;
};

// float4s per walk record (with its padding)
__host__ __device__ constexpr int bh_wrec_f4(int order) { return order >= 2 ? 5 : 3; }

// ------------------------------------------------- programmatic launch order
// A kernel launched by bh_launch_after starts while its predecessor in the
// stream still runs: its blocks come up and then wait in bh_after_previous()
// until the predecessor has finished and its writes are visible.  Every such
// kernel calls it before it touches memory that the library or the caller
// writes, so the order of the stream is kept; bh_let_next_start() allows the
// successor's blocks to come up.
template <class T>
__device__ __forceinline__ void bh_reload(T& p)
{
    size_t g = __cvta_generic_to_global(p);
    asm volatile("" : "+l"(g));
    p = static_cast<T>(__cvta_global_to_generic(g));
}
// p: the kernel's __restrict__ pointers.  Loads through such a pointer may be
// taken for loads of constant memory and moved over the wait; the pointers
// are made unknown after it, which ties every load to its place, but not that
// they point to global memory: without that, loads wait for stores to shared
// memory before them (bh_levels_kernel, 16384 particles in 256 systems, 14.2 us
// against 7.3; build and moments of 2^20 290 against 287 us).
template <class... T>
__device__ __forceinline__ void bh_after_previous(T&... p)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (bh_reload(p), ...);
}
__device__ __forceinline__ void bh_let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t bh_launch_after(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...);
}

// --------------------------------------------------------------- launches
// (bodies in the .cu files; all are stream-ordered and take device pointers)
namespace bh {

constexpr int kSortThreads = 512;       // threads of an onesweep block, passes 1-3 (30-bit keys)
constexpr int kSortThreadsFirst = 256;  // threads of pass 0 (30-bit keys: 16 keys per thread)
constexpr int kSortThreadsDeep = 256;   // threads of an onesweep block (63-bit keys)
constexpr int kLookbackBatch = 4;       // predecessors read per look-back step
constexpr int kSortTile = 4096;         // keys per tile (30-bit keys)
constexpr int kSortTileDeep = 2048;     // keys per tile (63-bit keys)
constexpr int kLevelTile = 2048;                       // positions per node-build block
constexpr int kFlagTile = 4096;                        // positions per group-compaction block

void launch_init(bh_dev_ctrl* ctrl, cudaStream_t s);
void launch_bbox(const float4* pos, int n, bh_dev_ctrl* ctrl, int grid, cudaStream_t s);
// keys: uint32_t[n] (30-bit keys) or, with deep, bh_key64[n] (63-bit keys)
void launch_keys(const float4* pos, int n, bh_dev_ctrl* ctrl, void* keys, int curve, bool deep, int grid,
                 cudaStream_t s);
void launch_sort(void* keys, void* keys_alt, uint32_t* vals, uint32_t* vals_alt, const float4* pos, float4* pos_s,
                 int n, unsigned long long* lookback, bh_dev_ctrl* ctrl, bool deep,
                 cudaStream_t s);
// sys / sys_off / sys_box: several independent systems (system of each
// Morton position, first particle of each system + total, root cube of each);
// null for a single system.
// dl: uint16_t[n] scratch; blk_lvl: (deepest level + 1) * ceil(n / kLevelTile) words
// flags: cleared for launch_groups (padded to whole kFlagTile blocks)
void launch_tree(const void* keys, bool deep, int n, int n_leaf, uint16_t* dl, uint32_t* blk_lvl, uint8_t* flags,
                 const bh_nodes& nd, int64_t node_cap, bh_dev_ctrl* ctrl, int grid, cudaStream_t s,
                 const uint32_t* sys = nullptr, const int32_t* sys_off = nullptr);
// g_order (n words): the groups by falling cost, if `ordered`
void launch_groups(const bh_nodes& nd, int n, int G, uint8_t* flags, uint32_t* blk, int32_t* g_first,
                   int32_t* g_count, int32_t* g_order, bool ordered, bh_dev_ctrl* ctrl, int grid, cudaStream_t s);
void launch_moments(const float4* pos_s, const void* keys, bool deep, const bh_nodes& nd, int order,
                    float theta, int fp64_threshold, int curve, int n, bh_dev_ctrl* ctrl, int grid, cudaStream_t s,
                    const uint32_t* sys = nullptr, const float4* sys_box = nullptr);
// Whether all levels' moments take one launch, and the launches of a set's moments.
inline bool bh_moments_small(int n) { return n <= 8192; }
inline int launches_moments(int n, bool deep) { return bh_moments_small(n) ? 1 : (deep ? 22 : 11) + 1; }  // large leaves, levels
// The whole build of a small set in one launch (false: the launch failed); the
// group order is not made (see bh_groups_ordered).
inline bool bh_small_set(int n, bool deep) { return n <= (deep ? 4096 : 8192); }
bool launch_small_build(const float4* pos, int n, int n_leaf, int G, int curve, bool deep, const bh_nodes& nd,
                        int64_t node_cap, void* keys, uint32_t* vals, float4* pos_s, int32_t* g_first, int32_t* g_count,
                        bh_dev_ctrl* ctrl, cudaStream_t s);
// What the walks are to expect: the particles, the largest system of a batched
// call (0: there is one system) and about how many groups: measured 0.65-0.75 G particles each, a
// whole system where it is no larger than a group, and one more in every other.
struct WalkSet {
    int n, largest = 0;
    double groups;
    WalkSet(int n_, int G) : n(n_), groups(n_ / (0.65 * G)) {}
    WalkSet(int n_, int largest_, double groups_) : n(n_), largest(largest_), groups(groups_) {}
    static double of_system(long long n, int G) { return n <= 0 ? 0.0 : n <= G ? 1.0 : n / (0.65 * G) + 1.0; }
    // small systems have short walks (see bh_team_warps); `below`: particles of the largest
    bool short_walks(int below) const { return largest > 0 && largest < below && largest < n; }
};
// Whether the groups are listed by cost for the walks (a launch, 4 us): not where
// all of them are walked at once and their order means little, by two blocks per
// SM or, where walks are short, 16 warps.
inline bool bh_groups_ordered(const WalkSet& set)
{
    return set.n > 16384 && set.groups > (set.short_walks(1024) ? 1600 : 200) / 0.65;
}
// One CTA per system: root cube, keys, stable radix sort and gather of each
// system's particles (systems contiguous, each <= kBatchMaxN particles).
constexpr int kBatchMaxN = 65536;
void launch_batch_sort(const float4* pos, const int32_t* sys_off, int nsys, void* keys, void* keys_alt,
                       uint32_t* vals, uint32_t* vals_alt, float4* pos_s, uint32_t* sys, float4* sys_box,
                       int curve, bool deep, bh_dev_ctrl* ctrl, cudaStream_t s);
}  // namespace bh
struct bh_mlp_dev;
namespace bh {
// learned-criterion inputs of the walk (null pointer: plain Eq. 2 criterion)
struct WalkLearned {
    const float4* mfeat;
    const bh_mlp_dev* mlp;
    float theta_guard;
};
constexpr int kTeamMaxGroup = 128;  // targets per group that the team walk holds
// Warps per group of the team walk (bh_walk_team.cu), 0: a warp per group
// (bh_walk_kernel).  Eight while every group can have a block of its own at once
// (two such blocks per SM; the walker, at about 1.5 us per 32 nodes, sets the pace), else
// four (four blocks per SM, as many walkers again): clumpy 16384, G = 96, 183 us
// with four and 147 with eight, Plummer 65536, G = 64, 657 and 694.
// One launch, us, on GB300, groups taken by falling cost on both sides:
//                                     one warp   block
//   Plummer 4096, order 1, G = 64          166      75
//   clumpy 16384, order 2, G = 96          468     125
//   Plummer 70000, order 1, G = 64         798     470
//   clumpy 100003, order 2, G = 96         679     540
//   Plummer 150000, order 2, G = 96       1864    1079
//   clumpy 150000, order 2, G = 96         830     729
//   clumpy 200000, order 2, G = 128        904     977
//   clumpy 100000, order 1, G = 64         283     320
//   Plummer 120000, order 2, G = 32        505     656
//   Plummer 262144, order 2, G = 96       1101    1428
// From about one group per warp of bh_walk_kernel's grid on (16 warps per SM) the
// groups fill the GPU by themselves and the walkers' idle issue slots cost more
// than the split gains.  (Near the limit it depends on the set as well: a Plummer
// sphere, whose walks are long, still gains, clumps or few terms lose up to 13%.)
// Batched calls whose largest system has fewer than 1024 (2048) particles have short
// walks, for which a block pays only up to two (eight) groups per SM.  The largest
// counts, as a batch ends with the walks of its largest system.  Whole calls, us,
// one warp | block, order 1, G = 96: 64 systems of 256 120 | 124, 32 of 256 117 | 107, 64
// of 256 to 2000 209 | 188, 128 of 1024 227 | 252, 64 of 1024 191 | 186, 16 of 256 to 4096
// 264 | 214, 64 of 2048 303 | 315, 16 of 8192 666 | 540, 5000 of 4 to 8 221 | 281.
inline int bh_team_warps(const WalkSet& set, int G, int sm_count)
{
    const double most = set.short_walks(1024) ? 2.0 : set.short_walks(2048) ? 8.0 : 16.0;
    if (G > kTeamMaxGroup || set.groups > most * sm_count) return 0;
    return set.groups <= 4.0 * sm_count ? 8 : 4;
}

// Whether the learned walk takes four blocks per SM instead of three: more warps,
// each slower with fewer registers, pay from about two groups per warp of the
// three blocks on.  Whole calls, clumpy, order 2, ms, three | four: G = 96 5000
// 0.301 | 0.359, 50000 0.694 | 0.890, 200000 0.920 | 1.024, 400000 1.537 | 1.520; G = 64
// 100000 0.616 | 0.743, 200000 0.948 | 0.910; G = 32 50000 0.452 | 0.475, 100000 0.677 |
// 0.636.  (Above G = 96 both forms take three or fewer.)
inline bool bh_learned_four(const WalkSet& set, int G, int sm_count) { return G > 96 || set.groups > 24.0 * sm_count; }

int launch_walk(const float4* pos_s, const uint32_t* perm, const int32_t* g_first, const int32_t* g_count,
                const int32_t* g_order,
                const bh_nodes& nd, int order, int G, float eps, float4* out, bh_dev_ctrl* ctrl,
                int sm_count, int block_threads, int blocks_per_sm, const WalkSet& set, bool deep, cudaStream_t s,
                const WalkLearned* learned = nullptr, int walk_variant = 0);
// failure-path self-tests: one bounded wait that nothing satisfies
void launch_selftest_ring(bh_dev_ctrl* c, cudaStream_t s);
void launch_selftest_tma(bh_dev_ctrl* c, cudaStream_t s);
void launch_selftest_lookback(bh_dev_ctrl* c, cudaStream_t s);
int launch_direct(const float4* src, int n_src, const float4* tgt, const int64_t* self, int n_tgt,
                  double eps, void* out, int precision, cudaStream_t s,
                  const float* eps_src = nullptr, const float* eps_tgt = nullptr);
void launch_kick_drift(float4* pos, float4* vel, const float4* acc, int n, float dt_kick, float dt_drift, int grid,
                       cudaStream_t s);

// kernel launches enqueued by one call of each stage (for bh_stats.launches)
// individual softening: h = eps^2 / 2 per particle (key order) and the mass-weighted mean of h per node
struct bh_soft {
    float* h = nullptr;        // n
    double2* sums = nullptr;   // per node: (sum m, sum m h)
    float* hbar = nullptr;     // per node
};
int launch_pwalk(const float4* pos_s, const uint32_t* perm, const bh_nodes& nd, int32_t* parent, int32_t* next,
                 int order, bool deep, int n, int node_cap, float eps, bool unsoftened_cells, float4* out, bh_dev_ctrl* ctrl,
                 int sm_count, cudaStream_t s, const bh_soft* soft = nullptr);
void launch_softening(const float* eps, const uint32_t* perm, const float4* pos_s, const bh_nodes& nd, int n,
                      bool deep, const bh_soft& soft, bh_dev_ctrl* ctrl, int grid, cudaStream_t s);

int launch_sph(const float4* pos_s, const uint32_t* perm, const int32_t* g_first, const int32_t* g_count,
               const bh_nodes& nd, float4* blo, float4* bhi, int G, const float* h, float h_const, int32_t* count,
               float* rho, int32_t* heavy, int n, bh_dev_ctrl* ctrl, int sm_count, int grid, int max_level, cudaStream_t s);

// launches per call (deep = 63-bit keys: 8 sort passes, 22 levels)
inline int launches_build(bool deep) { return deep ? 19 : 15; }  // init, bbox, keys, sort passes, 4 tree, 4 groups
constexpr int kLaunchesForce = 2;    // counter reset, walk
constexpr int kLaunchesPWalk = 4;    // parent links, next links, counter reset, walk
inline int launches_sph(bool deep) { return (deep ? 22 : 11) + 2; }  // node boxes per level, two walks
inline int launches_softening(bool deep) { return (deep ? 22 : 11) + 1; }  // gather, one per level

}  // namespace bh
