// bh_mlp.cu -- training and labelling kernels of the learned opening criterion.
//
// The criterion (an extension of Eq. 2's test) is trained on errors the method
// measures itself: for sampled groups the labelling kernel walks the tree
// with a permissive Eq. (2) guard and, for every node passing it, compares the
// node's particle-cell term with the direct sum over the node's particles on
// every group member, relative to the member's total acceleration.  The
// network is then fit by hand-written forward/backward kernels and Adam
// (Kingma & Ba 2015) on FP32 master weights.
#include <cmath>
#include <cstring>
#include <algorithm>

#include "bh_mlp.cuh"

namespace bh {

// ------------------------------------------------------------ features
__device__ __forceinline__ float bh_quad_aniso(const float4& q0, const float4& q1, float M, float side)
{
    // |I - (T/3) 1|_F / (M l^2) from (xx, yy, zz, xy), (xz, yz, 1.5T, 0.5T)
    const float T3 = (q0.x + q0.y + q0.z) * (1.0f / 3.0f);
    const float a = q0.x - T3, b = q0.y - T3, c = q0.z - T3;
    const float fro = sqrtf(a * a + b * b + c * c + 2.0f * (q0.w * q0.w + q1.x * q1.x + q1.y * q1.y));
    return (M > 0.f) ? fro / (M * side * side) : 0.f;
}

// Per node: (log10 M/M_tot, quadrupole anisotropy, level, log2(count)/24).
__global__ void __launch_bounds__(256) bh_mac_nodefeat_kernel(bh_nodes nd, int order, float4* __restrict__ mfeat,
                                                              const bh_dev_ctrl* __restrict__ c)
{
    const int nn = (int)c->n_nodes;
    if (nn == 0) return;
    const float mtot = nd.com_m[0].w, L = c->box[3];
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nn; v += gridDim.x * blockDim.x) {
        const float M = nd.com_m[v].w;
        const int lev = nd.level[v];
        const float side = ldexpf(L, -lev);
        float qa = 0.f;
        if (order >= 2) qa = bh_quad_aniso(nd.quad[2 * (size_t)v], nd.quad[2 * (size_t)v + 1], M, side);
        const float f2 = (M > 0.f && mtot > 0.f) ? log10f(M / mtot) : -30.0f;
        mfeat[v] = make_float4(f2, qa, (float)lev, log2f((float)nd.count[v]) * (1.0f / 24.0f));
    }
}

void launch_mac_nodefeat(const bh_nodes& nd, int order, float4* mfeat, bh_dev_ctrl* ctrl, int grid, cudaStream_t s)
{
    bh_mac_nodefeat_kernel<<<grid, 256, 0, s>>>(nd, order, mfeat, ctrl);
}

// ------------------------------------------------------------ labels
constexpr int kLabelWarps = 4;
constexpr int kLabelStack = 160;  // DFS: <= 7 pending siblings on each of 21 levels, + 8
constexpr int kLabelSlots = 8;    // members per lane (groups of up to 256)

struct LabelArgs {
    const float4* pos_s;
    const uint32_t* perm;
    const int32_t* g_first;
    const int32_t* g_count;
    const int32_t* groups;
    int n_groups;
    const int4* rec;
    const float4* com_m;
    const float* seff;
    const float4* quad;
    const float4* mfeat;
    const float4* acc_ref;
    float eps2;
    float log_floor;
    int order;
    float* X;
    float* Y;
    int32_t* pairs;
    long long cap;
    unsigned long long* count;
    bh_dev_ctrl* ctrl;
};

__global__ void __launch_bounds__(kLabelWarps * 32) bh_mac_label_kernel(LabelArgs A)
{
    __shared__ int s_stack[kLabelWarps][kLabelStack];
    __shared__ float4 s_tile[kLabelWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gw = blockIdx.x * kLabelWarps + w;
    if (gw >= A.n_groups) return;
    const int g = A.groups[gw];
    if (g < 0 || g >= (int)A.ctrl->n_groups) return;
    const int gb = A.g_first[g], gc = A.g_count[g], ge = gb + gc;
    if (gc > 32 * kLabelSlots) return;
    const float L = A.ctrl->box[3];
    float xi[kLabelSlots], yi[kLabelSlots], zi[kLabelSlots], at[kLabelSlots];
    float lo0 = INFINITY, lo1 = INFINITY, lo2 = INFINITY, hi0 = -INFINITY, hi1 = -INFINITY, hi2 = -INFINITY;
#pragma unroll
    for (int k = 0; k < kLabelSlots; k++) {
        const int o = k * 32 + lane;
        xi[k] = yi[k] = zi[k] = 0.f;
        at[k] = 1.f;
        if (o < gc) {
            const float4 p = A.pos_s[gb + o];
            xi[k] = p.x; yi[k] = p.y; zi[k] = p.z;
            const float4 a = A.acc_ref[A.perm[gb + o]];
            at[k] = sqrtf(a.x * a.x + a.y * a.y + a.z * a.z);
            lo0 = fminf(lo0, p.x); lo1 = fminf(lo1, p.y); lo2 = fminf(lo2, p.z);
            hi0 = fmaxf(hi0, p.x); hi1 = fmaxf(hi1, p.y); hi2 = fmaxf(hi2, p.z);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo0 = fminf(lo0, __shfl_xor_sync(BH_FULL_MASK, lo0, o));
        lo1 = fminf(lo1, __shfl_xor_sync(BH_FULL_MASK, lo1, o));
        lo2 = fminf(lo2, __shfl_xor_sync(BH_FULL_MASK, lo2, o));
        hi0 = fmaxf(hi0, __shfl_xor_sync(BH_FULL_MASK, hi0, o));
        hi1 = fmaxf(hi1, __shfl_xor_sync(BH_FULL_MASK, hi1, o));
        hi2 = fmaxf(hi2, __shfl_xor_sync(BH_FULL_MASK, hi2, o));
    }
    const float gcx = 0.5f * (lo0 + hi0), gcy = 0.5f * (lo1 + hi1), gcz = 0.5f * (lo2 + hi2);
    const float rg = 0.5f * sqrtf((hi0 - lo0) * (hi0 - lo0) + (hi1 - lo1) * (hi1 - lo1) + (hi2 - lo2) * (hi2 - lo2));
    int* stack = s_stack[w];
    int sp = 1;
    if (lane == 0) stack[0] = 0;
    __syncwarp();
    while (sp > 0) {
        const int v = stack[sp - 1];
        sp--;
        __syncwarp();
        const int4 r = A.rec[v];
        const float4 cm = A.com_m[v];
        const float dx = fmaxf(fmaxf(lo0 - cm.x, cm.x - hi0), 0.f);
        const float dy = fmaxf(fmaxf(lo1 - cm.y, cm.y - hi1), 0.f);
        const float dz = fmaxf(fmaxf(lo2 - cm.z, cm.z - hi2), 0.f);
        const bool member = (r.x < ge) && (r.x + r.y > gb);
        const bool guard = !member && (dx * dx + dy * dy + dz * dz > A.seff[v]);
        bool descend = !guard;
        if (guard) {
            float f[BH_MLP_NF], side;
            const bool ok = bh_mac_features(cm, A.mfeat[v], gcx, gcy, gcz, rg, L, f, side);
            float4 q0 = make_float4(0.f, 0.f, 0.f, 0.f), q1 = q0;
            if (A.order >= 2) {
                q0 = A.quad[2 * (size_t)v];
                q1 = A.quad[2 * (size_t)v + 1];
            }
            // particle-cell term on every member
            float px[kLabelSlots], py[kLabelSlots], pz[kLabelSlots];
#pragma unroll
            for (int k = 0; k < kLabelSlots; k++) {
                const float rx = xi[k] - cm.x, ry = yi[k] - cm.y, rz = zi[k] - cm.z;
                const float h2 = rx * rx + ry * ry + rz * rz + A.eps2;
                const float g1 = rsqrtf(h2), g2 = g1 * g1, g3 = g1 * g2, g5 = g3 * g2, g7 = g5 * g2;
                const float ir0 = q0.x * rx + q0.w * ry + q1.x * rz;
                const float ir1 = q0.w * rx + q0.y * ry + q1.y * rz;
                const float ir2 = q1.x * rx + q1.y * ry + q0.z * rz;
                const float q = rx * ir0 + ry * ir1 + rz * ir2;
                const float kk = q1.z * g5 - 7.5f * q * g7 - cm.w * g3;
                px[k] = kk * rx + 3.f * g5 * ir0;
                py[k] = kk * ry + 3.f * g5 * ir1;
                pz[k] = kk * rz + 3.f * g5 * ir2;
            }
            // exact sum over the node's particles (FP32 tiles, Kahan across tiles)
            float ex[kLabelSlots], ey[kLabelSlots], ez[kLabelSlots], cx[kLabelSlots], cy[kLabelSlots],
                cz[kLabelSlots];
#pragma unroll
            for (int k = 0; k < kLabelSlots; k++) ex[k] = ey[k] = ez[k] = cx[k] = cy[k] = cz[k] = 0.f;
            for (int j0 = r.x; j0 < r.x + r.y; j0 += 32) {
                const int jn = min(32, r.x + r.y - j0);
                s_tile[w][lane] = (lane < jn) ? A.pos_s[j0 + lane] : make_float4(1e18f, 1e18f, 1e18f, 0.f);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < kLabelSlots; k++) {
                    if (k * 32 >= gc) break;
                    float tx = 0.f, ty = 0.f, tz = 0.f;
                    for (int j = 0; j < 32; j++) {
                        const float4 s = s_tile[w][j];
                        const float ddx = s.x - xi[k], ddy = s.y - yi[k], ddz = s.z - zi[k];
                        const float r2 = ddx * ddx + ddy * ddy + ddz * ddz + A.eps2;
                        const float ri = rsqrtf(r2);
                        const float mr3 = s.w * ri * ri * ri;
                        tx = fmaf(mr3, ddx, tx);
                        ty = fmaf(mr3, ddy, ty);
                        tz = fmaf(mr3, ddz, tz);
                    }
                    float yv = tx - cx[k], tv = ex[k] + yv;
                    cx[k] = (tv - ex[k]) - yv; ex[k] = tv;
                    yv = ty - cy[k]; tv = ey[k] + yv;
                    cy[k] = (tv - ey[k]) - yv; ey[k] = tv;
                    yv = tz - cz[k]; tv = ez[k] + yv;
                    cz[k] = (tv - ez[k]) - yv; ez[k] = tv;
                }
                __syncwarp();
            }
            float worst = 0.f;
#pragma unroll
            for (int k = 0; k < kLabelSlots; k++) {
                if (k * 32 + lane < gc) {
                    const float ddx = px[k] - (ex[k] - cx[k]), ddy = py[k] - (ey[k] - cy[k]),
                                ddz = pz[k] - (ez[k] - cz[k]);
                    worst = fmaxf(worst, sqrtf(ddx * ddx + ddy * ddy + ddz * ddz) / at[k]);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) worst = fmaxf(worst, __shfl_xor_sync(BH_FULL_MASK, worst, o));
            const float label = log10f(fmaxf(worst, 1e-12f));
            if (ok && lane == 0) {
                const unsigned long long idx = atomicAdd(A.count, 1ull);
                if ((long long)idx < A.cap) {
                    for (int k = 0; k < BH_MLP_NF; k++) A.X[idx * BH_MLP_NF + k] = f[k];
                    A.Y[idx] = label;
                    if (A.pairs) {
                        A.pairs[2 * idx] = v;
                        A.pairs[2 * idx + 1] = g;
                    }
                }
            }
            descend = label > A.log_floor;
        }
        if (descend && r.z >= 0) {
            if (sp + r.w > kLabelStack) {
                if (lane == 0) bh_set_error(A.ctrl, BH_ERR_CAPACITY);
                return;
            }
            if (lane < r.w) stack[sp + r.w - 1 - lane] = r.z + lane;
            sp += r.w;
            __syncwarp();
        }
    }
}

// ------------------------------------------------------------ training
constexpr int kOffB1 = BH_MLP_NH * BH_MLP_NF, kOffW2 = kOffB1 + BH_MLP_NH, kOffB2 = kOffW2 + BH_MLP_NH * BH_MLP_NH,
              kOffW3 = kOffB2 + BH_MLP_NH, kOffB3 = kOffW3 + BH_MLP_NH;
constexpr int kAct = BH_MLP_NF + 4 * BH_MLP_NH + 1;  // floats of training scratch per sample (caller's buffer)
constexpr int kRow = BH_MLP_NPARAM + 1;              // a block's partial sums: gradient, loss
constexpr int kTrainBlocks = 304;                    // most blocks (rows of partial sums): two per SM

// FP32 forward of one sample per thread (training path without gradients).
__global__ void __launch_bounds__(256) bh_mlp_forward_kernel(const float* __restrict__ P, const float* __restrict__ X,
                                                             long long i0, int B, float* __restrict__ yhat)
{
    __shared__ float sp[BH_MLP_NPARAM];
    for (int i = threadIdx.x; i < BH_MLP_NPARAM; i += blockDim.x) sp[i] = P[i];
    __syncthreads();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    float x[BH_MLP_NF], h1[BH_MLP_NH];
    for (int k = 0; k < BH_MLP_NF; k++) x[k] = X[(i0 + b) * BH_MLP_NF + k];
#pragma unroll
    for (int j = 0; j < BH_MLP_NH; j++) {
        float a = sp[kOffB1 + j];
        for (int k = 0; k < BH_MLP_NF; k++) a = fmaf(sp[j * BH_MLP_NF + k], x[k], a);
        h1[j] = fmaxf(a, 0.f);
    }
    float y = sp[kOffB3];
    for (int j = 0; j < BH_MLP_NH; j++) {
        float a = sp[kOffB2 + j];
#pragma unroll
        for (int k = 0; k < BH_MLP_NH; k++) a = fmaf(sp[kOffW2 + j * BH_MLP_NH + k], h1[k], a);
        y = fmaf(sp[kOffW3 + j], fmaxf(a, 0.f), y);
    }
    yhat[b] = y;
}

// Forward, backward and the weights' gradient of a mini-batch, kSamples (32 or
// 64) at a time per block with every activation in shared memory.  Rounds are
// dealt to the blocks in turn; a block keeps the gradient sums of its rounds
// in registers and writes one row of kRow partial sums at the end.  rows == 1
// (one block): the row is the gradient itself.
//
// A step is bound by launches and the latency of its few dependent phases, not
// by its arithmetic (62 MFLOP for 8192 samples): the activations of a sample
// used to go through global memory (540 bytes) and 33 blocks read all of them
// again, each for one unit.  A step of 8192 samples on GB300, 16 steps per call:
// 127 us (forward and backward 40 us, gradient 82 us, update 4 us), then 20.6 us
// with this kernel and the sum of its rows, and 13.5 us with each of them
// launched while its predecessor runs (bh_launch_after).
template <int kSamples>
struct TrainSmem {
    float p[BH_MLP_NPARAM + 3];                      // the parameters
    float w2t[BH_MLP_NH][BH_MLP_NH];                 // W2 transposed: [input][unit]
    float w2[BH_MLP_NH][BH_MLP_NH];                  // W2: [unit][input]
    float x[kSamples][BH_MLP_NF + 1];
    float h1[kSamples][BH_MLP_NH + 1], h2[kSamples][BH_MLP_NH + 1];
    float d1[kSamples][BH_MLP_NH + 1], d2[kSamples][BH_MLP_NH + 1];
    float dy[kSamples], l[kSamples];
};

template <int kSamples>
__global__ void __launch_bounds__(256) bh_mlp_batch_grad_kernel(const float* __restrict__ P,
                                                                const float* __restrict__ X,
                                                                const float* __restrict__ Y,
                                                                const int32_t* __restrict__ order, long long i0, int B,
                                                                long long n, float under_w, float* __restrict__ rows,
                                                                float* __restrict__ loss)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem<kSamples>& S = *reinterpret_cast<TrainSmem<kSamples>*>(smem_raw);
    constexpr int kUnits = kSamples / 8;  // hidden units per thread
    const int tid = threadIdx.x;
    bh_let_next_start();
    // the first round's samples, which no kernel of this call writes, are
    // fetched before the previous step's parameters are waited for
    float t = 0.f, x0[BH_MLP_NF];
    auto fetch = [&](int b) {
        const bool in = b < B;
        const long long at = in ? (order ? (long long)order[(i0 + b) % n] : (i0 + b) % n) : 0;
        t = in ? Y[at] : 0.f;
#pragma unroll
        for (int k = 0; k < BH_MLP_NF; k++) x0[k] = in ? X[at * BH_MLP_NF + k] : 0.f;
    };
    if (tid < kSamples) fetch(blockIdx.x * kSamples + tid);
    bh_after_previous(P, rows, loss);
    for (int i = tid; i < BH_MLP_NPARAM; i += 256) S.p[i] = P[i];
    for (int i = tid; i < BH_MLP_NH * BH_MLP_NH; i += 256) {
        const float w = P[kOffW2 + i];
        S.w2[i / BH_MLP_NH][i % BH_MLP_NH] = w;
        S.w2t[i % BH_MLP_NH][i / BH_MLP_NH] = w;
    }
    const int s = tid % kSamples, u0 = tid / kSamples * kUnits;  // sample, first unit (a warp shares u0)
    // weight gradient of layer 2: units ja + 8 a, inputs ka + 8 b, samples q, q + 4, ...
    const int ja = (tid & 63) >> 3, ka = tid & 7, q = tid >> 6;
    float g2[4][4];
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) g2[a][b] = 0.f;
    float ge[2] = {0.f, 0.f};  // the thread's one or two other outputs
    const int nround = (B + kSamples - 1) / kSamples;
    for (int round = blockIdx.x; round < nround; round += gridDim.x) {
        const int b = round * kSamples + s;
        const bool in = b < B;
        __syncthreads();
        if (tid < kSamples) {
            if (round != blockIdx.x) fetch(b);
#pragma unroll
            for (int k = 0; k < BH_MLP_NF; k++) S.x[s][k] = x0[k];
        }
        __syncthreads();
        // layer 1
        {
            float x[BH_MLP_NF];
#pragma unroll
            for (int k = 0; k < BH_MLP_NF; k++) x[k] = S.x[s][k];
#pragma unroll
            for (int j = u0; j < u0 + kUnits; j++) {
                float a = S.p[kOffB1 + j];
#pragma unroll
                for (int k = 0; k < BH_MLP_NF; k++) a = fmaf(S.p[j * BH_MLP_NF + k], x[k], a);
                S.h1[s][j] = fmaxf(a, 0.f);
            }
        }
        __syncthreads();
        // layer 2
        {
            float a[kUnits];
#pragma unroll
            for (int j = 0; j < kUnits; j++) a[j] = S.p[kOffB2 + u0 + j];
#pragma unroll 8
            for (int k = 0; k < BH_MLP_NH; k++) {
                const float h = S.h1[s][k];
#pragma unroll
                for (int j = 0; j < kUnits; j += 4) {
                    const float4 w = *reinterpret_cast<const float4*>(&S.w2t[k][u0 + j]);
                    a[j] = fmaf(w.x, h, a[j]); a[j + 1] = fmaf(w.y, h, a[j + 1]);
                    a[j + 2] = fmaf(w.z, h, a[j + 2]); a[j + 3] = fmaf(w.w, h, a[j + 3]);
                }
            }
#pragma unroll
            for (int j = 0; j < kUnits; j++) S.h2[s][u0 + j] = fmaxf(a[j], 0.f);
        }
        __syncthreads();
        // output, loss and its derivative
        if (tid < kSamples) {
            float y = S.p[kOffB3];
#pragma unroll 8
            for (int k = 0; k < BH_MLP_NH; k++) y = fmaf(S.p[kOffW3 + k], S.h2[s][k], y);
            const float r = y - t, wgt = (y < t) ? under_w : 1.0f;
            S.l[s] = in ? wgt * r * r / (float)B : 0.f;
            S.dy[s] = in ? 2.0f * wgt * r / (float)B : 0.f;
        }
        __syncthreads();
        // back through layer 2 (its derivatives in registers for the thread's units, in memory for all)
        {
            const float dy = S.dy[s];
#pragma unroll
            for (int j = u0; j < u0 + kUnits; j++) S.d2[s][j] = S.h2[s][j] > 0.f ? dy * S.p[kOffW3 + j] : 0.f;
        }
        __syncthreads();
        {
            float d[kUnits];
#pragma unroll
            for (int k = 0; k < kUnits; k++) d[k] = 0.f;
#pragma unroll 8
            for (int j = 0; j < BH_MLP_NH; j++) {
                const float e = S.d2[s][j];
#pragma unroll
                for (int k = 0; k < kUnits; k += 4) {
                    const float4 w = *reinterpret_cast<const float4*>(&S.w2[j][u0 + k]);
                    d[k] = fmaf(e, w.x, d[k]); d[k + 1] = fmaf(e, w.y, d[k + 1]);
                    d[k + 2] = fmaf(e, w.z, d[k + 2]); d[k + 3] = fmaf(e, w.w, d[k + 3]);
                }
            }
#pragma unroll
            for (int k = 0; k < kUnits; k++) S.d1[s][u0 + k] = S.h1[s][u0 + k] > 0.f ? d[k] : 0.f;
        }
        // gradient of W2 (d2 and h1 are complete)
#pragma unroll 4
        for (int i = q; i < kSamples; i += 4) {
            float d[4], h[4];
#pragma unroll
            for (int a = 0; a < 4; a++) {
                d[a] = S.d2[i][ja + 8 * a];
                h[a] = S.h1[i][ka + 8 * a];
            }
#pragma unroll
            for (int a = 0; a < 4; a++)
#pragma unroll
                for (int e = 0; e < 4; e++) g2[a][e] = fmaf(d[a], h[e], g2[a][e]);
        }
        __syncthreads();
        // the other sums: W1 (192), b1 (32), b2 (32); the first 34 threads also W3, b3 and the loss
        {
            const float *f, *g;  // columns (stride NH + 1 = 33, or 7 for x)
            int gs = 0;
            if (tid < 192) { f = &S.d1[0][tid / BH_MLP_NF]; g = &S.x[0][tid % BH_MLP_NF]; gs = BH_MLP_NF + 1; }
            else if (tid < 224) { f = &S.d1[0][tid - 192]; g = nullptr; }
            else { f = &S.d2[0][tid - 224]; g = nullptr; }
            float acc0 = 0.f, acc1 = 0.f;
#pragma unroll 8
            for (int i = 0; i < kSamples; i += 2) {
                acc0 = fmaf(f[i * (BH_MLP_NH + 1)], g ? g[i * gs] : 1.0f, acc0);
                acc1 = fmaf(f[(i + 1) * (BH_MLP_NH + 1)], g ? g[(i + 1) * gs] : 1.0f, acc1);
            }
            ge[0] += acc0 + acc1;
            if (tid < BH_MLP_NH + 2) {
                acc0 = acc1 = 0.f;
                for (int i = 0; i < kSamples; i += 2) {
                    const float u = tid < BH_MLP_NH ? S.h2[i][tid] : 1.0f, w = tid < BH_MLP_NH ? S.h2[i + 1][tid] : 1.0f;
                    acc0 = fmaf(tid == BH_MLP_NH + 1 ? S.l[i] : S.dy[i], u, acc0);
                    acc1 = fmaf(tid == BH_MLP_NH + 1 ? S.l[i + 1] : S.dy[i + 1], w, acc1);
                }
                ge[1] += acc0 + acc1;
            }
        }
    }
    // the four sample slices of W2's gradient, then the row
    __syncthreads();
    float* red = &S.h1[0][0];  // [4][1024] over h1, h2, d1, d2
    static_assert(4 * kSamples * (BH_MLP_NH + 1) >= 4096, "room for the slices");
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int e = 0; e < 4; e++) red[q * 1024 + (ja + 8 * a) * BH_MLP_NH + ka + 8 * e] = g2[a][e];
    __syncthreads();
    float* row = rows + (size_t)blockIdx.x * (gridDim.x > 1 ? kRow : 0);
    for (int i = tid; i < 1024; i += 256) row[kOffW2 + i] = (red[i] + red[1024 + i]) + (red[2048 + i] + red[3072 + i]);
    if (tid < 224) row[tid] = ge[0];              // W1, b1 lie in this order
    else row[kOffB2 + tid - 224] = ge[0];
    if (tid < BH_MLP_NH) row[kOffW3 + tid] = ge[1];
    else if (tid == BH_MLP_NH) row[kOffB3] = ge[1];
    else if (tid == BH_MLP_NH + 1) {
        if (gridDim.x > 1) row[BH_MLP_NPARAM] = ge[1];
        else if (loss) *loss += ge[1];
    }
}

// Sum of the rows of partial sums (nrow >= 1), 32 columns per block; then the
// gradient (grad) or one Adam step (m, v, P).  loss += the rows' losses.
__global__ void __launch_bounds__(256) bh_mlp_update_kernel(const float* __restrict__ rows, int nrow,
                                                            float* __restrict__ grad, float* __restrict__ loss,
                                                            float* __restrict__ P, float* __restrict__ m,
                                                            float* __restrict__ v, long long t, float lr, float b1,
                                                            float b2, float eps)
{
    __shared__ float red[8][33];
    const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + c;
    bh_let_next_start();
    bh_after_previous(rows, grad, loss, P, m, v);
    float a0 = 0.f, a1 = 0.f;
    if (k < (nrow > 1 ? kRow : BH_MLP_NPARAM)) {  // (a single row is a bare gradient)
        int r = w;
#pragma unroll 8
        for (; r + 8 < nrow; r += 16) {
            a0 += rows[(size_t)r * kRow + k];
            a1 += rows[(size_t)(r + 8) * kRow + k];
        }
        if (r < nrow) a0 += rows[(size_t)r * kRow + k];
    }
    red[w][c] = a0 + a1;
    __syncthreads();
    if (w != 0 || k >= kRow) return;
    float g = 0.f;
#pragma unroll
    for (int i = 0; i < 8; i++) g += red[i][c];
    if (k == BH_MLP_NPARAM) {
        if (loss && nrow > 1) *loss += g;
        return;
    }
    if (grad) grad[k] = g;
    if (!P) return;
    const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
    const float mk = b1 * m[k] + (1.f - b1) * g;
    const float vk = b2 * v[k] + (1.f - b2) * g * g;
    m[k] = mk;
    v[k] = vk;
    P[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

// Inference path: the walk's tensor-core network, 32 samples per warp.
__global__ void __launch_bounds__(128) bh_mlp_mma_forward_kernel(const bh_mlp_dev* __restrict__ Wg,
                                                                 const float* __restrict__ X, long long n,
                                                                 float* __restrict__ y)
{
    __shared__ bh_mlp_dev W;
    __shared__ uint32_t xs[4][32 * 8];
    for (int i = threadIdx.x; i < (int)(sizeof(bh_mlp_dev) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t*>(&W)[i] = reinterpret_cast<const uint32_t*>(Wg)[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long s = ((long long)blockIdx.x * 4 + w) * 32 + lane;
    float f[BH_MLP_NF];
    for (int k = 0; k < BH_MLP_NF; k++) f[k] = (s < n) ? X[s * BH_MLP_NF + k] : 0.f;
    const float v = bh_mlp_warp(W, xs[w], f);
    if (s < n) y[s] = v;
}

// ------------------------------------------------------------ host side
static uint16_t bf16_bits(float x)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(x);
    uint16_t u;
    std::memcpy(&u, &b, 2);
    return u;
}

void mlp_pack(const float* P, const float* fmin, const float* fmax, float ltau, float theta_fb, bh_mlp_dev* out)
{
    std::memset(out, 0, sizeof(*out));
    auto pack = [](float lo, float hi) { return (uint32_t)bf16_bits(lo) | ((uint32_t)bf16_bits(hi) << 16); };
    // word w of a row of K = 32 holds k = 2w, 2w + 1; k-step s, lane t of the
    // quad takes words 8s + t and 8s + t + 4
    auto word32 = [&](int off, int w) { return pack(P[off + 2 * w], P[off + 2 * w + 1]); };
    for (int j = 0; j < 32; j++) {
        for (int w = 0; w < 4; w++) {
            const int k0 = 2 * w, k1 = 2 * w + 1;
            out->w1[j][w] = pack(k0 < BH_MLP_NF ? P[j * BH_MLP_NF + k0] : 0.f, k1 < BH_MLP_NF ? P[j * BH_MLP_NF + k1] : 0.f);
        }
        for (int ks = 0; ks < 2; ks++)
            for (int t = 0; t < 4; t++)
                out->w2[j][ks][t] = make_uint2(word32(kOffW2 + j * 32, 8 * ks + t), word32(kOffW2 + j * 32, 8 * ks + t + 4));
        out->b1[j] = P[kOffB1 + j];
        out->b2[j] = P[kOffB2 + j];
    }
    for (int ks = 0; ks < 2; ks++)
        for (int t = 0; t < 4; t++)
            out->w3[0][ks][t] = make_uint2(word32(kOffW3, 8 * ks + t), word32(kOffW3, 8 * ks + t + 4));
    out->b3[0] = P[kOffB3];
    for (int k = 0; k < 8; k++) {
        out->fmin[k] = k < BH_MLP_NF ? fmin[k] : -INFINITY;
        out->fmax[k] = k < BH_MLP_NF ? fmax[k] : INFINITY;
    }
    out->ltau = ltau;
    out->theta_fb = theta_fb;
}

int mac_label(const float4* pos_s, const uint32_t* perm, const int32_t* g_first, const int32_t* g_count,
              const int32_t* groups, int n_groups, const bh_nodes& nd, const float4* mfeat, const float4* acc_ref,
              float eps, float log_floor, int order, float* X, float* Y, int32_t* pairs, long long cap,
              unsigned long long* count, bh_dev_ctrl* ctrl, cudaStream_t s)
{
    if (n_groups <= 0) return BH_OK;
    LabelArgs a;
    a.pairs = pairs;
    a.pos_s = pos_s;
    a.perm = perm;
    a.g_first = g_first;
    a.g_count = g_count;
    a.groups = groups;
    a.n_groups = n_groups;
    a.rec = nd.rec;
    a.com_m = nd.com_m;
    a.seff = nd.seff;
    a.quad = nd.quad;
    a.mfeat = mfeat;
    a.acc_ref = acc_ref;
    a.eps2 = eps * eps;
    a.log_floor = log_floor;
    a.order = order;
    a.X = X;
    a.Y = Y;
    a.cap = cap;
    a.count = count;
    a.ctrl = ctrl;
    bh_mac_label_kernel<<<(n_groups + kLabelWarps - 1) / kLabelWarps, kLabelWarps * 32, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? BH_OK : BH_ERR_CUDA;
}

// A block's share of a mini-batch of B samples per round, and the blocks.
struct TrainPlan {
    void (*kernel)(const float*, const float*, const float*, const int32_t*, long long, int, long long, float, float*,
                   float*);
    int blocks;
    size_t smem;
};

template <int kSamples>
static TrainPlan train_plan(long long B)
{
    TrainPlan t{bh_mlp_batch_grad_kernel<kSamples>, (int)std::min<long long>((B + kSamples - 1) / kSamples, kTrainBlocks),
                sizeof(TrainSmem<kSamples>)};
    if (cudaFuncSetAttribute(t.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)t.smem) != cudaSuccess)
        t.blocks = 0;
    return t;
}

// 32 samples per block halve each phase of a round, and give twice the rows to
// sum.  They pay while every block has an SM to itself (152 x 32 = 4864
// samples).  Microseconds per step with 32 | 64 on GB300: 512 samples 10.5 |
// 13.0, 2048 11.6 | 13.6, 4096 10.8 | 14.4, 5000 16.0 | 14.4, 8192 16.4 | 13.5.
static TrainPlan train_plan_for(long long B)
{
    return B <= kTrainBlocks / 2 * 32 ? train_plan<32>(B) : train_plan<64>(B);
}

int mlp_train(const float* X, const float* Y, const int32_t* order, long long n, float* P, float* adam_m,
              float* adam_v, float* work, long long work_floats, long long steps, int batch, float lr,
              float under_w, float* loss, long long t0, cudaStream_t s)
{
    if (batch < 1 || n < 1 || steps < 0) return BH_ERR_INVALID;
    const long long need = (long long)batch * kAct + BH_MLP_NPARAM;
    if (work_floats < need) return BH_ERR_TOO_LARGE;
    const TrainPlan plan = train_plan_for(batch);
    if (plan.blocks == 0) return BH_ERR_CUDA;
    for (long long st = 0; st < steps; st++) {
        const long long i0 = ((t0 + st) * (long long)batch) % n;
        float* l = loss ? loss + st : nullptr;
        if (st == 0)  // its samples may still be in the making
            plan.kernel<<<plan.blocks, 256, plan.smem, s>>>(P, X, Y, order, i0, batch, n, under_w, work, l);
        else
            bh_launch_after(plan.kernel, plan.blocks, 256, plan.smem, s, P, X, Y, order, i0, batch, n, under_w, work, l);
        bh_launch_after(bh_mlp_update_kernel, (kRow + 31) / 32, 256, 0, s, work, plan.blocks, nullptr, l, P, adam_m,
                        adam_v, t0 + st + 1, lr, 0.9f, 0.999f, 1e-8f);
    }
    return cudaGetLastError() == cudaSuccess ? BH_OK : BH_ERR_CUDA;
}

int mlp_grad(const float* P, const float* X, const float* Y, long long n, float under_w, float* work,
             long long work_floats, float* grad, float* loss, cudaStream_t s)
{
    const long long need = n * kAct;
    if (work_floats < need) return BH_ERR_TOO_LARGE;
    if (n > (1ll << 30)) return BH_ERR_TOO_LARGE;
    // rows of partial sums fit in n * kAct floats whenever there are two or more (n > 32)
    const TrainPlan plan = train_plan_for(n);
    if (plan.blocks == 0) return BH_ERR_CUDA;
    plan.kernel<<<plan.blocks, 256, plan.smem, s>>>(P, X, Y, nullptr, 0, (int)n, n, under_w,
                                                    plan.blocks > 1 ? work : grad, loss);
    if (plan.blocks > 1)
        bh_mlp_update_kernel<<<(kRow + 31) / 32, 256, 0, s>>>(work, plan.blocks, grad, loss, nullptr, nullptr, nullptr,
                                                              1, 0.f, 0.9f, 0.999f, 1e-8f);
    return cudaGetLastError() == cudaSuccess ? BH_OK : BH_ERR_CUDA;
}

int mlp_forward(const float* P, const bh_mlp_dev* Wdev, const float* X, long long n, float* y, int precision,
                cudaStream_t s)
{
    if (n <= 0) return BH_OK;
    if (precision == 16) {
        bh_mlp_mma_forward_kernel<<<(int)((n + 127) / 128), 128, 0, s>>>(Wdev, X, n, y);
    } else {
        // FP32 training forward, in chunks the kernel's int batch can index
        for (long long i0 = 0; i0 < n; i0 += (1ll << 30)) {
            const int B = (int)std::min<long long>(n - i0, 1ll << 30);
            bh_mlp_forward_kernel<<<(B + 255) / 256, 256, 0, s>>>(P, X, i0, B, y + i0);
        }
    }
    return cudaGetLastError() == cudaSuccess ? BH_OK : BH_ERR_CUDA;
}

}  // namespace bh
