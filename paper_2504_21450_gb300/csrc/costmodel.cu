// costmodel.cu -- the learned cost model of libvlgt: per-tile features of the sparse
// phase space, a small MLP (8 -> 64 -> 64 -> 1, ReLU) with its own forward, backward
// and Adam kernels, and the capacity estimate that pre-sizes the block pools of a
// captured step sequence.
//
// The paper balances its spatial cells by a weight that grows with the complexity of
// each cell's velocity space (Section 2, load balancing) and notes that the coalesced
// ghost cells change that cost (Section 5).  Here the question is the same one asked
// ahead of time on one GPU: how many blocks will a region of space hold over the next
// steps.  The model predicts, per tile of edge^3 cells, log(1 + max over a horizon of
// the tile's blocks after the 27-cell union); summed over tiles this sizes the pools.
// It never touches f: it changes only how much memory a captured sequence reserves.
//
// All reductions are deterministic (fixed summation order; FP64, or triples of FP32 numbers
// whose values are added in FP64), so a training run is reproducible bit for bit.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "grid.h"

namespace vlgt {

namespace {

constexpr int kIn = VL_MLP_NIN, kH = VL_MLP_NHIDDEN, kP = VL_MLP_NPARAM;
// flat parameter layout: W1[kH][kIn], b1[kH], W2[kH][kH], b2[kH], w3[kH], b3
constexpr int oW1 = 0, ob1 = oW1 + kH * kIn, oW2 = ob1 + kH, ob2 = oW2 + kH * kH, ow3 = ob2 + kH,
              ob3 = ow3 + kH;
static_assert(ob3 + 1 == kP, "parameter layout");

constexpr int kThreads = 128;
inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

// ---- features ----------------------------------------------------------------------
struct TileGeom {
    GridGeom G;
    int edge;
    int nt[3];  // tiles per dimension
};

// Per tile: active blocks (kbits of the state) and blocks of the next step's union (ubits
// of the next layout), counts[tile] = {active, union}.  A CTA takes a tile and a part of the
// block ids, so that a few hundred tiles still fill the chip (one CTA per tile took 0.80 ms
// on 216 tiles x 4096 ids, 0.14 with the ids split); integer sums, so their order does
// not matter.
__global__ void __launch_bounds__(256) k_tile_counts(TileGeom T, int ids, const uint64_t* __restrict__ kbits,
                                                     const uint64_t* __restrict__ ubits,
                                                     unsigned long long* __restrict__ counts)
{
    const GridGeom& G = T.G;
    const int tile = blockIdx.x;
    const int tc[3] = {tile % T.nt[0], (tile / T.nt[0]) % T.nt[1], tile / (T.nt[0] * T.nt[1])};
    int lo[3], ext[3];
    for (int d = 0; d < 3; d++) {
        lo[d] = tc[d] * T.edge;
        ext[d] = min(T.edge, G.n[d] - lo[d]);
    }
    // (block id, tile row) pairs, the tile's x range masked in each word
    const int rows = ext[1] * ext[2];
    const int b0 = blockIdx.y * ids, b1 = min(G.nb, b0 + ids);
    unsigned act = 0, un = 0;
    for (int i = threadIdx.x; i < (b1 - b0) * rows; i += blockDim.x) {
        const int b = b0 + i / rows;
        const int r = i % rows;
        const int64_t row = (int64_t)(lo[1] + r % ext[1]) + (int64_t)G.n[1] * (lo[2] + r / ext[1]);
        const int64_t base = (int64_t)b * G.RW + row * G.W;
        for (int x = lo[0]; x < lo[0] + ext[0];) {  // words overlapping the x range
            const int w = x >> 6;
            const int xe = min(lo[0] + ext[0], (w + 1) * 64);
            const int nbit = xe - x;
            const uint64_t m = (nbit == 64 ? ~0ull : ((1ull << nbit) - 1ull)) << (x & 63);
            act += __popcll(kbits[base + w] & m);
            un += __popcll(ubits[base + w] & m);
            x = xe;
        }
    }
    act = __reduce_add_sync(0xffffffffu, act);
    un = __reduce_add_sync(0xffffffffu, un);
    if ((threadIdx.x & 31) == 0) {
        if (act) atomicAdd(&counts[2 * tile], (unsigned long long)act);
        if (un) atomicAdd(&counts[2 * tile + 1], (unsigned long long)un);
    }
}

// Per tile: its block counts, and FP64 sums over the tile's cells of n, V_d, v_th and the
// relative density gradient, from the per-cell moments (n, nV_d, P_dd).
__global__ void __launch_bounds__(256) k_tile_features(TileGeom T, const unsigned long long* __restrict__ counts,
                                                       const double* __restrict__ mom,
                                                       float* __restrict__ feat, float* __restrict__ uni)
{
    const GridGeom& G = T.G;
    const int tile = blockIdx.x;
    const int tc[3] = {tile % T.nt[0], (tile / T.nt[0]) % T.nt[1], tile / (T.nt[0] * T.nt[1])};
    int lo[3], ext[3];
    for (int d = 0; d < 3; d++) {
        lo[d] = tc[d] * T.edge;
        ext[d] = min(T.edge, G.n[d] - lo[d]);
    }
    // per-cell moment features
    double s[6] = {0, 0, 0, 0, 0, 0};  // n, Vx, Vy, Vz, v_th, and (max) |grad n| / n
    const int ncell = ext[0] * ext[1] * ext[2];
    for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
        const int x = lo[0] + c % ext[0], y = lo[1] + (c / ext[0]) % ext[1], z = lo[2] + c / (ext[0] * ext[1]);
        const int64_t cell = x + (int64_t)G.n[0] * (y + (int64_t)G.n[1] * z);
        const double* m = mom + cell * 7;
        const double n = m[0];
        s[0] += n;
        if (n > 0.0) {
            for (int d = 0; d < 3; d++) s[1 + d] += m[1 + d] / n;
            s[4] += sqrt((m[4] + m[5] + m[6]) / (3.0 * n));
            const int xc[3] = {x, y, z};
            double g2 = 0.0;
            for (int d = 0; d < 3; d++) {
                int up[3] = {xc[0], xc[1], xc[2]}, dn[3] = {xc[0], xc[1], xc[2]};
                up[d] = wrapi(xc[d] + 1, G.n[d]);
                dn[d] = wrapi(xc[d] - 1, G.n[d]);
                const double nu = mom[(up[0] + (int64_t)G.n[0] * (up[1] + (int64_t)G.n[1] * up[2])) * 7];
                const double nd = mom[(dn[0] + (int64_t)G.n[0] * (dn[1] + (int64_t)G.n[1] * dn[2])) * 7];
                const double gd = 0.5 * (nu - nd);
                g2 += gd * gd;
            }
            s[5] = fmax(s[5], sqrt(g2) / n);
        }
    }
    // deterministic CTA reduction: warp trees, then warps in order
    __shared__ double sh[8][6];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        for (int k = 0; k < 5; k++) s[k] += __shfl_down_sync(0xffffffffu, s[k], o);
        s[5] = fmax(s[5], __shfl_down_sync(0xffffffffu, s[5], o));
    }
    if (lane == 0)
        for (int k = 0; k < 6; k++) sh[warp][k] = s[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[6] = {0, 0, 0, 0, 0, 0};
        const unsigned long long A = counts[2 * tile], U = counts[2 * tile + 1];
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            for (int k = 0; k < 5; k++) t[k] += sh[w][k];
            t[5] = fmax(t[5], sh[w][5]);
        }
        float* f = feat + (int64_t)tile * kIn;
        f[0] = (float)log1p((double)A);
        f[1] = (float)log1p((double)U);
        f[2] = (float)log1p(t[0] / ncell);
        for (int d = 0; d < 3; d++) f[3 + d] = (float)(t[1 + d] / ncell);
        f[6] = (float)(t[4] / ncell);
        f[7] = (float)t[5];
        uni[tile] = (float)U;
    }
}

// targets[t][i] = log(1 + max_{j < horizon} uni[t + j][i])
__global__ void k_cost_targets(const float* __restrict__ trace, int nsnap, int64_t ntiles, int horizon,
                               float* __restrict__ targets)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nt = nsnap - horizon + 1;
    if (i >= (int64_t)nt * ntiles) return;
    const int t = (int)(i / ntiles);
    const int64_t k = i - (int64_t)t * ntiles;
    float m = 0.0f;
    for (int j = 0; j < horizon; j++) m = fmaxf(m, trace[(int64_t)(t + j) * ntiles + k]);
    targets[i] = (float)log1p((double)m);
}

// ---- MLP -----------------------------------------------------------------------------
// A CTA of 512 threads works on batches of 16 samples with the parameters and the batch's
// activations in shared memory.  In a layer a thread owns one unit and two samples, so that
// a weight is read once for both; every dot product runs in the order of its index, so
// an output does not depend on the batch it is in.
constexpr int kMlpThreads = 512;
constexpr int kMlpBatch = 16;
constexpr int kPad = kH + 1;  // row pitch of W2: both its rows and its columns are read by a warp

struct MlpSmem {
    float w1[kH][kIn + 1], w2[kH][kPad];
    float b1[kH], b2[kH], w3[kH], b3;
    alignas(16) float x[kMlpBatch][kIn];
    alignas(16) float h1[kMlpBatch][kH], h2[kMlpBatch][kH], d1[kMlpBatch][kH], d2[kMlpBatch][kH];
    float y[kMlpBatch], dy[kMlpBatch];
};

__device__ __forceinline__ void load_params(const float* __restrict__ params, MlpSmem& S)
{
    for (int i = threadIdx.x; i < kP; i += blockDim.x) {
        const float v = params[i];
        if (i < ob1) S.w1[i / kIn][i % kIn] = v;
        else if (i < oW2) S.b1[i - ob1] = v;
        else if (i < ob2) S.w2[(i - oW2) / kH][(i - oW2) % kH] = v;
        else if (i < ow3) S.b2[i - ob2] = v;
        else if (i < ob3) S.w3[i - ow3] = v;
        else S.b3 = v;
    }
}

// Forward pass of samples s0 .. s0+m-1 (m <= kMlpBatch): y = b3 + w3 . relu(W2 relu(W1 x +
// b1) + b2).  Ends with a barrier.
__device__ __forceinline__ void forward_batch(MlpSmem& S, const float* __restrict__ x, int64_t s0, int m)
{
    const int tid = threadIdx.x, u = tid & (kH - 1), a = 2 * (tid / kH), b = a + 1;
    if (tid < kMlpBatch * kIn) S.x[tid / kIn][tid % kIn] = tid / kIn < m ? x[s0 * kIn + tid] : 0.0f;
    __syncthreads();
    {
        float p = S.b1[u], q = p;
#pragma unroll
        for (int i = 0; i < kIn; i++) {
            const float w = S.w1[u][i];
            p = fmaf(w, S.x[a][i], p);
            q = fmaf(w, S.x[b][i], q);
        }
        S.h1[a][u] = fmaxf(p, 0.0f);
        S.h1[b][u] = fmaxf(q, 0.0f);
    }
    __syncthreads();
    {
        float p = S.b2[u], q = p;
#pragma unroll
        for (int k = 0; k < kH; k += 4) {
            const float4 ha = *reinterpret_cast<const float4*>(&S.h1[a][k]);
            const float4 hb = *reinterpret_cast<const float4*>(&S.h1[b][k]);
            const float va[4] = {ha.x, ha.y, ha.z, ha.w}, vb[4] = {hb.x, hb.y, hb.z, hb.w};
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const float w = S.w2[u][k + i];
                p = fmaf(w, va[i], p);
                q = fmaf(w, vb[i], q);
            }
        }
        S.h2[a][u] = fmaxf(p, 0.0f);
        S.h2[b][u] = fmaxf(q, 0.0f);
    }
    __syncthreads();
    if ((tid & 31) == 0) {  // one sample per warp
        const int s = tid >> 5;
        float out = S.b3;
#pragma unroll 16
        for (int j = 0; j < kH; j++) out = fmaf(S.w3[j], S.h2[s][j], out);
        S.y[s] = out;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kMlpThreads) k_mlp_forward(const float* __restrict__ params,
                                                             const float* __restrict__ x, int64_t n,
                                                             float* __restrict__ y)
{
    __shared__ MlpSmem S;
    load_params(params, S);
    for (int64_t s0 = (int64_t)blockIdx.x * kMlpBatch; s0 < n; s0 += (int64_t)gridDim.x * kMlpBatch) {
        const int m = (int)min((int64_t)kMlpBatch, n - s0);
        forward_batch(S, x, s0, m);
        if (threadIdx.x < m) y[s0 + threadIdx.x] = S.y[threadIdx.x];
    }
}

// A sum held as three FP32 numbers: a product's rounding error by an fma and the rounding
// errors of the high and middle sums by TwoSum (Knuth 1969), all exact, so that only the low
// sum rounds, 2^-72 below the value.  Its FP64 value is rounded once (2^-53), where an FP64
// sum of the same products rounds each time.  What lies below FP32's smallest number, 2^-149,
// is lost; the gradient is FP32.
struct TripleSum {
    float h, m, l;
    static __device__ __forceinline__ float two_sum(float a, float b, float& err)
    {
        const float s = a + b, t = s - a;
        err = (a - (s - t)) + (b - t);
        return s;
    }
    __device__ __forceinline__ void add(float p)
    {
        float r, r1;
        h = two_sum(h, p, r);
        m = two_sum(m, r, r1);
        l += r1;
    }
    __device__ __forceinline__ void add_product(float a, float b)
    {
        const float p = a * b, e = fmaf(a, b, -p);
        float r, r1, r2;
        h = two_sum(h, p, r);
        m = two_sum(m, r, r1);
        m = two_sum(m, e, r2);
        l += r1 + r2;
    }
    // an overflowed sum has no lower parts
    __device__ __forceinline__ double value() const
    {
        return fabsf(h) < INFINITY ? (double)h + ((double)m + (double)l) : (double)h;
    }
};

// Gradient of L = (1/n) sum (y - t)^2 and the sum of squares over samples blockIdx.x * per
// .. + per - 1: into part [blockIdx.x][kP + 1] (kDirect: one CTA, the gradient and L).
// dL/d(pre-activation) of layer 2 is d2, of layer 1 d1; the ReLU passes the gradient where
// its output > 0.
// The 4801 sums over samples are what bounds an epoch.  FP64 instructions are scarce (two
// per clock and SM), so a thread keeps its ten sums as FP32 triples over the CTA's samples
// and only their values are added in FP64.  Measured with 5696 samples: 60 us an epoch; one
// thread per parameter with FP64 sums over all samples took 833, and pairs (48 bits, less
// than FP64's 53) 48.  The gradient is the same to its last bit's rounding (largest error
// against FP64 autograd, relative to the largest entry, 500 to 20000 samples: 3.5e-8 to 4.5e-8
// in all three).
template <bool kDirect>
__global__ void __launch_bounds__(kMlpThreads) k_mlp_slab(const float* __restrict__ params,
                                                          const float* __restrict__ x,
                                                          const float* __restrict__ t, int64_t n, int64_t per,
                                                          double* __restrict__ part, float* __restrict__ grad,
                                                          double* __restrict__ loss)
{
    __shared__ MlpSmem S;
    __shared__ double sq[kMlpBatch];
    load_params(params, S);
    const int tid = threadIdx.x;
    const int u = tid & (kH - 1), a = 2 * (tid / kH), b = a + 1;
    // this thread's parameters: W2 rows 2 j2, 2 j2 + 1, columns 4 k4 .. + 3; W1 entry tid; and of
    // threads 0 .. 192 one of b1, b2, w3, b3
    const int j2 = 2 * (tid >> 4), k4 = 4 * (tid & 15);
    TripleSum g2[2][4] = {}, g1 = {}, g0 = {};
    double err = 0.0;  // of the sample whose output this thread has (first lane of a warp)
    const int64_t begin = (int64_t)blockIdx.x * per, end = min(n, begin + per);
    for (int64_t s0 = begin; s0 < end; s0 += kMlpBatch) {
        const int m = (int)min((int64_t)kMlpBatch, end - s0);
        forward_batch(S, x, s0, m);
        if ((tid & 31) == 0) {
            const int s = tid >> 5;
            float g = 0.0f;
            if (s < m) {
                const float ts = t[s0 + s];
                g = 2.0f * (S.y[s] - ts) / (float)n;
                const double d = (double)S.y[s] - ts;
                err += d * d;
            }
            S.dy[s] = g;
        }
        __syncthreads();
        S.d2[a][u] = S.h2[a][u] > 0.0f ? S.dy[a] * S.w3[u] : 0.0f;
        S.d2[b][u] = S.h2[b][u] > 0.0f ? S.dy[b] * S.w3[u] : 0.0f;
        __syncthreads();
        {
            float p = 0.0f, q = 0.0f;
#pragma unroll
            for (int j = 0; j < kH; j += 4) {
                const float4 da = *reinterpret_cast<const float4*>(&S.d2[a][j]);
                const float4 db = *reinterpret_cast<const float4*>(&S.d2[b][j]);
                const float va[4] = {da.x, da.y, da.z, da.w}, vb[4] = {db.x, db.y, db.z, db.w};
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const float w = S.w2[j + i][u];
                    p = fmaf(w, va[i], p);
                    q = fmaf(w, vb[i], q);
                }
            }
            S.d1[a][u] = S.h1[a][u] > 0.0f ? p : 0.0f;
            S.d1[b][u] = S.h1[b][u] > 0.0f ? q : 0.0f;
        }
        __syncthreads();
        for (int s = 0; s < m; s++) {
            const float2 d = *reinterpret_cast<const float2*>(&S.d2[s][j2]);
            const float4 h = *reinterpret_cast<const float4*>(&S.h1[s][k4]);
            const float dv[2] = {d.x, d.y}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int k = 0; k < 4; k++) g2[i][k].add_product(dv[i], hv[k]);
            g1.add_product(S.d1[s][tid / kIn], S.x[s][tid % kIn]);
            if (tid < kH) g0.add(S.d1[s][u]);
            else if (tid < 2 * kH) g0.add(S.d2[s][u]);
            else if (tid < 3 * kH) g0.add_product(S.dy[s], S.h2[s][u]);
            else if (tid == 3 * kH) g0.add(S.dy[s]);
        }
        __syncthreads();  // the batch's activations are no longer read
    }
    auto put = [&](int p, const TripleSum& g) {
        if (kDirect) grad[p] = (float)g.value();
        else part[(int64_t)blockIdx.x * (kP + 1) + p] = g.value();
    };
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int k = 0; k < 4; k++) put(oW2 + (j2 + i) * kH + k4 + k, g2[i][k]);
    put(oW1 + tid, g1);
    if (tid < kH) put(ob1 + u, g0);
    else if (tid < 2 * kH) put(ob2 + u, g0);
    else if (tid < 3 * kH) put(ow3 + u, g0);
    else if (tid == 3 * kH) put(ob3, g0);
    if ((tid & 31) == 0) sq[tid >> 5] = err;
    __syncthreads();
    if (tid == 0) {
        double e = 0.0;
        for (int s = 0; s < kMlpBatch; s++) e += sq[s];
        if (!kDirect) part[(int64_t)blockIdx.x * (kP + 1) + kP] = e;
        else if (loss) *loss = e / (double)n;
    }
}
static_assert(kMlpThreads == kH * kIn && kMlpThreads * 8 == kH * kH && kMlpThreads == kMlpBatch * 32 &&
                  kMlpThreads * 2 == kMlpBatch * kH,
              "threads of a batch");

// Adam (Kingma & Ba 2015) with bias correction: c1 = 1/(1 - beta1^t), c2 = 1/(1 - beta2^t).
struct AdamArgs {
    float *params, *m, *v;
    float lr, c1, c2;
};
__device__ __forceinline__ void adam_update(const AdamArgs& A, int p, float g)
{
    const float mm = VL_MLP_BETA1 * A.m[p] + (1.0f - VL_MLP_BETA1) * g;
    const float vv = VL_MLP_BETA2 * A.v[p] + (1.0f - VL_MLP_BETA2) * g * g;
    A.m[p] = mm;
    A.v[p] = vv;
    A.params[p] -= A.lr * (mm * A.c1) / (sqrtf(vv * A.c2) + VL_MLP_EPS);
}

__global__ void k_mlp_adam(AdamArgs A, const float* __restrict__ grad)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < kP) adam_update(A, p, grad[p]);
}

// Sum of the parts in a fixed order: 32 parameters and 8 interleaved chains of parts per
// CTA.  kAdam: the update; else the gradient.  Entry kP is the sum of squares.
template <bool kAdam>
__global__ void __launch_bounds__(256) k_mlp_join(const double* __restrict__ part, int nparts, int64_t n,
                                                  AdamArgs A, float* __restrict__ grad, double* __restrict__ loss)
{
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    double a = 0.0;
    if (p <= kP)
        for (int s = c; s < nparts; s += 8) a += part[(int64_t)s * (kP + 1) + p];
    sh[c][lane] = a;
    __syncthreads();
    if (c != 0 || p > kP) return;
    for (int i = 1; i < 8; i++) a += sh[i][lane];
    if (p == kP) {
        if (loss) *loss = a / (double)n;
    } else if (kAdam) {
        adam_update(A, p, (float)a);
    } else {
        grad[p] = (float)a;
    }
}

// capacity = ceil((1 + margin) * sum_i max(exp(y_i) - 1, 0)), FP64, one CTA, fixed order.
__global__ void k_capacity_sum(const float* __restrict__ y, int64_t n, double margin, int64_t* out)
{
    __shared__ double sh[kThreads];
    double a = 0.0;
    for (int64_t s = threadIdx.x; s < n; s += blockDim.x) a += fmax(expm1((double)y[s]), 0.0);
    sh[threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int i = 0; i < (int)blockDim.x; i++) tot += sh[i];
        *out = (int64_t)ceil((1.0 + margin) * tot);
    }
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Workspace of a training step, of vl_mlp_workspace_bytes: the loss, the gradient, then
// the CTAs' parts.  About one kB per sample, so that a part covers about 38 samples, up to
// kMaxParts parts: one per SM of a GB300, a constant, so that the order of the sums and with it
// their last bits depend on the number of samples alone, and not on the GPU.
constexpr int kMaxParts = 152;
constexpr size_t kWsGrad = 256, kWsParts = kWsGrad + ((size_t)kP * 4 + 255) / 256 * 256;

size_t train_ws_bytes(int64_t n)
{
    return 2 * align256((size_t)n * 4) + 4 * align256((size_t)n * kH * 4) + kWsParts;
}

// Queues gradient (and, with A, the Adam update) of one full batch.
vl_status queue_gradient(const float* params, const float* x, const float* t, int64_t n, void* workspace,
                         float* grad_out, const AdamArgs* A, double* loss_out, cudaStream_t s)
{
    char* ws = static_cast<char*>(workspace);
    // the kernels write the loss in place unless the caller's pointer is not aligned for it
    const bool copy_loss = loss_out && ((uintptr_t)loss_out & 7);
    double* loss = copy_loss ? reinterpret_cast<double*>(ws) : loss_out;
    float* grad = grad_out ? grad_out : reinterpret_cast<float*>(ws + kWsGrad);
    double* part = reinterpret_cast<double*>(ws + kWsParts);
    const int64_t room = (int64_t)((train_ws_bytes(n) - kWsParts) / ((kP + 1) * sizeof(double)));
    const int64_t most = std::max<int64_t>(1, std::min<int64_t>(kMaxParts, room));
    const int64_t per = (n + most - 1) / most;
    const int parts = (int)((n + per - 1) / per);
    const AdamArgs none{};
    if (parts == 1) {
        k_mlp_slab<true><<<1, kMlpThreads, 0, s>>>(params, x, t, n, per, nullptr, grad, loss);
        if (A) k_mlp_adam<<<nblk(kP, 128), 128, 0, s>>>(*A, grad);
    } else {
        k_mlp_slab<false><<<parts, kMlpThreads, 0, s>>>(params, x, t, n, per, part, nullptr, nullptr);
        if (A) k_mlp_join<true><<<nblk(kP + 1, 32), 256, 0, s>>>(part, parts, n, *A, nullptr, loss);
        else k_mlp_join<false><<<nblk(kP + 1, 32), 256, 0, s>>>(part, parts, n, none, grad, loss);
    }
    note_launch();
    if (A || parts > 1) note_launch();
    if (copy_loss) cudaMemcpyAsync(loss_out, loss, 8, cudaMemcpyDeviceToDevice, s);
    return cudaGetLastError() == cudaSuccess ? VL_OK : VL_ECUDA;
}

// CTAs of a forward pass: one per batch, up to four per SM.
unsigned forward_ctas(int64_t n)
{
    return (unsigned)std::min<int64_t>((n + kMlpBatch - 1) / kMlpBatch, 152 * 4);
}

vl_status launch_status()
{
    return cudaGetLastError() == cudaSuccess ? VL_OK : VL_ECUDA;
}

}  // namespace

vl_status tile_features(Grid* g, int edge, float* feat, float* uni)
{
    const GridGeom& G = g->geom;
    if (edge < 1 || edge > 64 || !feat || !uni) return fail(g, VL_EINVAL, "vl_tile_features: bad arguments");
    if (!g->has_state) return fail(g, VL_ESTATE, "vl_tile_features: no state");
    int64_t ntiles = 1;
    TileGeom T;
    T.G = G;
    T.edge = edge;
    for (int d = 0; d < 3; d++) {
        T.nt[d] = (G.n[d] + edge - 1) / edge;
        ntiles *= T.nt[d];
    }
    // per-cell moments, then the tiles' block counts
    double* mom = (double*)g->alloc((size_t)G.N * 7 * 8 + (size_t)ntiles * 16);
    if (!mom) return fail(g, VL_ENOMEM, "vl_tile_features: scratch allocation failed");
    unsigned long long* counts = reinterpret_cast<unsigned long long*>(mom + G.N * 7);
    cudaMemsetAsync(counts, 0, (size_t)ntiles * 16, g->stream);
    void* parts = nullptr;
    vl_status st = queue_cell_moments(g, mom, &parts);
    if (st != VL_OK) {
        cudaStreamSynchronize(g->stream);
        g->release(parts);
        g->release(mom);
        return st;
    }
    // the next layout's ubits become the 27-cell union of the state (the next step
    // rebuilds that layout anyway)
    launch_union(g, g->lay[g->cur], g->lay[1 - g->cur], nullptr);
    // about eight CTAs per SM, parts of at least 16 ids
    const int split = (int)std::max<int64_t>(1, std::min<int64_t>((G.nb + 15) / 16, 152 * 8 / ntiles));
    const int ids = (G.nb + split - 1) / split;
    k_tile_counts<<<dim3((unsigned)ntiles, (unsigned)((G.nb + ids - 1) / ids)), 256, 0, g->stream>>>(
        T, ids, g->lay[g->cur].kbits, g->lay[1 - g->cur].ubits, counts);
    note_launch();
    k_tile_features<<<(unsigned)ntiles, 256, 0, g->stream>>>(T, counts, mom, feat, uni);
    note_launch();
    cudaError_t e = cudaStreamSynchronize(g->stream);
    g->release(parts);
    g->release(mom);
    return e == cudaSuccess ? VL_OK : cuda_fail(g, e, "vl_tile_features");
}

}  // namespace vlgt

using namespace vlgt;

extern "C" int64_t vl_tile_count(const vl_space_desc* space, int edge)
{
    if (!space || edge < 1) return -1;
    int64_t t = 1;
    for (int d = 0; d < 3; d++) t *= (space->n[d] + edge - 1) / edge;
    return t;
}

extern "C" vl_status vl_cost_targets(const float* union_trace, int nsnap, int64_t ntiles, int horizon,
                                     float* targets, void* stream)
{
    if (!union_trace || !targets || ntiles < 0 || horizon < 1 || nsnap < horizon) return VL_EINVAL;
    const int64_t n = (int64_t)(nsnap - horizon + 1) * ntiles;
    if (n == 0) return VL_OK;
    k_cost_targets<<<nblk(n, 256), 256, 0, (cudaStream_t)stream>>>(union_trace, nsnap, ntiles, horizon, targets);
    note_launch();
    return launch_status();
}

extern "C" vl_status vl_mlp_forward(const float* params, const float* x, int64_t n, float* y, void* stream)
{
    if (!params || n < 0 || (n > 0 && (!x || !y))) return VL_EINVAL;
    if (n == 0) return VL_OK;
    k_mlp_forward<<<forward_ctas(n), kMlpThreads, 0, (cudaStream_t)stream>>>(params, x, n, y);
    note_launch();
    return launch_status();
}

extern "C" size_t vl_mlp_workspace_bytes(int64_t n)
{
    return n < 0 ? 0 : train_ws_bytes(n);
}

extern "C" vl_status vl_mlp_train_step(float* params, float* adam_m, float* adam_v, const float* x,
                                       const float* t, int64_t n, int step, float lr, void* workspace,
                                       size_t workspace_bytes, double* loss, void* stream)
{
    if (!params || !adam_m || !adam_v || !x || !t || n <= 0 || step < 1 || !(lr >= 0.0f) || !workspace)
        return VL_EINVAL;
    if (workspace_bytes < train_ws_bytes(n) || ((uintptr_t)workspace & 255)) return VL_EINVAL;
    const double c1 = 1.0 / (1.0 - std::pow((double)VL_MLP_BETA1, step));
    const double c2 = 1.0 / (1.0 - std::pow((double)VL_MLP_BETA2, step));
    const AdamArgs A{params, adam_m, adam_v, lr, (float)c1, (float)c2};
    return queue_gradient(params, x, t, n, workspace, nullptr, &A, loss, (cudaStream_t)stream);
}

extern "C" vl_status vl_mlp_gradient(const float* params, const float* x, const float* t, int64_t n,
                                     void* workspace, size_t workspace_bytes, float* grad, double* loss,
                                     void* stream)
{
    if (!params || !x || !t || n <= 0 || !workspace || !grad) return VL_EINVAL;
    if (workspace_bytes < train_ws_bytes(n) || ((uintptr_t)workspace & 255)) return VL_EINVAL;
    return queue_gradient(params, x, t, n, workspace, grad, nullptr, loss, (cudaStream_t)stream);
}

extern "C" vl_status vl_mlp_capacity(const float* params, const float* features, int64_t ntiles,
                                     double margin, void* workspace, size_t workspace_bytes,
                                     int64_t* capacity, void* stream)
{
    if (!params || !features || ntiles <= 0 || !workspace || !capacity || !(margin >= 0.0)) return VL_EINVAL;
    if (workspace_bytes < align256((size_t)ntiles * 4) + 8 || ((uintptr_t)workspace & 255)) return VL_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    float* y = static_cast<float*>(workspace);
    int64_t* out = reinterpret_cast<int64_t*>(static_cast<char*>(workspace) + align256((size_t)ntiles * 4));
    k_mlp_forward<<<forward_ctas(ntiles), kMlpThreads, 0, s>>>(params, features, ntiles, y);
    k_capacity_sum<<<1, kThreads, 0, s>>>(y, ntiles, margin, out);
    note_launch();
    note_launch();
    cudaError_t e = cudaMemcpyAsync(capacity, out, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? VL_OK : VL_ECUDA;
}
