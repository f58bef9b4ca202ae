// moments.cu -- FP64 velocity moments per cell (n, n V_d, P_dd) and the total mass.
//
// FP64 instructions are scarce on this chip (two per clock and SM, conversions included),
// so the sums are taken in pairs of FP32 numbers without loss: TwoSum (Knuth 1969) gives
// the rounding error of an FP32 addition exactly, and a short tree of them carries a sum as
// high + low part with 48 bits.  A block's 64 values are reduced that way to its twelve
// partial sums over vx, vy and vz (its share of the cell's three marginals
// M_d[i] = sum of f over the velocity cells with index i along d); only those are added up
// in FP64.  n, V and P follow from the marginals in FP64 with P summed about V, as a sum
// over single values would give them: one pass over f instead of two, 0.4 FP64
// instructions per value instead of 28.
//
// A warp takes eight cells (blocks.cuh).
//
// Measured (64x32x16 cells x 32^3 velocity cells, 4.3 GB of f, 0.63 ms at the copy rate):
// 1.16 ms per call, total mass 0.69; the kernel for any mesh, which sums every value
// in FP64 with one warp per cell, 49.8 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "blocks.cuh"
#include "grid.h"

namespace vlgt {

namespace {

constexpr int kMaxRun = 8;       // blocks summed in FP32 pairs before the sum goes to FP64
constexpr int kWarps = 8;        // warps of a CTA, at most

struct VMesh {
    double vmin[3], dv[3];
    int nv[3];
};

// A sum held as high + low part.
struct Pair {
    float h, l;
};
__device__ __forceinline__ Pair two_sum(float a, float b)
{
    const float s = a + b, t = s - a;
    return {s, (a - (s - t)) + (b - t)};
}
__device__ __forceinline__ Pair add(const Pair& a, const Pair& b)
{
    const Pair s = two_sum(a.h, b.h);
    return {s.h, s.l + (a.l + b.l)};
}
__device__ __forceinline__ Pair sum4(float a, float b, float c, float d)
{
    const Pair p = two_sum(a, b), q = two_sum(c, d), s = two_sum(p.h, q.h);
    return {s.h, s.l + (p.l + q.l)};
}
__device__ __forceinline__ Pair shfl_xor(const Pair& a, int m)
{
    return {__shfl_xor_sync(0xffffffffu, a.h, m), __shfl_xor_sync(0xffffffffu, a.l, m)};
}
__device__ __forceinline__ double value(const Pair& a) { return (double)a.h + (double)a.l; }

// Entry k = lane & 3 of the sum over four neighbouring lanes of p[0..3].
__device__ __forceinline__ Pair transpose_sum(const Pair (&p)[4], int k)
{
    const bool hi = k & 2, odd = k & 1;
    const Pair a0 = add(hi ? p[2] : p[0], shfl_xor(hi ? p[0] : p[2], 2));
    const Pair a1 = add(hi ? p[3] : p[1], shfl_xor(hi ? p[1] : p[3], 2));
    return add(odd ? a1 : a0, shfl_xor(odd ? a0 : a1, 1));
}

// Groups of eight cells along x, row by row.
struct Groups {
    int per_row;     // groups of a row
    int64_t total;   // groups
    int split, ids;  // parts of the block ids, ids of a part
};

// n V_d and P_dd of the group's cells from their marginals acc[(first index of d + i) *
// kGroup + cell].
__device__ __forceinline__ void write_moments(const GridGeom& G, const VMesh& V, const Groups& P, int64_t grp,
                                              const double* acc, double* out)
{
    const int lane = threadIdx.x & 31, j = lane >> 2, d = lane & 3;
    const int64_t row = grp / P.per_row;
    const int x = (int)(grp - row * P.per_row) * kGroup + j;
    const double dv3 = V.dv[0] * V.dv[1] * V.dv[2];
    const int nd = d == 0 ? V.nv[0] : d == 1 ? V.nv[1] : d == 2 ? V.nv[2] : 0;
    const double* M = acc + (d == 0 ? 0 : d == 1 ? V.nv[0] : V.nv[0] + V.nv[1]) * kGroup + j;
    const double vmin = d == 0 ? V.vmin[0] : d == 1 ? V.vmin[1] : V.vmin[2];
    const double dv = d == 0 ? V.dv[0] : d == 1 ? V.dv[1] : V.dv[2];
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int i = 0; i < nd; i++) {
        const double f = M[i * kGroup];
        s0 += f;
        s1 += (vmin + (i + 0.5) * dv) * f;
    }
    const double n = __shfl_sync(0xffffffffu, s0, lane & ~3);
    const double mean = n != 0.0 ? s1 / n : 0.0;
    for (int i = 0; i < nd; i++) {
        const double w = (vmin + (i + 0.5) * dv) - mean;
        s2 += w * w * M[i * kGroup];
    }
    if (x < G.n[0] && d < 3) {
        double* o = out + (row * G.n[0] + x) * 7;
        if (d == 0) o[0] = n * dv3;
        o[1 + d] = s1 * dv3;
        o[4 + d] = s2 * dv3;
    }
}

// kSplit: the marginals of this part of the block ids go to part [blockIdx.y][group] of
// scratch, else the moments to out.
template <int kCodec, bool kSplit>
__global__ void __launch_bounds__(kWarps * 32, 3) k_marginals(GridGeom G, LayoutView L, VMesh V, Groups P,
                                                              double* __restrict__ out)
{
    extern __shared__ double s_acc[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, j = lane >> 2, k = lane & 3;
    const int64_t grp = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (grp >= P.total) return;
    const int nvt = V.nv[0] + V.nv[1] + V.nv[2];
    double* acc = s_acc + (size_t)warp * nvt * kGroup;
    for (int i = lane; i < nvt * kGroup; i += 32) acc[i] = 0.0;
    __syncwarp();
    // this lane's entries: cell j, index 4 * block + k of each marginal
    double* ax = acc + k * kGroup + j;
    double* ay = ax + V.nv[0] * kGroup;
    double* az = ay + V.nv[1] * kGroup;
    // this lane's vx rows (vy = k, vz = q), each summed over vx and over consecutive blocks of
    // one row of blocks along vx: the vy and vz marginals of those blocks come from them
    Pair Z[4] = {};
    int run = 0, row_of_run = -1;
    auto flush = [&]() {
        if (run == 0) return;
        ay[(row_of_run % G.nby) * 4 * kGroup] += value(add(add(Z[0], Z[1]), add(Z[2], Z[3])));
        az[(row_of_run / G.nby) * 4 * kGroup] += value(transpose_sum(Z, k));
#pragma unroll
        for (int q = 0; q < 4; q++) Z[q] = {0.f, 0.f};
        run = 0;
    };
    const int b_begin = blockIdx.y * P.ids, b_end = min(G.nb, b_begin + P.ids);
    const int64_t row = grp / P.per_row;
    const int x0 = (int)(grp - row * P.per_row) * kGroup;
    auto load = [&](int, bool has, int64_t chunk, uint32_t cnt) {
        Rows<kCodec> r;
        r.load(L, chunk, cnt, k, has);
        return r;
    };
    for_blocks<Rows<kCodec>>(G, L, row, x0, 0xffu, b_begin, b_end, load, [&](int b, const Rows<kCodec>& r, bool, int64_t, uint32_t) {
        const int brow = b / G.nbx, bx = b - brow * G.nbx;
        if (brow != row_of_run || run == kMaxRun) {
            flush();
            row_of_run = brow;
        }
        float f[4][4];
        Pair X[4], S[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 v = r.get(q);
            f[q][0] = v.x;
            f[q][1] = v.y;
            f[q][2] = v.z;
            f[q][3] = v.w;
            S[q] = add(Z[q], sum4(v.x, v.y, v.z, v.w));
        }
#pragma unroll
        for (int i = 0; i < 4; i++) X[i] = sum4(f[0][i], f[1][i], f[2][i], f[3][i]);
        const Pair x = transpose_sum(X, k);
        // sums that leave FP32's range on the way (2^125: four of them still fit), infinities
        // and NaN: FP64 for this block
        const bool wide =
            !((fabsf(S[0].h) + fabsf(S[1].h)) + (fabsf(S[2].h) + fabsf(S[3].h)) + fabsf(x.h) < 0x1p125f);
        if (__any_sync(0xffffffffu, wide)) {
            double dx[4], dz[4], dy = 0.0;
            for (int i = 0; i < 4; i++) {
                dx[i] = ((double)f[0][i] + f[1][i]) + ((double)f[2][i] + f[3][i]);
                dz[i] = ((double)f[i][0] + f[i][1]) + ((double)f[i][2] + f[i][3]);
                dy += dz[i];
            }
            for (int i = 0; i < 4; i++)
                for (int o = 1; o < 4; o <<= 1) {
                    dx[i] += __shfl_xor_sync(0xffffffffu, dx[i], o);
                    dz[i] += __shfl_xor_sync(0xffffffffu, dz[i], o);
                }
            const double xk = k == 0 ? dx[0] : k == 1 ? dx[1] : k == 2 ? dx[2] : dx[3];
            const double zk = k == 0 ? dz[0] : k == 1 ? dz[1] : k == 2 ? dz[2] : dz[3];
            ax[bx * 4 * kGroup] += xk;
            ay[(brow % G.nby) * 4 * kGroup] += dy;
            az[(brow / G.nby) * 4 * kGroup] += zk;
            return;
        }
        ax[bx * 4 * kGroup] += value(x);
#pragma unroll
        for (int q = 0; q < 4; q++) Z[q] = S[q];
        run++;
    });
    flush();
    __syncwarp();
    if (kSplit) {
        double* o = out + ((int64_t)blockIdx.y * P.total + grp) * nvt * kGroup;
        for (int i = lane; i < nvt * kGroup; i += 32) o[i] = acc[i];
    } else {
        write_moments(G, V, P, grp, acc, out);
    }
}

// Moments from the parts' marginals, added in order.
__global__ void k_join_marginals(GridGeom G, VMesh V, Groups P, const double* __restrict__ parts,
                                 double* __restrict__ out)
{
    extern __shared__ double s_acc[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t grp = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (grp >= P.total) return;
    const int n = (V.nv[0] + V.nv[1] + V.nv[2]) * kGroup;
    double* acc = s_acc + (size_t)warp * n;
    for (int i = lane; i < n; i += 32) {
        double s = 0.0;
        for (int p = 0; p < P.split; p++) s += parts[((int64_t)p * P.total + grp) * n + i];
        acc[i] = s;
    }
    __syncwarp();
    write_moments(G, V, P, grp, acc, out);
}

// Density of every cell over this part of the block ids: dens[blockIdx.y][cell].
template <int kCodec>
__global__ void __launch_bounds__(kWarps * 32, 4) k_density(GridGeom G, LayoutView L, VMesh V, Groups P,
                                                            double* __restrict__ dens)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, j = lane >> 2, k = lane & 3;
    const int64_t grp = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (grp >= P.total) return;
    double sum = 0.0;
    Pair p{0.f, 0.f};
    int run = 0;
    const int b_begin = blockIdx.y * P.ids, b_end = min(G.nb, b_begin + P.ids);
    const int64_t row = grp / P.per_row;
    const int x0 = (int)(grp - row * P.per_row) * kGroup;
    auto load = [&](int, bool has, int64_t chunk, uint32_t cnt) {
        Rows<kCodec> r;
        r.load(L, chunk, cnt, k, has);
        return r;
    };
    for_blocks<Rows<kCodec>>(G, L, row, x0, 0xffu, b_begin, b_end, load, [&](int, const Rows<kCodec>& r, bool, int64_t, uint32_t) {
        Pair s{0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 v = r.get(q);
            const Pair t = sum4(v.x, v.y, v.z, v.w);
            s = q == 0 ? t : add(s, t);
        }
        const Pair t = add(p, s);
        if (fabsf(t.h) < INFINITY) {
            p = t;
        } else {  // infinities, NaN, sums beyond FP32's range
            for (int q = 0; q < 4; q++) {
                const float4 v = r.get(q);
                sum += ((double)v.x + v.y) + ((double)v.z + v.w);
            }
        }
        if (++run == kMaxRun) {
            sum += value(p);
            p = {0.f, 0.f};
            run = 0;
        }
    });
    sum += value(p);
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    const int x = x0 + j;
    if (k == 0 && x < G.n[0]) dens[(int64_t)blockIdx.y * G.N + row * G.n[0] + x] = sum * (V.dv[0] * V.dv[1] * V.dv[2]);
}

// total += sum of v[0 .. n-1]
__global__ void k_sum(const double* __restrict__ v, int64_t n, double* __restrict__ total)
{
    double s = 0.0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x)
        s += v[c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s != 0.0) atomicAdd(total, s);
}

VMesh vmesh_of(const Grid* g)
{
    VMesh V;
    for (int d = 0; d < 3; d++) {
        V.vmin[d] = g->vmesh.vmin[d];
        V.dv[d] = g->vmesh.dv[d];
        V.nv[d] = g->vmesh.nv[d];
    }
    return V;
}

Groups groups_of(const Grid* g, int nsm)
{
    const GridGeom& G = g->geom;
    Groups P;
    P.per_row = (G.n[0] + kGroup - 1) / kGroup;
    P.total = (int64_t)P.per_row * G.R;
    const Parts s = parts_of(G.nb, P.total, (int64_t)nsm * 16, 64);  // a part has marginals to join
    P.split = s.split;
    P.ids = s.ids;
    return P;
}

// Shared memory of the marginals per warp, and the widest velocity mesh they fit for.
size_t warp_bytes(const Grid* g)
{
    return (size_t)(g->vmesh.nv[0] + g->vmesh.nv[1] + g->vmesh.nv[2]) * kGroup * sizeof(double);
}
constexpr size_t kSmemCta = 100 * 1024;  // two CTAs per SM

int sm_count(const Grid* g)
{
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, g->dev.device);
    return std::max(n, 1);
}

}  // namespace

bool moments_fit(const Grid* g) { return warp_bytes(g) <= kSmemCta; }

// Small grids take scratch from the caller's allocator, returned in *scratch.
vl_status queue_moments(Grid* g, double* d_out, void** scratch)
{
    const GridGeom& G = g->geom;
    const LayoutView L = g->lay[g->cur].view();
    const VMesh V = vmesh_of(g);
    const Groups P = groups_of(g, sm_count(g));
    const size_t wb = warp_bytes(g);
    const int warps = (int)std::max<size_t>(1, std::min<size_t>(kWarps, kSmemCta / wb));
    const unsigned ctas = (unsigned)((P.total + warps - 1) / warps);
    const int smem = (int)(warps * wb);
    double* parts = nullptr;
    *scratch = nullptr;
    if (P.split > 1) {
        parts = (double*)g->alloc((size_t)P.split * P.total * wb);
        if (!parts) return fail(g, VL_ENOMEM, "moments: scratch allocation failed");
        *scratch = parts;
    }
    with_codec(g->codec, [&](auto c) {
        constexpr int kc = decltype(c)::value;
        auto kern = P.split > 1 ? k_marginals<kc, true> : k_marginals<kc, false>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        kern<<<dim3(ctas, P.split), warps * 32, smem, g->stream>>>(G, L, V, P, parts ? parts : d_out);
    });
    note_launch();
    if (P.split > 1) {
        cudaFuncSetAttribute(k_join_marginals, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        k_join_marginals<<<ctas, warps * 32, smem, g->stream>>>(G, V, P, parts, d_out);
        note_launch();
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? VL_OK : cuda_fail(g, e, "moments launch");
}

vl_status total_mass(Grid* g, double* mass)
{
    const GridGeom& G = g->geom;
    const VMesh V = vmesh_of(g);
    const Groups P = groups_of(g, sm_count(g));
    // densities of the parts, then the total
    double* dens = (double*)g->alloc(((size_t)P.split * G.N + 1) * sizeof(double));
    if (!dens) return fail(g, VL_ENOMEM, "vl_mass: scratch allocation failed");
    double* acc = dens + (size_t)P.split * G.N;
    cudaMemsetAsync(acc, 0, sizeof(double), g->stream);
    with_codec(g->codec, [&](auto c) {
        k_density<decltype(c)::value>
            <<<dim3((unsigned)((P.total + kWarps - 1) / kWarps), P.split), kWarps * 32, 0, g->stream>>>(
                G, g->lay[g->cur].view(), V, P, dens);
    });
    note_launch();
    const int64_t n = (int64_t)P.split * G.N;
    k_sum<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 4), 256, 0, g->stream>>>(dens, n, acc);
    note_launch();
    double h = 0.0;
    cudaMemcpyAsync(&h, acc, sizeof(double), cudaMemcpyDeviceToHost, g->stream);
    const cudaError_t e = cudaStreamSynchronize(g->stream);
    g->release(dens);
    if (e != cudaSuccess) return cuda_fail(g, e, "vl_mass");
    *mass = h * g->space.dx[0] * g->space.dx[1] * g->space.dx[2];
    return VL_OK;
}

}  // namespace vlgt
