// moments.cu -- FP64 velocity moments per cell (n, n V_d, P_dd) and the total mass.
//
// FP64 instructions are scarce on this chip (two per clock and SM, conversions included),
// so a block's values are added as integer multiples of two powers of two and a small FP32
// rest, exactly but for that rest (Places, below).  A block's 64 values are reduced that way
// to its twelve partial sums over vx, vy and vz (its share of the cell's three marginals
// M_d[i] = sum of f over the velocity cells with index i along d); only those are added up
// in FP64.  n, V and P follow from the marginals in FP64 with P summed about V, as a sum
// over single values would give them: one pass over f instead of two, 0.4 FP64
// instructions per value instead of 28.
//
// A warp takes eight cells (blocks.cuh).
//
// Measured (64x32x16 cells x 32^3 velocity cells, 4.3 GB of f, 0.63 ms at the copy rate):
// 1.55 ms per call, bound by instruction issue (splits and sums); total mass 0.67; the kernel
// for any mesh, which sums every value in FP64 with one warp per cell, 49.8 ms.  Sums in pairs
// of FP32 numbers (48 bits) took 1.26 and 0.64 ms, but were less precise than FP64 sums of
// single values: largest relative error of n against 128-bit sums 5.6e-15 on a 4^3 mesh
// and 1.9e-15 on 8^3, here 1.3e-16 and 2.1e-16, FP64 sums 1.2e-16 and 2.3e-16.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "blocks.cuh"
#include "grid.h"

namespace vlgt {

namespace {

constexpr int kMaxRun = 8;       // blocks summed before the sum goes to FP64: 2^29 multiples at most
constexpr int kWarps = 8;        // warps of a CTA, at most

struct VMesh {
    double vmin[3], dv[3];
    int nv[3];
};

// Values split at two fixed places: with s1 = 1.5 * 2^E, s2 = 1.5 * 2^(E-23) and |f| < 2^(E-1),
// t1 = f + s1 and t2 = (f - (t1 - s1)) + s2 round f to multiples of 2^(E-23) and 2^(E-46), and
// every subtraction is exact (Dekker 1971; the fixed place is that of Rump, Ogita & Oishi
// 2008).  Within its binade a float's bits count its multiples, so sums of t1 and t2 are taken
// over the bits as integers, exactly, modulo 2^32.  What is left, below 2^(E-47), is added in
// FP32: an error below 2^(E-70) per addition, far below that of an FP64 sum.
constexpr unsigned kHead = 10;             // room above the largest value, in bits
constexpr unsigned kWide = 0x7e000000u;    // bits of 2^125: from here on FP64

struct Split {  // one value, or a sum: multiples (biased), multiples (biased), rest
    unsigned a, b;
    float c;
};
struct Places {
    float s1, s2;
    // for values up to that with the bits m.  E >= -100 keeps s2 and its multiples normal; the
    // rest is then exact
    __device__ __forceinline__ void set(unsigned m)
    {
        const unsigned e = min(max((m >> 23) + 2u + kHead, 27u), 253u);
        s1 = __uint_as_float(e << 23 | 0x400000u);
        s2 = __uint_as_float((e - 23u) << 23 | 0x400000u);
    }
    // bits of 2^(E-1)
    __device__ __forceinline__ unsigned limit() const { return __float_as_uint(s1) - 0xc00000u; }
    // value i of four; two are split at a time, in packed FP32
    __device__ __forceinline__ Split split(const float (&f)[4], int i) const
    {
        const float2 v = make_float2(f[i & 2], f[i | 1]), p1 = make_float2(s1, s1), p2 = make_float2(s2, s2);
        const float2 t1 = add2(v, p1), r1 = sub2(v, sub2(t1, p1)), t2 = add2(r1, p2), r2 = sub2(r1, sub2(t2, p2));
        return i & 1 ? Split{__float_as_uint(t1.y), __float_as_uint(t2.y), r2.y}
                     : Split{__float_as_uint(t1.x), __float_as_uint(t2.x), r2.x};
    }
    __device__ __forceinline__ double unit() const  // 2^(E-46)
    {
        return __hiloint2double((int)((__float_as_uint(s1) >> 3) - 0x80000u + ((1023u - 127u - 46u) << 20)), 0);
    }
    // multiples of unit() in a sum over n values
    __device__ __forceinline__ long long multiples(const Split& x, unsigned n) const
    {
        return (long long)(int)(x.a - n * __float_as_uint(s1)) * (1 << 23) + (int)(x.b - n * __float_as_uint(s2));
    }
    __device__ __forceinline__ double value(const Split& x, unsigned n) const
    {
        return fma((double)multiples(x, n), unit(), (double)x.c);
    }
};

// Bits of the largest magnitude of three; NaN counts as larger than infinity.
__device__ __forceinline__ float top3(float a, float b, float c)
{
    float d;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ unsigned top(const float (&f)[4][4])
{
    float m = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; q++) m = top3(top3(m, f[q][0], f[q][1]), f[q][2], f[q][3]);
    return __float_as_uint(m) & 0x7fffffffu;
}

// Entry k = lane & 3 of the sum over four neighbouring lanes of p[0..3].
template <class T>
__device__ __forceinline__ T transpose_sum(const T (&p)[4], int k)
{
    const bool hi = k & 2, odd = k & 1;
    const T a0 = (hi ? p[2] : p[0]) + __shfl_xor_sync(0xffffffffu, hi ? p[0] : p[2], 2);
    const T a1 = (hi ? p[3] : p[1]) + __shfl_xor_sync(0xffffffffu, hi ? p[1] : p[3], 2);
    return (odd ? a1 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 1);
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
    // four chains each (index modulo 4): shorter sums round less
    double a[4] = {}, b[4] = {};
    for (int i = 0; i < nd; i += 4)
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const double f = M[(i + q) * kGroup];
            a[q] += f;
            b[q] += (vmin + (i + q + 0.5) * dv) * f;
        }
    const double s0 = (a[0] + a[1]) + (a[2] + a[3]), s1 = (b[0] + b[1]) + (b[2] + b[3]);
    const double n = __shfl_sync(0xffffffffu, s0, lane & ~3);
    const double mean = n != 0.0 ? s1 / n : 0.0;
    for (int q = 0; q < 4; q++) a[q] = 0.0;
    for (int i = 0; i < nd; i += 4)
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const double w = (vmin + (i + q + 0.5) * dv) - mean;
            a[q] += w * w * M[(i + q) * kGroup];
        }
    const double s2 = (a[0] + a[1]) + (a[2] + a[3]);
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
    unsigned za[4] = {}, zb[4] = {};
    float zc[4] = {};
    Places at;
    at.set(0u);
    int run = 0, row_of_run = -1;
    auto flush = [&]() {
        if (run == 0) return;
        const Split y{za[0] + za[1] + za[2] + za[3], zb[0] + zb[1] + zb[2] + zb[3], (zc[0] + zc[1]) + (zc[2] + zc[3])};
        const Split z{transpose_sum(za, k), transpose_sum(zb, k), transpose_sum(zc, k)};
        ay[(row_of_run % G.nby) * 4 * kGroup] += at.value(y, 16u * run);
        az[(row_of_run / G.nby) * 4 * kGroup] += at.value(z, 16u * run);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            za[q] = zb[q] = 0u;
            zc[q] = 0.0f;
        }
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
        float f[4][4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 v = r.get(q);
            f[q][0] = v.x;
            f[q][1] = v.y;
            f[q][2] = v.z;
            f[q][3] = v.w;
        }
        unsigned m = top(f);
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
        if (brow != row_of_run || run == kMaxRun || __any_sync(0xffffffffu, m >= at.limit())) {
            if (__any_sync(0xffffffffu, m >= kWide)) {
                // values near the end of FP32's range, infinities and NaN: FP64 for this block
                double dx[4], dz[4], dy = 0.0;
                for (int i = 0; i < 4; i++) {
                    dx[i] = ((double)f[0][i] + f[1][i]) + ((double)f[2][i] + f[3][i]);
                    dz[i] = ((double)f[i][0] + f[i][1]) + ((double)f[i][2] + f[i][3]);
                    dy += dz[i];
                }
                ax[bx * 4 * kGroup] += transpose_sum(dx, k);
                ay[(brow % G.nby) * 4 * kGroup] += dy;
                az[(brow / G.nby) * 4 * kGroup] += transpose_sum(dz, k);
                return;
            }
            flush();
            at.set(m);
            row_of_run = brow;
        }
        unsigned xa[4] = {}, xb[4] = {};
        float xc[4] = {};
#pragma unroll
        for (int q = 0; q < 4; q++)
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const Split p = at.split(f[q], i);
                za[q] += p.a;
                zb[q] += p.b;
                zc[q] += p.c;
                xa[i] += p.a;
                xb[i] += p.b;
                xc[i] += p.c;
            }
        run++;
        const Split x{transpose_sum(xa, k), transpose_sum(xb, k), transpose_sum(xc, k)};
        // at most 2^49 multiples in magnitude: as an FP64 number by its bits, without a conversion
        const double n = __longlong_as_double(at.multiples(x, 16u) + 0x4338000000000000ll) - 0x1.8p52;
        ax[bx * 4 * kGroup] += fma(n, at.unit(), (double)x.c);
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
    Split p{0u, 0u, 0.0f};
    Places at;
    at.set(0u);
    unsigned run = 0;
    const int b_begin = blockIdx.y * P.ids, b_end = min(G.nb, b_begin + P.ids);
    const int64_t row = grp / P.per_row;
    const int x0 = (int)(grp - row * P.per_row) * kGroup;
    auto load = [&](int, bool has, int64_t chunk, uint32_t cnt) {
        Rows<kCodec> r;
        r.load(L, chunk, cnt, k, has);
        return r;
    };
    for_blocks<Rows<kCodec>>(G, L, row, x0, 0xffu, b_begin, b_end, load, [&](int, const Rows<kCodec>& r, bool, int64_t, uint32_t) {
        float f[4][4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 v = r.get(q);
            f[q][0] = v.x;
            f[q][1] = v.y;
            f[q][2] = v.z;
            f[q][3] = v.w;
        }
        const unsigned m = top(f);
        if (run == kMaxRun || m >= at.limit()) {
            if (m >= kWide) {  // values near the end of FP32's range, infinities and NaN
                for (int q = 0; q < 4; q++) sum += ((double)f[q][0] + f[q][1]) + ((double)f[q][2] + f[q][3]);
                return;
            }
            sum += at.value(p, 16u * run);
            p = {0u, 0u, 0.0f};
            run = 0;
            at.set(m);
        }
#pragma unroll
        for (int q = 0; q < 4; q++)
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const Split v = at.split(f[q], i);
                p.a += v.a;
                p.b += v.b;
                p.c += v.c;
            }
        run++;
    });
    sum += at.value(p, 16u * run);
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    const int x = x0 + j;
    if (k == 0 && x < G.n[0]) dens[(int64_t)blockIdx.y * G.N + row * G.n[0] + x] = sum * (V.dv[0] * V.dv[1] * V.dv[2]);
}

// out[blockIdx.x] = sum of this CTA's share of v[0 .. n-1], in an order that n and the grid fix;
// compensated (TwoSum, Knuth 1969), so that its length costs no precision.
__global__ void __launch_bounds__(256) k_sum(const double* __restrict__ v, int64_t n, double* __restrict__ out)
{
    __shared__ double sh[2][8];
    double s = 0.0, e = 0.0;
    auto add = [&](double a) {
        const double t = s + a, b = t - s;
        e += (s - (t - b)) + (a - b);
        s = t;
    };
    for (int64_t c = (int64_t)blockIdx.x * 256 + threadIdx.x; c < n; c += (int64_t)gridDim.x * 256) add(v[c]);
    for (int o = 16; o > 0; o >>= 1) {
        const double a = __shfl_xor_sync(0xffffffffu, s, o), b = __shfl_xor_sync(0xffffffffu, e, o);
        add(a);
        e += b;
    }
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = s;
        sh[1][threadIdx.x >> 5] = e;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 8; w++) {
        add(sh[0][w]);
        e += sh[1][w];
    }
    // infinities have no low part
    out[blockIdx.x] = fabs(s) < (double)INFINITY ? s + e : s;
}
constexpr int kSums = 152;  // CTAs of the first stage

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

// Sixteen warps for each of a GB300's SMs; a constant, so that the parts, and with them the last
// bits of the sums over parts, depend on the grid alone, and not on the GPU.
constexpr int64_t kWantWarps = 152 * 16;

Groups groups_of(const Grid* g)
{
    const GridGeom& G = g->geom;
    Groups P;
    P.per_row = (G.n[0] + kGroup - 1) / kGroup;
    P.total = (int64_t)P.per_row * G.R;
    const Parts s = parts_of(G.nb, P.total, kWantWarps, 64);  // a part has marginals to join
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
// The limit of a launch belongs to the kernel, not to the grid, and can be lowered: it is set
// to the same value before every launch, so that a grid on another host thread never takes it
// away between the two calls.
template <class Kernel>
void raise_smem(Kernel kern)
{
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemCta);
}

}  // namespace

bool moments_fit(const Grid* g) { return warp_bytes(g) <= kSmemCta; }

// Small grids take scratch from the caller's allocator, returned in *scratch.
vl_status queue_moments(Grid* g, double* d_out, void** scratch)
{
    const GridGeom& G = g->geom;
    const LayoutView L = g->lay[g->cur].view();
    const VMesh V = vmesh_of(g);
    const Groups P = groups_of(g);
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
        raise_smem(kern);
        kern<<<dim3(ctas, P.split), warps * 32, smem, g->stream>>>(G, L, V, P, parts ? parts : d_out);
    });
    note_launch();
    if (P.split > 1) {
        raise_smem(k_join_marginals);
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
    const Groups P = groups_of(g);
    // densities of the parts, the sums of shares of them, the total
    const int64_t n = (int64_t)P.split * G.N;
    const int sums = (int)std::min<int64_t>((n + 255) / 256, kSums);
    double* dens = (double*)g->alloc(((size_t)n + sums + 1) * sizeof(double));
    if (!dens) return fail(g, VL_ENOMEM, "vl_mass: scratch allocation failed");
    double* acc = dens + n + sums;
    with_codec(g->codec, [&](auto c) {
        k_density<decltype(c)::value>
            <<<dim3((unsigned)((P.total + kWarps - 1) / kWarps), P.split), kWarps * 32, 0, g->stream>>>(
                G, g->lay[g->cur].view(), V, P, dens);
    });
    note_launch();
    k_sum<<<sums, 256, 0, g->stream>>>(dens, n, dens + n);
    k_sum<<<1, 256, 0, g->stream>>>(dens + n, sums, acc);
    note_launch();
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
