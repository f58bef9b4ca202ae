// lists.cu -- conversion between the pool and per-cell block lists, cell by cell.
//
// A block is 256 contiguous bytes of a cell's list and four 64-byte chunks of the pool, and
// neighbouring cells' chunks of one id lie side by side in the pool.  A warp takes eight
// neighbouring cells (blocks.cuh) and walks the ids that any of them holds: per id and chunk
// it moves up to 512 contiguous bytes on the pool's side and 64 on each list's, and the lists
// grow as eight streams.  A cell's position in its list is a running count, so no per-block
// index is built or read; where the ids are split over warps, counts per part give each
// part's first position.  Bound by memory: both sides are moved once, in whole sectors.
//
// Measured (64x64x16 cells x 32^3, 33.5 million blocks, 8.6 GB of values; 2.53 ms at the copy
// rate): out 2.80 ms and in 2.56 ms; one thread per value, with the block's slot and cell
// looked up by each, 9.36 and 10.1.  Counting the blocks of 32768 cells x 4096 ids: 0.07 ms,
// one thread per cell 0.77.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "blocks.cuh"
#include "grid.h"

namespace vlgt {

namespace {

constexpr int kWarps = 8;

// Groups of a window: the aligned groups of eight cells of every grid row it touches.
struct WindowGroups {
    Window W;
    Parts parts;
    int per_row;
    int64_t total;
};

// This lane's place in a group: lane 4 j + k (kQuad) or lane j (< 8) is cell j.
struct Place {
    int64_t row;   // grid row
    int64_t cell;  // window cell, when `in`
    int x0;
    unsigned mask;  // the group's cells that lie in the window
    bool in;
};
template <bool kQuad>
__device__ __forceinline__ Place place(const GridGeom& G, const WindowGroups& P, int64_t grp)
{
    const int lane = threadIdx.x & 31, j = kQuad ? lane >> 2 : lane;
    const int64_t r = grp / P.per_row;
    Place p;
    p.x0 = (int)(grp - r * P.per_row) * kGroup;
    const int wy = (int)(r % P.W.s[1]), wz = (int)(r / P.W.s[1]);
    p.row = wrapi(P.W.o[1] + wy, G.n[1]) + (int64_t)G.n[1] * wrapi(P.W.o[2] + wz, G.n[2]);
    const int wx = wrapi(p.x0 + j - P.W.o[0], G.n[0]);
    p.in = (kQuad || lane < kGroup) && p.x0 + j < G.n[0] && wx < P.W.s[0];
    p.cell = wx + (int64_t)P.W.s[0] * r;
    const unsigned b = __ballot_sync(0xffffffffu, p.in);
    if (kQuad) {
        p.mask = 0u;
#pragma unroll
        for (int i = 0; i < kGroup; i++) p.mask |= ((b >> (4 * i)) & 1u) << i;
    } else {
        p.mask = b & 0xffu;
    }
    return p;
}

// Blocks of every window cell with an id of the part: cnt[part][cell].
__global__ void __launch_bounds__(kWarps * 32) k_part_counts(GridGeom G, const uint64_t* __restrict__ kbits,
                                                             WindowGroups P, uint32_t* __restrict__ cnt)
{
    const int64_t grp = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (grp >= P.total) return;
    const int lane = threadIdx.x & 31;
    const Place p = place<false>(G, P, grp);
    if (!p.mask) return;
    const int64_t word = p.row * G.W + (p.x0 >> 6);
    const int b1 = min(G.nb, (int)(blockIdx.y + 1) * P.parts.ids);
    uint32_t n = 0;
    constexpr int kAhead = 4;  // rounds of 32 words in flight
    for (int b = blockIdx.y * P.parts.ids + lane; b - lane < b1; b += 32 * kAhead) {
        uint64_t k[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; i++) k[i] = b + 32 * i < b1 ? kbits[(int64_t)(b + 32 * i) * G.RW + word] : 0ull;
#pragma unroll
        for (int i = 0; i < kAhead; i++) {
            const unsigned k8 = (unsigned)(k[i] >> (p.x0 & 63)) & p.mask;
            if (!__any_sync(0xffffffffu, k8 != 0u)) continue;
#pragma unroll
            for (int j = 0; j < kGroup; j++) {
                const unsigned cells = __ballot_sync(0xffffffffu, (k8 >> j) & 1u);
                if (lane == j) n += __popc(cells);
            }
        }
    }
    if (p.in) cnt[(int64_t)blockIdx.y * P.W.ncell + p.cell] = n;
}

// cnt[part][cell] -> blocks of the cell in earlier parts; total[cell] (optional) their sum.
__global__ void k_part_starts(int64_t ncell, int parts, uint32_t* __restrict__ cnt, uint32_t* __restrict__ total)
{
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    uint32_t n = 0;
    for (int p = 0; p < parts; p++) {
        const uint32_t k = cnt[p * ncell + c];
        cnt[p * ncell + c] = n;
        n += k;
    }
    if (total) total[c] = n;
}

__device__ __forceinline__ float4 load_row(const float* p, bool aligned)
{
    return aligned ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void store_row(float* p, const float4& v, bool aligned)
{
    if (aligned) {
        *reinterpret_cast<float4*>(p) = v;
    } else {
        p[0] = v.x;
        p[1] = v.y;
        p[2] = v.z;
        p[3] = v.w;
    }
}

// Pool -> lists (ids and values).  start: nullptr with one part.
// kWide: a cell's block goes through shared memory and is written as 256 contiguous bytes by
// 16 lanes -- for a host buffer, which takes them at 189 GB/s against 177 in 64-byte pieces;
// device memory merges those in L2.
constexpr int kCellPitch = 68;  // floats; cells 4 banks apart
template <int kCodec, bool kWide>
__global__ void __launch_bounds__(kWarps * 32, 4) k_blocks_out(GridGeom G, LayoutView L, WindowGroups P,
                                                               const int64_t* __restrict__ off,
                                                               const uint32_t* __restrict__ start,
                                                               uint16_t* __restrict__ ids,
                                                               float* __restrict__ vals, bool aligned)
{
    const int64_t grp = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (grp >= P.total) return;
    const int k = threadIdx.x & 3;
    const Place p = place<true>(G, P, grp);
    if (!p.mask) return;
    int64_t t = p.in ? off[p.cell] : 0;
    if (p.in && start) t += start[(int64_t)blockIdx.y * P.W.ncell + p.cell];
    const int b0 = blockIdx.y * P.parts.ids, b1 = min(G.nb, b0 + P.parts.ids);
    __shared__ __align__(16) float s_wide[kWide ? kWarps * kGroup * kCellPitch : 4];
    const int lane = threadIdx.x & 31;
    float* const wide = s_wide + (kWide ? (threadIdx.x >> 5) * kGroup * kCellPitch : 0);
    auto load = [&](int, bool has, int64_t chunk, uint32_t cnt) {
        Rows<kCodec> r;
        r.load(L, chunk, cnt, k, has);
        return r;
    };
    auto body = [&](int b, const Rows<kCodec>& r, bool has, int64_t, uint32_t) {
        if (has && k == 0) ids[t] = (uint16_t)b;
        if constexpr (kWide) {
            __syncwarp();
            float* mine = wide + (lane >> 2) * kCellPitch + 4 * k;
#pragma unroll
            for (int q = 0; q < 4; q++) store_row(mine + q * kChunk, r.get(q), true);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kGroup / 2; i++) {
                // cells 2 i and 2 i + 1, sixteen lanes each
                const int j = 2 * i + (lane >> 4), piece = 4 * (lane & 15);
                const int64_t tj = __shfl_sync(0xffffffffu, has ? t : -1, 4 * j);
                if (tj >= 0)
                    store_row(vals + tj * 64 + piece, *reinterpret_cast<const float4*>(wide + j * kCellPitch + piece),
                              aligned);
            }
        } else if (has) {
            float* dst = vals + t * 64 + 4 * k;
#pragma unroll
            for (int q = 0; q < 4; q++) store_row(dst + q * kChunk, r.get(q), aligned);
        }
        if (has) t++;
    };
    for_blocks<Rows<kCodec>>(G, L, p.row, p.x0, p.mask, b0, b1, load, body);
}

struct ListRows {
    float4 v[4];
};

// Lists -> pool, into the slots of the blocks that the layout holds (kbits): the lists hold
// exactly those, in ascending order.
template <int kCodec>
__global__ void __launch_bounds__(kWarps * 32, 4) k_blocks_in(GridGeom G, LayoutView L, WindowGroups P,
                                                              const int64_t* __restrict__ off,
                                                              const uint32_t* __restrict__ start,
                                                              const float* __restrict__ vals, bool aligned)
{
    using T = typename Codec<kCodec>::T;
    const int64_t grp = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (grp >= P.total) return;
    const int k = threadIdx.x & 3;
    const Place p = place<true>(G, P, grp);
    if (!p.mask) return;
    int64_t t = p.in ? off[p.cell] : 0;
    if (p.in && start) t += start[(int64_t)blockIdx.y * P.W.ncell + p.cell];
    const int b0 = blockIdx.y * P.parts.ids, b1 = min(G.nb, b0 + P.parts.ids);
    auto load = [&](int, bool has, int64_t, uint32_t) {
        ListRows r;
        const float* src = vals + t * 64 + 4 * k;
#pragma unroll
        for (int q = 0; q < 4; q++) r.v[q] = has ? load_row(src + q * kChunk, aligned) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (has) t++;
        return r;
    };
    for_blocks<ListRows>(G, L, p.row, p.x0, p.mask, b0, b1, load,
                         [&](int, const ListRows& r, bool has, int64_t chunk, uint32_t cnt) {
#pragma unroll
                             for (int q = 0; q < 4; q++) {
                                 const int64_t c = chunk + (int64_t)q * cnt;
                                 T* dst = static_cast<T*>(L.pool) + c * kChunk + 4 * k;
                                 const float4 v = r.v[q];
                                 if constexpr (kCodec == 0) {
                                     if (has) *reinterpret_cast<float4*>(dst) = v;
                                 } else {
                                     // the chunk's largest magnitude, over its four lanes, as bits
                                     // (ordered like the magnitudes, NaN last)
                                     unsigned m = max(max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y))),
                                                      max(__float_as_uint(fabsf(v.z)), __float_as_uint(fabsf(v.w))));
                                     m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
                                     m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
                                     const ChunkScale cs = chunk_scale(__uint_as_float(m));
                                     const float f[4] = {v.x, v.y, v.z, v.w};
                                     uint2 raw;
                                     T* h = reinterpret_cast<T*>(&raw);
#pragma unroll
                                     for (int i = 0; i < 4; i++) h[i] = Codec<kCodec>::enc(f[i], cs.inv);
                                     if (has) {
                                         *reinterpret_cast<uint2*>(dst) = raw;
                                         if (k == 0) L.scale[c] = cs.s;
                                     }
                                 }
                             }
                         });
}

// Checks the lists (err bit 1: id out of range, bit 2: ids not strictly increasing within
// a cell) and marks their blocks in ubits; one warp per cell.  Nothing is walked when the
// offsets are known to be invalid (err bit 0, from the check queued before): each cell could
// then claim the whole list, and the work would be cells times blocks.
__global__ void __launch_bounds__(kWarps * 32) k_mark_cells(GridGeom G, const int64_t* __restrict__ off,
                                                            const uint16_t* __restrict__ ids, int64_t M,
                                                            uint64_t* __restrict__ ubits, int* __restrict__ err)
{
    const int64_t c = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (c >= G.N || (*(volatile const int*)err & 1)) return;
    const int64_t lo = max((int64_t)0, off[c]), hi = min(M, off[c + 1]);
    const int x = (int)(c % G.n[0]);
    uint64_t* words = ubits + c / G.n[0] * G.W + (x >> 6);
    int bad = 0;
    for (int64_t t = lo + (threadIdx.x & 31); t < hi; t += 32) {
        const int b = ids[t];
        if (t > lo && ids[t - 1] >= b) bad |= 4;
        if (b >= G.nb) {
            bad |= 2;
            continue;
        }
        atomicOr((unsigned long long*)&words[(int64_t)b * G.RW], (unsigned long long)(1ull << (x & 63)));
    }
    if (bad) atomicOr(err, bad);
}

WindowGroups groups_of(const GridGeom& G, const Window& W)
{
    WindowGroups P;
    P.W = W;
    for (int d = 0; d < 3; d++) P.W.o[d] = ((W.o[d] % G.n[d]) + G.n[d]) % G.n[d];
    P.per_row = (G.n[0] + kGroup - 1) / kGroup;
    P.total = (int64_t)P.per_row * W.s[1] * W.s[2];
    P.parts = parts_of(G.nb, P.total, 152 * 32, 8);
    return P;
}

dim3 grid_of(const WindowGroups& P)
{
    return dim3((unsigned)((P.total + kWarps - 1) / kWarps), (unsigned)P.parts.split);
}

}  // namespace

int list_parts(const Grid* g, const Window& W) { return groups_of(g->geom, W).parts.split; }

void launch_list_counts(Grid* g, const uint64_t* kbits, const Window& W, uint32_t* cnt, uint32_t* total)
{
    const WindowGroups P = groups_of(g->geom, W);
    if (P.parts.split == 1 && !total) return;  // every list starts at its offset
    uint32_t* dst = P.parts.split == 1 ? total : cnt;
    k_part_counts<<<grid_of(P), kWarps * 32, 0, g->stream>>>(g->geom, kbits, P, dst);
    note_launch();
    if (P.parts.split == 1) return;
    k_part_starts<<<(unsigned)((W.ncell + 255) / 256), 256, 0, g->stream>>>(W.ncell, P.parts.split, cnt, total);
    note_launch();
}

void launch_blocks_out(Grid* g, const Layout& L, const Window& W, const int64_t* off, const uint32_t* start,
                       uint16_t* ids, float* vals, bool host)
{
    const WindowGroups P = groups_of(g->geom, W);
    if (P.parts.split == 1) start = nullptr;
    with_codec(g->codec, [&](auto c) {
        constexpr int kc = decltype(c)::value;
        auto kern = host ? k_blocks_out<kc, true> : k_blocks_out<kc, false>;
        kern<<<grid_of(P), kWarps * 32, 0, g->stream>>>(g->geom, L.view(), P, off, start, ids, vals,
                                                        ((uintptr_t)vals & 15) == 0);
    });
    note_launch();
}

void launch_blocks_in(Grid* g, const Layout& L, const Window& W, const int64_t* off, const uint32_t* start,
                      const float* vals)
{
    const WindowGroups P = groups_of(g->geom, W);
    if (P.parts.split == 1) start = nullptr;
    with_codec(g->codec, [&](auto c) {
        k_blocks_in<decltype(c)::value><<<grid_of(P), kWarps * 32, 0, g->stream>>>(
            g->geom, L.view(), P, off, start, vals, ((uintptr_t)vals & 15) == 0);
    });
    note_launch();
}

void launch_mark_cells(Grid* g, const int64_t* off, const uint16_t* ids, int64_t M, uint64_t* ubits, int* err)
{
    k_mark_cells<<<(unsigned)((g->geom.N + kWarps - 1) / kWarps), kWarps * 32, 0, g->stream>>>(g->geom, off, ids, M,
                                                                                               ubits, err);
    note_launch();
}

}  // namespace vlgt
