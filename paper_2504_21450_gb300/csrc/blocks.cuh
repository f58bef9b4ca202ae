// blocks.cuh -- walk over the blocks of a few cells, shared by the kernels that read or write
// whole blocks (moments, per-cell lists).
//
// A warp takes a group of eight cells that are neighbours along x (aligned, so that they
// share one bitmap word), four lanes per cell: lane 4 j + k has the vx row k (16 bytes in
// FP32) of every chunk of cell j, so a load or store covers up to eight 64-byte chunks in a
// row of the pool.  The block ids are walked in ascending order, 32 bitmap words at a time,
// with the next block's values in flight while one is used.
#pragma once
#include "common.cuh"

namespace vlgt {

constexpr int kGroup = 8;  // cells of a warp

// One vx row of each of a block's four chunks, as stored.
template <int kCodec>
struct Rows {
    float4 v[4];
    __device__ __forceinline__ void load(const LayoutView& L, int64_t chunk, uint32_t cnt, int k, bool has)
    {
#pragma unroll
        for (int q = 0; q < 4; q++)
            v[q] = has ? __ldcs(reinterpret_cast<const float4*>(static_cast<const float*>(L.pool) +
                                                                 (chunk + (int64_t)q * cnt) * kChunk) + k)
                       : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ float4 get(int q) const { return v[q]; }
};
template <int kCodec>
struct Codes {
    uint2 v[4];
    float s[4];
    __device__ __forceinline__ void load(const LayoutView& L, int64_t chunk, uint32_t cnt, int k, bool has)
    {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int64_t c = chunk + (int64_t)q * cnt;
            v[q] = has ? __ldcs(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(L.pool) + c * kChunk) + k)
                       : make_uint2(0u, 0u);
            s[q] = has ? L.scale[c] : 0.0f;
        }
    }
    __device__ __forceinline__ float4 get(int q) const
    {
        using T = typename Codec<kCodec>::T;
        const T* h = reinterpret_cast<const T*>(&v[q]);
        return make_float4(Codec<kCodec>::dec(h[0], s[q]), Codec<kCodec>::dec(h[1], s[q]),
                           Codec<kCodec>::dec(h[2], s[q]), Codec<kCodec>::dec(h[3], s[q]));
    }
};
template <> struct Rows<1> : Codes<1> {};
template <> struct Rows<2> : Codes<2> {};

// The blocks with ids b_begin .. b_end-1 that any of the cells of `mask` (bit j: cell x0 + j)
// of a row holds, in ascending order.  load(id, has, chunk, cnt) -> payload is called for a
// block before the body of the one before it; body(id, payload, has, chunk, cnt).  has: this
// lane's cell is of the mask and holds the block, in slot `chunk` of chunk 0 (chunk q lies
// q * cnt further).
template <class Payload, class Load, class Body>
__device__ __forceinline__ void for_blocks(const GridGeom& G, const LayoutView& L, int64_t row, int x0,
                                           unsigned mask, int b_begin, int b_end, Load&& load, Body&& body)
{
    const int lane = threadIdx.x & 31, j = lane >> 2;
    const int64_t word = row * G.W + (x0 >> 6);
    const int sh = x0 & 63;
    auto kept = [&](int b) -> uint64_t { return b < b_end ? L.kbits[(int64_t)b * G.RW + word] : 0ull; };
    uint64_t kw = kept(b_begin + lane);
    for (int b0 = b_begin; b0 < b_end; b0 += 32) {
        const unsigned k8 = (unsigned)(kw >> sh) & mask;
        unsigned m = __ballot_sync(0xffffffffu, k8 != 0u);
        kw = kept(b0 + 32 + lane);  // the next words, while this batch is used
        if (!m) continue;
        // lane i: cells (kept, slots), first chunk and chunk stride of block id b0 + i
        unsigned bits = 0u;
        int64_t first = 0;
        uint32_t cnt = 0u;
        if (k8) {
            const int b = b0 + lane;
            const uint64_t u = L.ubits[(int64_t)b * G.RW + word];
            bits = k8 | ((unsigned)(u >> sh) & 0xffu) << 8;
            first = L.base[b] * 4 + L.woff[(int64_t)b * G.RW + word] + __popcll(u & ((1ull << sh) - 1ull));
            cnt = L.cnt[b];
        }
        struct Entry {
            Payload p;
            int64_t chunk;
            uint32_t cnt;
            bool has;
        };
        Entry cur, nxt;
        auto fetch = [&](int i, Entry& e) {
            const unsigned bi = __shfl_sync(0xffffffffu, bits, i);
            e.cnt = __shfl_sync(0xffffffffu, cnt, i);
            e.has = (bi >> j) & 1u;
            e.chunk = __shfl_sync(0xffffffffu, first, i) + __popc((bi >> 8) & ((1u << j) - 1u));
            e.p = load(b0 + i, e.has, e.chunk, e.cnt);
        };
        int i = __ffs(m) - 1;
        fetch(i, cur);
        while (true) {
            m &= m - 1u;
            const int in = m ? __ffs(m) - 1 : -1;
            if (in >= 0) fetch(in, nxt);
            body(b0 + i, cur.p, cur.has, cur.chunk, cur.cnt);
            if (in < 0) break;
            i = in;
            cur = nxt;
        }
    }
}

// A box of cells of the periodic grid, x fastest.
struct Window {
    int o[3], s[3];  // origin (any integers) and extents (at most the grid's)
    int64_t ncell;
};

// Block ids split over CTAs where the groups alone leave the chip idle: a group's ids are a
// serial chain, about 0.7 us a block.  As many parts as give `want` warps, of at least
// `least` ids.
struct Parts {
    int split, ids;  // parts, ids of a part
};
inline Parts parts_of(int nb, int64_t groups, int64_t want, int least)
{
    const int64_t most = (nb + least - 1) / least;
    int64_t split = want / (groups > 0 ? groups : 1);
    split = split < 1 ? 1 : split > most ? most : split;
    Parts p;
    p.ids = (int)(((nb + split - 1) / split + 7) / 8 * 8);
    p.split = (nb + p.ids - 1) / p.ids;
    return p;
}

}  // namespace vlgt
