// gt3.cu -- Ghost Translation (GT3) on one GPU, plane-batched kernel (paper Section 3).
//
// Same computation as the row-segment kernel of fused.cu: a work item is (block id b,
// velocity chunk q, tile of 16 x 16 cells across the two in-plane axes); the tile plus
// its 3-cell ghost halo (Section 3.1: the 2-cell stencil and one face neighbour) is
// staged into shared memory plane by plane along the third (streamed) axis, exactly once
// per step, and all three sweeps run on it.  What differs is how the work is laid out on
// the SM:
//   * planes are processed in batches of three, in two batch buffers.  Sixteen warps sweep;
//     four more stage, up to two batches ahead and across items, with TMA bulk copies (one
//     per contiguous run of a row; 16-byte cp.async for the short run where a dense row
//     wraps around the periodic grid).  A batch's mbarrier tells the sweeping warps that it
//     is staged, a second one tells the staging warps that it is swept.  (Until the staging
//     had warps of its own, the four warps that sit out sweep 1 did it; on sparse and 16-bit
//     states it took 7000-8400 cycles of a 13000-cycle batch and the others waited: 19.5
//     against 16.2 ms per step on 128x32x16 cells of the shock, 10.3 against 8.8 ms in
//     bfloat16 on 64x64x16 cells of the uniform workload; dense FP32 is as fast either way.)
//     The sweeping warps synchronise twice a batch, after sweep 0 and after sweep 1;
//   * every walk moves two velocity cells in packed f32x2 registers: sweep 0 runs on the
//     21 halo lines that sweep 1 reads (3 planes x 21 lines x 8 lane pairs = 504 walks),
//     sweep 1 on the 16 tile lines (384 walks), both in place in shared memory.  Only the
//     21 x 21 cells that the walks read are staged;
//   * sweep 2 is streamed: each compute thread keeps the windows of four velocity cells
//     (one vx row of a chunk) of two tile cells in registers, reads them with 16-byte
//     shared loads and writes 16-byte global stores, so a warp writes 8 whole cells.
// All walks start on the upwind side (Walk2), so the velocity cells of an item must all
// move the same way along each axis: no velocity block may straddle v_d = 0 (the host
// checks), and the streamed axis must not be x (the chunk's vx cells have different
// Courant numbers along x, and x is the contiguous axis of the staged rows).
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "grid.h"

namespace vlgt {

namespace {

constexpr int kT = 16;                      // tile edge along both in-plane axes
constexpr int kE = kT + 2 * kHalo;          // 22 staged cells per in-plane axis
constexpr int kNB = 3;                      // planes per batch
constexpr int kNC = 512;                    // sweeping threads (warps 0-15)
constexpr int kNS = 128;                    // staging threads (warps 16-19)
constexpr int kNT = kNC + kNS;
// Registers per thread: the CTA is launched with 96 (640 threads); the staging warps give
// some back and the sweeping ones take them: 512 x 104 + 128 x 64 = 640 x 96.  (112 and 32
// make the staging code spill; 13.94 against 13.98 ms on 64x64x32 cells.)
constexpr int kRegsSweep = 104, kRegsStage = 64;
static_assert(kNC * kRegsSweep + kNS * kRegsStage <= kNT * 96, "register split within the launch's total");
constexpr int kLines = kT + 5;              // sweep-0 lines: those sweep 1 reads
constexpr int kFirst = kHalo + 2;           // first streamed plane that completes an output

constexpr int kRP = kE * kChunk + 16;       // staged row pitch in floats: rows 16 banks apart
constexpr int kPS = kE * kRP + 16;          // plane pitch in floats
constexpr int kNX = kNB * kLines * 8;       // sweep-0 walks per batch (lane pairs)
constexpr int kNY = kNB * kT * 8;           // sweep-1 walks per batch
static_assert(kNX <= kNC && kNY <= kNC, "walks of a batch must fit the threads");
static_assert(kT * kT * 4 == 2 * kNC, "sweep 2: two tile cells x one vx row per thread");
// 16-bit storage with sweep 0 along x: the codes of a staged row are packed (8 floats per
// cell) at the end of the row that sweep 0 reaches last -- from float kCodesHi when it
// walks up, from float 0 when it walks down
constexpr int kCodesHi = kRP - kE * kChunk / 2;

// One work item: block id b, velocity chunk q, tile origin and extent.
struct Item {
    int b, q, tx0, tr0, ex, er;
    int dense_in, dense_out, up0, up1, up2;
    int64_t ibase, obase, okeep;
};

// What the threads read for an item: its staged rows and its sweep constants.
struct ItemTables {
    float4 kc[3][kChunk];  // WalkConst (g, A, B, up) per sweep and velocity cell
    int run[kE][3];        // contiguous runs of a staged row along x: first column, x, length
    int rrow[kE];          // row-space part of each row
    int xs[kE];            // x of each column
    int nrun;
    int r0, u0;            // first staged row and column (kLines of each are staged)
};

struct Gt3Smem {
    float buf[2][kNB][kPS];   // staged planes, swept in place (two batches in flight)
    int orank[2][kNB][kT * kT];  // sparse output slots of the tile cells, per plane
    Item item[2];             // per item parity, like the tables and the work index
    ItemTables tab[2];
    long long work[2];
    uint64_t bar[2];          // per batch buffer: staged
    uint64_t empty[2];        // per batch buffer: swept, may be staged again
    int abort;                // a sweeping warp's wait ran out
    int late;                 // the staging warps' wait ran out
};
// 16-bit storage: the chunk scales of the staged cells, [2][kNB][kE][kSP] floats after
// Gt3Smem (per batch buffer and plane, staged row-major like the cells).  The row pitch
// is odd, so that the staging threads, one per row, write 32 different banks.
constexpr int kSP = kE + 1;
constexpr int kScales = 2 * kNB * kE * kSP;
template <int kCodec>
constexpr size_t smem_bytes() { return sizeof(Gt3Smem) + (kCodec ? kScales * sizeof(float) : 0); }
__device__ __forceinline__ float* scales_of(Gt3Smem& S) { return reinterpret_cast<float*>(&S + 1); }
static_assert(smem_bytes<1>() <= 227 * 1024, "shared memory of one CTA");

struct Gt3Args {
    GridGeom G;
    LayoutView in, out;
    int ax[3];          // physical axis of sweep 0, 1, 2 (axis 2 is streamed, never x)
    int ar;             // the in-plane axis that is not x
    int64_t stride[3];  // cell-index stride of each physical axis (1, nx, nx*ny)
    const float4* walk; // [3][nvmax] WalkConst (g, A, B, up) per axis and velocity index
    int nvmax;
    float thr;
    int ntile0;         // tiles along x
    uint32_t ntiles;    // tiles per block id
    const uint32_t* items;   // (block id, tile) pairs as b * ntiles + tile, in that order
    const int64_t* npairs;   // their number
    uint8_t* keepq;
    StepCounters* ctr;
    int testing;        // testing hooks, see kTestLate and kTestSlots
    uint64_t* cta_done; // optional [gridDim.x]: %globaltimer when the CTA ran out of work
};

// Testing hooks (Gt3Args::testing).  kTestLate: a staging wait not complete at its first poll
// is reported as overdue (VL_ETIMEOUT), then waited for.  kTestSlots: the staging warps sleep
// before they write a batch's output slots, so that a sweeping warp which were not made to
// wait for them would read those of an earlier batch.
constexpr int kTestLate = 1, kTestSlots = 2;
constexpr unsigned kTestSlotsNs = 50000;  // a batch is swept in about 5 us

__device__ __forceinline__ unsigned su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint64_t* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_add_tx(uint64_t* bar, unsigned bytes)
{
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;\n" ::"r"(su32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(su32(bar)) : "memory");
}
// Waits for the phase for up to about kSuspendNs before it says no.  Asleep, a waiting warp
// takes no issue slots from the warps that sweep on its scheduler: without the hint the thread
// that waits for an empty buffer polled some 200 times a batch (64x64x32 cells of the uniform
// workload 13.60 ms a sweep, now 13.42; 50x37x29 in z, x, y order 7.50, now 7.40; the shock
// and bfloat16, where staging has less time to spare, 0.3 and 0.2 % less).
constexpr unsigned kSuspendNs = 20000;
__device__ __forceinline__ bool bar_try(uint64_t* bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(bar)), "r"(parity), "r"(kSuspendNs)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_test(uint64_t* bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t now_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}
__device__ __forceinline__ void copy_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            su32(dst)),
        "l"(src), "r"(bytes), "r"(su32(bar))
        : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
// 16-byte copy global -> shared; src_bytes = 0 fills the 16 bytes with zeros
__device__ __forceinline__ void cp16(void* dst, const void* src, int src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(su32(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
}
// 4-byte copy global -> shared; src_bytes = 0 writes 0
__device__ __forceinline__ void cp4(void* dst, const void* src, int src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(su32(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
}
// the barrier's pending count drops by one once this thread's earlier cp.async copies land
__device__ __forceinline__ void cp_arrive(uint64_t* bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(su32(bar)) : "memory");
}

// Two 16-bit codes (lanes l, l+1) as floats times their chunk's scale, as Codec::dec
// does per value (the scale is a power of two: exact).
template <int kCodec>
__device__ __forceinline__ float2 dec2(uint32_t w, float2 s)
{
    float2 f;
    if constexpr (kCodec == 1) f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
    else f = __half22float2(*reinterpret_cast<const __half2*>(&w));
    return mul2(f, s);
}
// Two floats times 1/scale rounded to 16-bit codes, as Codec::enc does per value.
template <int kCodec>
__device__ __forceinline__ uint32_t enc2(float2 f, float2 inv)
{
    const float2 x = mul2(f, inv);
    uint32_t w;
    if constexpr (kCodec == 1) {
        const __nv_bfloat162 h = __float22bfloat162_rn(x);
        w = *reinterpret_cast<const uint32_t*>(&h);
    } else {
        const __half2 h = __float22half2_rn(x);
        w = *reinterpret_cast<const uint32_t*>(&h);
    }
    return w;
}

// A staging wait gives up after one second of device time or 2^24 polls (a batch is a
// few tens of kB staged in microseconds): reaching either means a fault upstream.
constexpr unsigned kPolls = 1u << 24;
constexpr uint64_t kWaitLimitNs = 1000000000ull;

__device__ __forceinline__ bool bar_wait_bounded(uint64_t* bar, unsigned parity)
{
    if (bar_try(bar, parity)) return true;
    unsigned polls = 0;
    const uint64_t t0 = now_ns();
    while (!bar_try(bar, parity)) {
        if (++polls > kPolls || ((polls & 63u) == 0 && now_ns() - t0 > kWaitLimitNs)) return false;
    }
    return true;
}

__device__ __forceinline__ float2 lds2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void sts2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }

// row-space contribution (row = y + ny*z) of coordinate c along physical axis d (1 or 2)
__device__ __forceinline__ int rowpart(int d, int c, int ny) { return d == 1 ? c : c * ny; }

// Named barriers: the staging warps, the sweeping warps.
constexpr int kBarStage = 1, kBarSweep = 2;
__device__ __forceinline__ void named_sync(int id, int n)
{
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}
// Item w of the list: chunk w % 4 of pair w / 4.
__device__ __forceinline__ void decode_item(const Gt3Args& P, int64_t w, Item& it)
{
    const GridGeom& G = P.G;
    const uint32_t pair = P.items[w >> 2];
    const int b = (int)(pair / P.ntiles);
    const uint32_t tile = pair - (uint32_t)b * P.ntiles;
    const int q = (int)(w & 3);
    it.b = b;
    it.q = q;
    it.tx0 = (int)(tile % P.ntile0) * kT;
    it.tr0 = (int)(tile / P.ntile0) * kT;
    it.ex = min(kT, G.n[0] - it.tx0);
    it.er = min(kT, G.n[P.ar] - it.tr0);
    it.dense_in = (P.in.dense[b] & 3) == 3;
    it.dense_out = (P.out.dense[b] & 1) != 0;
    it.ibase = ((int64_t)P.in.base[b] * 4 + (int64_t)q * P.in.cnt[b]) * kChunk;
    it.okeep = (int64_t)P.out.base[b];
    it.obase = (it.okeep * 4 + (int64_t)q * P.out.cnt[b]) * kChunk;
    // directions along the three sweep axes: the same for every velocity cell of the item
    // (the host checks that no block straddles v = 0)
    const int bc[3] = {b % G.nbx, (b / G.nbx) % G.nby, b / (G.nbx * G.nby)};
    int up[3];
    for (int j = 0; j < 3; j++) {
        const int d = P.ax[j];
        up[j] = P.walk[d * P.nvmax + bc[d] * 4 + (d == 2 ? q : 0)].w != 0.0f;
    }
    it.up0 = up[0];
    it.up1 = up[1];
    it.up2 = up[2];
}

// The tables of an item (the staging threads, sl = 0 .. kNS-1).
__device__ __forceinline__ void item_tables(const Gt3Args& P, const Item& it, ItemTables& t, int sl)
{
    const GridGeom& G = P.G;
    const int nx = G.n[0], nr = G.n[P.ar];
    for (int i = sl; i < 3 * kChunk + 2 * kE + 1; i += kNS) {
        if (i < 3 * kChunk) {
            // sweep constants of the item's 16 velocity cells (v = vx + 4 vy, vz = q)
            const int j = i >> 4, l = i & 15;
            const int d = P.ax[j];
            const int bc = d == 0 ? it.b % G.nbx : (d == 1 ? (it.b / G.nbx) % G.nby : it.b / (G.nbx * G.nby));
            const int wi = d == 0 ? (l & 3) : (d == 1 ? (l >> 2) : it.q);
            t.kc[j][l] = P.walk[d * P.nvmax + bc * 4 + wi];
        } else if (i < 3 * kChunk + kE) {
            const int u = i - 3 * kChunk;
            t.xs[u] = wrapi(it.tx0 - kHalo + u, nx);
        } else if (i < 3 * kChunk + 2 * kE) {
            const int u = i - 3 * kChunk - kE;
            t.rrow[u] = rowpart(P.ar, wrapi(it.tr0 - kHalo + u, nr), G.n[1]);
        } else {
            // a walk reads 3 cells upwind of the tile and 2 downwind of it, so one of the
            // outermost rows and columns is not needed
            const bool x_first = P.ax[0] == 0;
            t.r0 = (x_first ? it.up1 : it.up0) ? 0 : 1;
            t.u0 = (x_first ? it.up0 : it.up1) ? 0 : 1;
            int u0 = t.u0, nrun = 0;
            const int end = u0 + kLines;
            while (u0 < end) {
                const int x = wrapi(it.tx0 - kHalo + u0, nx);
                const int len = min(end - u0, nx - x);
                t.run[nrun][0] = u0;
                t.run[nrun][1] = x;
                t.run[nrun][2] = len;
                nrun++;
                u0 += len;
            }
            t.nrun = nrun;
        }
    }
}

// Staging of batch k of an item (planes kNB k .. kNB k + 2 of its stream) into buffer
// g & 1, g = the CTA's running batch index; run by the kNS staging threads (sl = 0..127),
// one staged row per thread, and every staging thread arrives on the batch's barrier
// once its copies have landed.  What staging threads write themselves (an item's description
// and tables, zeroed cells, output slots) is published by arrivals that release it: a
// cp.async arrival does not release its thread's own stores, so each staging warp adds one
// plain arrival, the last thing it does for a batch, after its lanes' stores (__syncwarp).
// Nothing that a sweeping warp reads is written after it.  Contiguous runs of a row go by TMA
// bulk copies; the short run where a dense row wraps around the periodic grid (kShortRun cells
// or fewer) goes by 16-byte cp.async copies instead: the SM's bulk-copy unit takes a roughly
// fixed time per request, and these runs would add half as many requests again.  The chunk
// scale of each staged cell goes into the scale table with a 4-byte cp.async copy (0 for an
// absent cell).  With sweep 0 along x the row's codes are packed
// at one end of the row (kCodesHi) by bulk copies per contiguous run: sweep 0 walks
// towards that end and writes its FP32 result two cells behind the one it reads, which
// overwrites only codes read at least three positions earlier.  Otherwise the 32 bytes of
// codes of each cell go to the upper half of its own 64-byte slot with two 16-byte
// cp.async copies, so that each line of sweep 0 overwrites only codes it has read.
constexpr int kShortRun = 4;

// cells of an item's staged row that go by bulk copies (runs longer than kShortRun)
__device__ __forceinline__ int bulk_cells(const ItemTables& t)
{
    int c = 0;
    for (int k2 = 0; k2 < t.nrun; k2++)
        if (t.run[k2][2] > kShortRun) c += t.run[k2][2];
    return c;
}

template <int kCodec, bool kA0X>
__device__ __forceinline__ void stage_batch(const Gt3Args& P, Gt3Smem& S, const Item& it,
                                            const ItemTables& t, int k, unsigned g, int sl)
{
    const GridGeom& G = P.G;
    const int nx = G.n[0], ny = G.n[1], a2 = P.ax[2], n2 = G.n[a2];
    const int nsteps = n2 + kFirst;
    const unsigned slot = g & 1u;
    uint64_t* bar = &S.bar[slot];
    const int nj = min(kNB, nsteps - kNB * k);
    const int nrun = t.nrun;
    // staged row (and output row) of this thread: rows go round-robin over the four
    // staging warps, whose lanes issue their copies one after another
    const int sw = (sl & 31) * (kNS / 32) + (sl >> 5);
    const float* ipool = static_cast<const float*>(P.in.pool);
    auto plane_of = [&](int s) { return it.up2 ? s - kHalo : n2 + 2 - s; };
    auto out_of = [&](int s) { return it.up2 ? s - kFirst : n2 + 4 - s; };
    // this thread's half of a tile row whose output slots it writes below
    const int oj = sw / (2 * kT), orr = (sw >> 1) - oj * kT;
    const bool slots = !it.dense_out && sw < nj * 2 * kT && kNB * k + oj >= kFirst;
    if constexpr (kCodec != 0) {
        using T = typename Codec<kCodec>::T;
        const T* cpool = static_cast<const T*>(P.in.pool) + it.ibase;  // codes of rank 0
        const float* spool = P.in.scale + it.ibase / kChunk;            // scale of rank 0
        if (sw < nj * kLines) {
            const int j = sw / kLines, rho = t.r0 + sw - j * kLines;
            const int pz = wrapi(plane_of(kNB * k + j), n2);
            const int64_t row = (int64_t)t.rrow[rho] + rowpart(a2, pz, ny);
            float* drow = &S.buf[slot][j][rho * kRP];
            float* srow = scales_of(S) + ((slot * kNB + j) * kE + rho) * kSP;
            if constexpr (kA0X) {
                float* codes = drow + (it.up0 ? kCodesHi : 0);
                fence_async_smem();
                if (it.dense_in) {
                    const int64_t r0 = row * nx;
                    for (int k2 = 0; k2 < nrun; k2++) {
                        const int u0 = t.run[k2][0], x0 = t.run[k2][1], len = t.run[k2][2];
                        float* d = codes + u0 * (kChunk / 2);
                        const T* src = cpool + (r0 + x0) * kChunk;
                        if (len > kShortRun) {
                            copy_g2s(d, src, (unsigned)(len * kChunk * sizeof(T)), bar);
                        } else {
                            for (int i = 0; i < len * 2; i++) cp16(d + 4 * i, src + 8 * i, 16);
                        }
                    }
                    for (int u = t.u0; u < t.u0 + kLines; u++) cp4(srow + u, spool + r0 + t.xs[u], 4);
                } else {
                    // runs of present cells (consecutive slots) as bulk copies, each announced
                    // to the barrier before it is issued; absent cells get zero codes and scale
                    const int64_t wbase = (int64_t)it.b * G.RW + row * G.W;
                    for (int k2 = 0; k2 < nrun; k2++) {
                        const int u0 = t.run[k2][0], x0 = t.run[k2][1], len = t.run[k2][2];
                        const int w0 = x0 >> 6, sh = x0 & 63;
                        const bool two = sh + len > 64;
                        const uint64_t ua = P.in.ubits[wbase + w0];
                        const uint64_t ub = two ? P.in.ubits[wbase + w0 + 1] : 0ull;
                        const uint32_t oa = P.in.woff[wbase + w0];
                        const uint32_t ob = two ? P.in.woff[wbase + w0 + 1] : 0u;
                        const uint64_t lenmask = (1ull << len) - 1ull;  // len <= 22
                        uint64_t pm = (P.in.kbits[wbase + w0] & ua) >> sh;
                        if (two) pm |= (P.in.kbits[wbase + w0 + 1] & ub) << (64 - sh);
                        pm &= lenmask;
                        uint64_t absent = ~pm & lenmask;
                        while (absent) {
                            const int u = u0 + __ffsll((long long)absent) - 1;
                            absent &= absent - 1ull;
                            cp16(codes + u * (kChunk / 2), cpool, 0);
                            cp16(codes + u * (kChunk / 2) + 4, cpool, 0);
                            cp4(srow + u, spool, 0);
                        }
                        uint64_t m = pm;
                        while (m) {
                            const int u = __ffsll((long long)m) - 1;
                            const int rl = __ffsll((long long)~(m >> u)) - 1;
                            const int x = x0 + u;
                            const bool lw = (x >> 6) == w0;
                            const int64_t r = (int64_t)(lw ? oa : ob) + __popcll((lw ? ua : ub) & ((1ull << (x & 63)) - 1ull));
                            const unsigned bytes = (unsigned)(rl * kChunk * sizeof(T));
                            bar_add_tx(bar, bytes);
                            copy_g2s(codes + (u0 + u) * (kChunk / 2), cpool + r * kChunk, bytes, bar);
                            for (int i = 0; i < rl; i++) cp4(srow + u0 + u + i, spool + r + i, 4);
                            m &= ~(((1ull << rl) - 1ull) << u);
                        }
                    }
                }
            } else {
                for (int u = t.u0; u < t.u0 + kLines; u++) {
                    const int x = t.xs[u];
                    int64_t r;
                    if (it.dense_in) {
                        r = row * nx + x;
                    } else {
                        const int64_t wi = (int64_t)it.b * G.RW + row * G.W + (x >> 6);
                        const uint64_t bit = 1ull << (x & 63);
                        const uint64_t uw = P.in.ubits[wi];
                        r = ((uw & P.in.kbits[wi] & bit) != 0ull) ? (int64_t)P.in.woff[wi] + __popcll(uw & (bit - 1ull))
                                                                   : -1;
                    }
                    float* dst = drow + u * kChunk + 8;
                    const T* src = r >= 0 ? cpool + r * kChunk : cpool;
                    const int nbytes = r >= 0 ? 16 : 0;
                    cp16(dst, src, nbytes);
                    cp16(dst + 4, src + 8, nbytes);
                    cp4(srow + u, r >= 0 ? spool + r : spool, r >= 0 ? 4 : 0);
                }
            }
        }
        // dense rows with sweep 0 along x: the batch's code bytes, announced without an
        // arrival (the phase also waits for every staging thread's arrival below)
        if (kA0X && it.dense_in && sl == 0)
            bar_add_tx(bar, (unsigned)(nj * kLines * bulk_cells(t) * kChunk * sizeof(T)));
    } else if (it.dense_in) {
        // the batch's bulk-copy bytes, announced once (the copies of the other staging
        // threads may complete before or after it; the phase also waits for every staging
        // thread's arrival)
        if (sl == 0) bar_add_tx(bar, (unsigned)(nj * kLines * bulk_cells(t) * kChunk * sizeof(float)));
        if (sw < nj * kLines) {
            const int j = sw / kLines, rho = t.r0 + sw - j * kLines;
            const int pz = wrapi(plane_of(kNB * k + j), n2);
            const int64_t row = (int64_t)t.rrow[rho] + rowpart(a2, pz, ny);
            const float* src = ipool + it.ibase + row * nx * kChunk;
            float* dst = &S.buf[slot][j][rho * kRP];
            fence_async_smem();
            for (int k2 = 0; k2 < nrun; k2++) {
                const int u0 = t.run[k2][0], x0 = t.run[k2][1], len = t.run[k2][2];
                if (len > kShortRun) {
                    copy_g2s(dst + u0 * kChunk, src + x0 * kChunk, (unsigned)(len * kChunk * sizeof(float)), bar);
                } else {
                    for (int i = 0; i < len * (kChunk / 4); i++)
                        cp16(dst + u0 * kChunk + 4 * i, src + x0 * kChunk + 4 * i, 16);
                }
            }
        }
    } else {
        // runs of present cells (consecutive slots) as bulk copies, each announced to the
        // barrier before it is issued; absent cells are zeroed
        if (sw < nj * kLines) {
            const int j = sw / kLines, rho = t.r0 + sw - j * kLines;
            const int pz = wrapi(plane_of(kNB * k + j), n2);
            const int64_t row = (int64_t)t.rrow[rho] + rowpart(a2, pz, ny);
            const int64_t wbase = (int64_t)it.b * G.RW + row * G.W;
            float* dst = &S.buf[slot][j][rho * kRP];
            fence_async_smem();
            for (int k2 = 0; k2 < nrun; k2++) {
                const int u0 = t.run[k2][0], x0 = t.run[k2][1], len = t.run[k2][2];
                const int w0 = x0 >> 6, sh = x0 & 63;
                const bool two = sh + len > 64;
                const uint64_t ua = P.in.ubits[wbase + w0];
                const uint64_t ub = two ? P.in.ubits[wbase + w0 + 1] : 0ull;
                const uint32_t oa = P.in.woff[wbase + w0];
                const uint32_t ob = two ? P.in.woff[wbase + w0 + 1] : 0u;
                const uint64_t lenmask = (1ull << len) - 1ull;  // len <= 22
                uint64_t pm = (P.in.kbits[wbase + w0] & ua) >> sh;
                if (two) pm |= (P.in.kbits[wbase + w0 + 1] & ub) << (64 - sh);
                pm &= lenmask;
                uint64_t absent = ~pm & lenmask;
                while (absent) {
                    const int u = __ffsll((long long)absent) - 1;
                    absent &= absent - 1ull;
                    float4* z = reinterpret_cast<float4*>(dst + (u0 + u) * kChunk);
                    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                    z[0] = zero;
                    z[1] = zero;
                    z[2] = zero;
                    z[3] = zero;
                }
                uint64_t m = pm;
                while (m) {
                    const int u = __ffsll((long long)m) - 1;
                    const int rl = __ffsll((long long)~(m >> u)) - 1;
                    const int x = x0 + u;
                    const bool lw = (x >> 6) == w0;
                    const int64_t r = (int64_t)(lw ? oa : ob) + __popcll((lw ? ua : ub) & ((1ull << (x & 63)) - 1ull));
                    const unsigned bytes = (unsigned)(rl * kChunk * sizeof(float));
                    bar_add_tx(bar, bytes);
                    copy_g2s(dst + (u0 + u) * kChunk, ipool + it.ibase + r * kChunk, bytes, bar);
                    m &= ~(((1ull << rl) - 1ull) << u);
                }
            }
        }
    }
    // every thread arrives after announcing its bytes, so the phase cannot end before every
    // announcement; deferred until its cp.async copies land where there may be any
    if (kCodec != 0 || it.dense_in) cp_arrive(bar);
    else bar_arrive(bar);
    // output slots of the tile cells of a sparse next layout, two threads per tile row.  (Read
    // before the copies are issued, with the thread's arrival after the stores, the bitmap
    // words cost registers on every state: 8.73 against 8.71 ms a sweep in bfloat16, 64x64x16
    // cells of the uniform workload, 15.99 against 15.97 on 128x32x16 of the shock.)
    if (slots) {
        uint64_t uw = 0ull;
        uint32_t ow = 0u;
        if (orr < it.er) {
            const int64_t row = (int64_t)rowpart(P.ar, it.tr0 + orr, ny) + rowpart(a2, out_of(kNB * k + oj), ny);
            const int64_t wi = (int64_t)it.b * G.RW + row * G.W + (it.tx0 >> 6);
            uw = P.out.ubits[wi];
            ow = P.out.woff[wi];
        }
        if (P.testing & kTestSlots) __nanosleep(kTestSlotsNs);
        int* orow = &S.orank[slot][oj][orr * kT];
#pragma unroll
        for (int i8 = 0; i8 < kT / 2; i8++) {
            const int i = (sw & 1) * (kT / 2) + i8;
            const int bit = (it.tx0 + i) & 63;  // the 16 cells share one bitmap word
            const bool has = i < it.ex && ((uw >> bit) & 1ull);
            orow[i] = has ? (int)(ow + __popcll(uw & ((1ull << bit) - 1ull))) : -1;
        }
    }
    // publishes what the warp's lanes have written, the slots above among them
    __syncwarp();
    if ((sl & 31) == 0) bar_arrive(bar);
}

// The staging warps: they run up to two batches ahead of the sweeping warps, across
// items.  The index of the next item is taken one item ahead.
template <bool kA0X, int kCodec>
__device__ __forceinline__ void stage_loop(const Gt3Args& P, Gt3Smem& S, int sl, int nbatch, int64_t nwork)
{
    long long wnext = 0;
    if (sl == 0) wnext = (long long)atomicAdd(&P.ctr->work_next, 1ull);
    // Buffer g & 1 is free once batch g - 2 is swept; the sweeping warps have then also left
    // the item before the one of that batch, whose description and tables are overwritten.
    // One thread waits, and the others learn of it at the staging warps' barrier.
    auto wait_empty = [&](unsigned g) {
        if (g >= 2 && sl == 0 && !bar_wait_bounded(&S.empty[g & 1u], ((g >> 1) - 1u) & 1u)) S.late = 1;
    };
    unsigned g = 0;
    bool late = false;
    for (int par = 0; !late; par ^= 1) {
        wait_empty(g);
        if (sl == 0) {
            S.work[par] = wnext;
            if (wnext < nwork && !S.late) {
                decode_item(P, wnext, S.item[par]);
                wnext = (long long)atomicAdd(&P.ctr->work_next, 1ull);
            }
        }
        named_sync(kBarStage, kNS);
        late = S.late != 0;
        if (late) break;
        if (S.work[par] >= nwork) {
            // nothing more to stage: the phase completes and tells the sweeping warps to end
            bar_arrive(&S.bar[g & 1u]);
            if ((sl & 31) == 0) bar_arrive(&S.bar[g & 1u]);
            return;
        }
        const Item& it = S.item[par];
        item_tables(P, it, S.tab[par], sl);
        for (int k = 0; k < nbatch; k++, g++) {
            if (k > 0) wait_empty(g);
            named_sync(kBarStage, kNS);
            late = S.late != 0;
            if (late) break;
            stage_batch<kCodec, kA0X>(P, S, it, S.tab[par], k, g, sl);
        }
    }
    // the sweeping warps stopped: leave no copy in flight (the last two batches staged)
    if (sl == 0) atomicOr(&P.ctr->error, 4);
    for (unsigned i = 1; i <= 2 && i <= g; i++) bar_wait_bounded(&S.bar[(g - i) & 1u], ((g - i) >> 1) & 1u);
}

template <bool kLim, bool kA0X, int kCodec>
__global__ void __launch_bounds__(kNT, 1) k_gt3(Gt3Args P)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    Gt3Smem& S = *reinterpret_cast<Gt3Smem*>(smraw);
    const GridGeom& G = P.G;
    if (aborted(G.abort)) return;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int ar = P.ar, a2 = P.ax[2];
    const int n2 = G.n[a2];
    const int nsteps = n2 + kFirst;       // planes streamed per item (3 before, 2 after)
    const int nbatch = (nsteps + kNB - 1) / kNB;  // at least 2
    const int64_t nwork = 4 * *P.npairs;
    const int str_r = (int)P.stride[ar], str_2 = (int)P.stride[a2];
    const unsigned zrow8 = 8u * (unsigned)str_r;
    // staged offsets of a position along sweep axis 0 / 1 (in floats)
    constexpr int kS0 = kA0X ? kChunk : kRP;
    constexpr int kS1 = kA0X ? kRP : kChunk;
    // the same for the scale table (one float per staged cell)
    constexpr int kC0 = kA0X ? 1 : kSP;
    constexpr int kC1 = kA0X ? kSP : 1;

    if (tid == 0) {
        for (int i = 0; i < 2; i++) {
            bar_init(&S.bar[i], kNS + kNS / 32);  // every staging thread, and each staging warp
            bar_init(&S.empty[i], kNC / 32);      // every sweeping warp
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        S.abort = S.late = 0;
        S.work[0] = S.work[1] = 0;
    }
    __syncthreads();
    if (tid >= kNC) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kRegsStage));
        stage_loop<kA0X, kCodec>(P, S, tid - kNC, nbatch, nwork);
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kRegsSweep));
    unsigned gb = 0;                    // batches before the current item (barrier phases)
    float msum = 0.0f, mcomp = 0.0f;    // Kahan-compensated FP32 mass of this thread
    bool stop = false;

    // a staged batch, or the end of the work list
    auto wait_staged = [&](unsigned g) {
        const unsigned slot = g & 1u, parity = (g >> 1) & 1u;
        if ((P.testing & kTestLate) && tid == 0 && !bar_test(&S.bar[slot], parity)) atomicOr(&P.ctr->error, 4);
        if (!bar_wait_bounded(&S.bar[slot], parity)) {
            atomicOr(&P.ctr->error, 4);
            S.abort = 1;
        }
    };
    for (int par = 0; !stop; par ^= 1) {
        wait_staged(gb);
        named_sync(kBarSweep, kNC);
        if (S.abort || S.work[par] >= nwork) break;
        const Item& it = S.item[par];
        const ItemTables& tab = S.tab[par];
        using T = typename Codec<kCodec>::T;
        const bool up0 = it.up0 != 0, up1 = it.up1 != 0, up2 = it.up2 != 0;
        const bool dense_out = it.dense_out != 0;
        // ---- sweep-2 state of this thread: two tile cells, one vx row of the chunk ----
        const int zq = tid & 3;             // vy of the thread's vx row
        const int zcx = (tid >> 2) & 15, zcr = tid >> 6;  // tile cells (zcx, zcr) and (zcx, zcr + 8)
        const bool zv0 = zcx < it.ex && zcr < it.er, zv1 = zcx < it.ex && zcr + 8 < it.er;
        const int zoff = (kHalo + zcr) * kRP + (kHalo + zcx) * kChunk + 4 * zq;
        // dense next layout: the slot of the first cell in the plane that is emitted next
        // (slots of one block id are below 2^31 like the cells)
        unsigned zslot = (unsigned)(it.tx0 + zcx + (it.tr0 + zcr) * str_r + (up2 ? 0 : (n2 - 1) * str_2));
        const unsigned zstep = up2 ? str_2 : -str_2;
        T* const zpool = static_cast<T*>(P.out.pool) + it.obase + 4 * zq;
        uint8_t* const kq = P.keepq + it.okeep * 4 + it.q;
        float* const zscale = kCodec ? P.out.scale + it.obase / kChunk : nullptr;
        // the four threads of a cell vote on its keep flag, which the first of them writes
        // (nobody when none are wanted)
        const unsigned vote = P.keepq && zq == 0 ? 0xfu << (lane & ~3) : 0u;
        const float thr = P.thr;
        Walk2<kLim, 1> zw[4];
#pragma unroll
        for (int i = 0; i < 4; i++) zw[i].reset();
        const WalkConst2 kz = pack_const(tab.kc[2][4 * zq], tab.kc[2][4 * zq]);  // the streamed axis is not x: equal over vx

        for (int k = 0; k < nbatch; k++) {
            const unsigned g = gb + (unsigned)k;
            const unsigned slot = g & 1u;
            if (k > 0) wait_staged(g);
            float* B = S.buf[slot][0];
            const int nj = min(kNB, nsteps - kNB * k);
            // sweep 0 along axis 0 on the halo lines that sweep 1 reads
            if (tid < kNX) {
                const int j = tid / (kLines * 8), rem = tid - j * (kLines * 8);
                const int line = rem >> 3, l0 = 2 * (rem & 7);
                if (j < nj) {
                    const WalkConst2 kx = pack_const(tab.kc[0][l0], tab.kc[0][l0 + 1]);
                    float* p = B + j * kPS + (line + (up1 ? 0 : 1)) * kS1 + l0;
                    // 16-bit storage: chunk scales of the line's cells
                    const float* ps = scales_of(S) + (slot * kNB + j) * kE * kSP + (line + (up1 ? 0 : 1)) * kC1;
                    // the two staged values of position m: FP32, or two 16-bit codes in the
                    // upper half of the cell's slot
                    // packed codes of the line (sweep 0 along x), see stage_batch
                    const uint32_t* pc = reinterpret_cast<const uint32_t*>(
                                             B + j * kPS + (line + (up1 ? 0 : 1)) * kRP + (up0 ? kCodesHi : 0)) +
                                         (l0 >> 1);
                    auto in = [&](int m) -> float2 {
                        if constexpr (kCodec == 0) {
                            return lds2(p + m * kS0);
                        } else {
                            const float sc = ps[m * kC0];
                            const uint32_t w = kA0X ? pc[m * (kChunk / 2)]
                                                    : reinterpret_cast<const uint32_t*>(p - l0 + m * kS0)[8 + (l0 >> 1)];
                            return dec2<kCodec>(w, make_float2(sc, sc));
                        }
                    };
                    Walk2<kLim, 1> wk;
                    wk.reset();
                    if (up0) {
#pragma unroll
                        for (int m = 0; m < kLines; m++) {
                            const float2 r = wk.push(in(m), kx);
                            if (m >= 5) sts2(p + (m - 2) * kS0, r);
                        }
                    } else {
#pragma unroll
                        for (int m = 0; m < kLines; m++) {
                            const float2 r = wk.push(in(kLines - m), kx);
                            if (m >= 5) sts2(p + (kLines + 2 - m) * kS0, r);
                        }
                    }
                }
            }
            named_sync(kBarSweep, kNC);  // sweep 0 complete
            if (S.abort) {
                stop = true;
                break;
            }
            if (tid < kNY) {
                // sweep 1 along axis 1 on the tile lines
                const int j = tid >> 7, rem = tid & 127;
                const int line = rem >> 3, l0 = 2 * (rem & 7);
                if (j < nj) {
                    const WalkConst2 ky = pack_const(tab.kc[1][l0], tab.kc[1][l0 + 1]);
                    float* p = B + j * kPS + (kHalo + line) * kS0 + l0;
                    Walk2<kLim, 1> wk;
                    wk.reset();
                    if (up1) {
#pragma unroll
                        for (int m = 0; m < kLines; m++) {
                            const float2 r = wk.push(lds2(p + m * kS1), ky);
                            if (m >= 5) sts2(p + (m - 2) * kS1, r);
                        }
                    } else {
#pragma unroll
                        for (int m = 0; m < kLines; m++) {
                            const float2 r = wk.push(lds2(p + (kLines - m) * kS1), ky);
                            if (m >= 5) sts2(p + (kLines + 2 - m) * kS1, r);
                        }
                    }
                }
            }
            // the in-place writes of this batch precede the bulk copies that refill the
            // buffer two batches on
            fence_async_smem();
            named_sync(kBarSweep, kNC);  // sweep 1 complete
            // sweep 2: push the batch's planes through the streamed windows and emit
            auto zplane = [&](int j) {
                const int s = kNB * k + j;
                const float* src = B + j * kPS + zoff;
                const float4 y0 = *reinterpret_cast<const float4*>(src);
                const float4 y1 = *reinterpret_cast<const float4*>(src + 8 * kRP);
                float2 v[4];
                v[0] = zw[0].push(make_float2(y0.x, y0.y), kz);
                v[1] = zw[1].push(make_float2(y0.z, y0.w), kz);
                v[2] = zw[2].push(make_float2(y1.x, y1.y), kz);
                v[3] = zw[3].push(make_float2(y1.z, y1.w), kz);
                if (s < kFirst) return;
                // slots of the two cells (-1: none): in a dense next layout the cell index
                int r0 = -1, r1 = -1;
                if (dense_out) {
                    r0 = zv0 ? (int)zslot : -1;
                    r1 = zv1 ? (int)(zslot + zrow8) : -1;
                    zslot += zstep;
                } else {
                    const int* orow = &S.orank[slot][j][zcr * kT + zcx];
                    r0 = zv0 ? orow[0] : -1;
                    r1 = zv1 ? orow[8 * kT] : -1;
                }
                float psum = 0.0f;
                // 16-bit storage: the scales of the two cells' chunks, from the largest magnitude
                // over the four threads (vx rows) of a cell
                ChunkScale cs0{1.0f, 1.0f}, cs1{1.0f, 1.0f};
                if constexpr (kCodec != 0) {
                    auto top = [](const float2& p, const float2& q) {
                        return fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fmaxf(fabsf(q.x), fabsf(q.y)));
                    };
                    cs0 = chunk_scale(group_max<4>(top(v[0], v[1])));
                    cs1 = chunk_scale(group_max<4>(top(v[2], v[3])));
                }
                // one vx row (4 values) of a cell; the values summed and compared are those that
                // the state now holds (16-bit storage: the codes decoded).  No branches: the
                // stores are predicated
                auto emit = [&](int r, float2 v0, float2 v1, const ChunkScale& cs) -> bool {
                    const bool has = r >= 0;
                    T* dst = zpool + (int64_t)r * kChunk;
                    if constexpr (kCodec == 0) {
                        if (has) *reinterpret_cast<float4*>(dst) = make_float4(v0.x, v0.y, v1.x, v1.y);
                    } else {
                        const float2 inv = make_float2(cs.inv, cs.inv), sc = make_float2(cs.s, cs.s);
                        const uint32_t w0 = enc2<kCodec>(v0, inv), w1 = enc2<kCodec>(v1, inv);
                        if (has) *reinterpret_cast<uint2*>(dst) = make_uint2(w0, w1);
                        if (has && zq == 0) zscale[r] = cs.s;
                        v0 = dec2<kCodec>(w0, sc);
                        v1 = dec2<kCodec>(w1, sc);
                    }
                    psum += has ? (v0.x + v0.y) + (v1.x + v1.y) : 0.0f;
                    return has && fmaxf(fmaxf(v0.x, v0.y), fmaxf(v1.x, v1.y)) >= thr;
                };
                const bool keep0 = emit(r0, v[0], v[1], cs0), keep1 = emit(r1, v[2], v[3], cs1);
                // per-chunk keep flags: the four threads of a cell vote
                const unsigned b0 = __ballot_sync(0xffffffffu, keep0), b1 = __ballot_sync(0xffffffffu, keep1);
                if (b0 & vote) kq[(int64_t)r0 * 4] = 1;
                if (b1 & vote) kq[(int64_t)r1 * 4] = 1;
                const float y = psum - mcomp;
                const float t = msum + y;
                mcomp = (t - msum) - y;
                msum = t;
            };
            if (nj == kNB) {
#pragma unroll
                for (int j = 0; j < kNB; j++) zplane(j);
            } else {
                for (int j = 0; j < nj; j++) zplane(j);
            }
            // this warp has read the buffer
            __syncwarp();
            if (lane == 0) bar_arrive(&S.empty[slot]);
        }
        gb += (unsigned)nbatch;
    }
    // the sum runs over all items of the CTA: its low part goes with it
    double m = (double)msum - (double)mcomp;
    for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
    if (lane == 0 && m != 0.0) atomicAdd(&P.ctr->mass, m);
    if (P.cta_done && tid == 0) P.cta_done[blockIdx.x] = now_ns();
}

template <bool kLim, bool kA0X, int kCodec>
vl_status launch_gt3(Grid* g, const Gt3Args& P)
{
    auto kern = k_gt3<kLim, kA0X, kCodec>;
    // setmaxnreg draws on the registers of the launch: never start a kernel whose share
    // is smaller than the split
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || fa.numRegs * kNT < kNC * kRegsSweep + kNS * kRegsStage)
        return fail(g, VL_ECUDA, "plane-batched fused sweep: register count of the kernel");
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<kCodec>());
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, g->dev.device);
    Gt3Args Q = P;
    if (nsm > kMaxCtas) Q.cta_done = nullptr;
    g->cta_count = Q.cta_done ? nsm : 0;
    g->cta_groups = 1;
    kern<<<nsm, kNT, smem_bytes<kCodec>(), g->stream>>>(Q);
    note_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(g, e, "plane-batched fused sweep launch");
    return VL_OK;
}

}  // namespace

bool gt3_fits(const vl_vmesh_desc& vmesh, const double c_scale[3], const int order[3])
{
    if (order[2] == 0) return false;  // streamed axis must not be x
    // every velocity block moves one way along each axis
    for (int d = 0; d < 3; d++)
        for (int bi = 0; bi < vmesh.nv[d] / 4; bi++) {
            const double lo = vmesh.vmin[d] + (4 * bi + 0.5) * vmesh.dv[d];
            const double hi = vmesh.vmin[d] + (4 * bi + 3.5) * vmesh.dv[d];
            if ((lo * c_scale[d] >= 0.0) != (hi * c_scale[d] >= 0.0)) return false;
        }
    return true;
}

bool gt3_applies(const Grid* g, const StepArgs& a)
{
    return a.ghost == 3 && gt3_fits(g->vmesh, a.c_scale, a.order);
}

int64_t gt3_tiles(const GridGeom& G, const int order[3])
{
    const int ar = order[0] == 0 ? order[1] : order[0];
    return (int64_t)((G.n[0] + kT - 1) / kT) * ((G.n[ar] + kT - 1) / kT);
}

// One launch over caller-provided buffers of a dense FP32 layout: items are all nb * tiles
// pairs in order, npairs their number, no keep flags (the caller's threshold is +inf).
vl_status launch_gt3_dense(const GridGeom& G, const LayoutView& in, const LayoutView& out, const int order[3],
                           int limiter, const float4* ctab, int nvmax, const uint32_t* items,
                           const int64_t* npairs, StepCounters* ctr, int device, cudaStream_t stream)
{
    Gt3Args P;
    P.G = G;
    P.in = in;
    P.out = out;
    for (int j = 0; j < 3; j++) P.ax[j] = order[j];
    P.ar = order[0] == 0 ? order[1] : order[0];
    P.stride[0] = 1;
    P.stride[1] = G.n[0];
    P.stride[2] = (int64_t)G.n[0] * G.n[1];
    P.walk = ctab;
    P.nvmax = nvmax;
    P.thr = INFINITY;
    P.ntile0 = (G.n[0] + kT - 1) / kT;
    P.ntiles = (uint32_t)gt3_tiles(G, order);
    P.items = items;
    P.npairs = npairs;
    P.keepq = nullptr;
    P.ctr = ctr;
    P.testing = 0;
    P.cta_done = nullptr;
    Grid tmp;  // launch helper needs the device and the stream only
    tmp.dev.device = device;
    tmp.stream = stream;
    if (order[0] == 0) return limiter ? launch_gt3<true, true, 0>(&tmp, P) : launch_gt3<false, true, 0>(&tmp, P);
    return limiter ? launch_gt3<true, false, 0>(&tmp, P) : launch_gt3<false, false, 0>(&tmp, P);
}

vl_status run_gt3(Grid* g, const StepArgs& a)
{
    const GridGeom& G = g->geom;
    Layout& A = g->lay[g->cur];
    Layout& B = g->lay[1 - g->cur];
    const int ar = a.order[0] == 0 ? a.order[1] : a.order[0];
    const int ntile0 = (G.n[0] + kT - 1) / kT;
    const int ntile1 = (G.n[ar] + kT - 1) / kT;
    const int64_t ntiles = (int64_t)ntile0 * ntile1;
    if (ntiles > 0xffffffffLL) return fail(g, VL_EINVAL, "fused form: too many tiles");
    const int64_t need = ntiles * G.nb;
    vl_status wst = fused_worklist_alloc(g, a);
    if (wst != VL_OK) return wst;
    if (need > g->ntiles_alloc) return fail(g, VL_EINVAL, "fused form: work list too small");
    TileArgs T;
    T.G = G;
    T.ubits = B.ubits;
    T.ax[0] = 0;
    T.ax[1] = ar;
    T.ax[2] = a.order[2];
    T.ntile0 = ntile0;
    T.ntile1 = ntile1;
    T.ty = kT;
    launch_tile_list(g, T, need, ntiles, true);

    Gt3Args P;
    P.G = G;
    P.in = A.view();
    P.out = B.view();
    for (int j = 0; j < 3; j++) P.ax[j] = a.order[j];
    P.ar = ar;
    P.stride[0] = 1;
    P.stride[1] = G.n[0];
    P.stride[2] = (int64_t)G.n[0] * G.n[1];
    P.walk = a.walk;
    P.nvmax = a.nvmax;
    P.thr = (float)g->threshold;
    P.ntile0 = ntile0;
    P.ntiles = (uint32_t)ntiles;
    P.items = g->items;
    P.npairs = g->item_base + G.nb;
    P.keepq = B.keepq;
    P.ctr = a.ctr;
    P.testing = (fault_requested("timeout") ? kTestLate : 0) | (fault_requested("slow_slots") ? kTestSlots : 0);
    P.cta_done = a.stamp_ctas ? g->cta_done : nullptr;
    record_sweep_event(a.ev0, g->stream, a.ev_node);
    const bool a0x = a.order[0] == 0;
    vl_status st = VL_OK;
    with_codec(g->codec, [&](auto c) {
        constexpr int kc = decltype(c)::value;
        if (a0x) st = a.limiter ? launch_gt3<true, true, kc>(g, P) : launch_gt3<false, true, kc>(g, P);
        else st = a.limiter ? launch_gt3<true, false, kc>(g, P) : launch_gt3<false, false, kc>(g, P);
    });
    record_sweep_event(a.ev1, g->stream, a.ev_node);
    return st;
}

}  // namespace vlgt
