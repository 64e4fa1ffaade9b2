// Tiled semi-Lagrangian gather for sm_103a.
//
// A CTA owns a TILE1 x TILE2 x TILE3 block of arrival points (x3 fastest; a
// warp covers 32 consecutive x3 nodes of one x2 row, each thread TILE1
// points along x1).  Because the velocity is smooth, the departure points of
// a tile fall in a small box of the grid.  The CTA reduces the box bounds of
// its stencils, copies the box (periodically wrapped) from global memory into
// shared memory with cp.async, and then evaluates every stencil from shared
// memory, so the 64 (cubic) or 8 (linear) reads per point hit on-chip memory
// instead of issuing scattered L1/L2 requests.  A tile whose box does not fit
// (very large local compression of the characteristic map) falls back to the
// direct global-memory gather for that tile only.  The result of each point
// goes to an epilogue functor that fuses the step's source terms.
#pragma once

#include <climits>

#include "common.cuh"

namespace claire {

#ifndef CLAIRE_TILE1
#define CLAIRE_TILE1 4  // arrival points per thread along x1
#endif
#ifndef CLAIRE_TILE_MIN_BLOCKS
#define CLAIRE_TILE_MIN_BLOCKS 4  // resident CTAs per SM the register budget targets
#endif

#ifndef CLAIRE_FFMA2
#define CLAIRE_FFMA2 1  // packed FP32x2 FMA (sm_100+) for the separable stencil contraction
#endif
#ifndef CLAIRE_LDS_ASM
#define CLAIRE_LDS_ASM 1  // explicit 32-bit ld.shared with immediate offsets for the stencil reads
#endif
#ifndef CLAIRE_BOX_CAP
#define CLAIRE_BOX_CAP 11776  // floats of dynamic shared memory per CTA (46 KB)
#endif

#ifndef CLAIRE_TILE2
#define CLAIRE_TILE2 8  // x2 rows per tile: one warp each
#endif

constexpr int TILE1 = CLAIRE_TILE1, TILE2 = CLAIRE_TILE2, TILE3 = 32;

// CTAs of the tiled gathers (in this translation unit) whose box did not fit
// and which took the global-memory path; one atomic per such CTA, read by
// claire_gather_fallback_tiles.
static __device__ unsigned long long g_gather_global_tiles = 0;
constexpr int kTileThreads = TILE2 * 32;
constexpr int kBoxCapFloats = CLAIRE_BOX_CAP;

// Trilinear FP32 tiles: a point reads 8 values, so a tile is mostly the latency of
// its staging, and six CTAs per SM with boxes of 36 KB (a stencil two nodes wide
// needs half the box) hide it better than four of 46 KB: 256 x 300 x 256
// transport of eight steps 1277 -> 1130 us (five: 1205, seven: 1122 but 5 %
// slower adjoint steps).  16-bit fields, whose boxes also hold the staging copy,
// lose 2 % with six and keep four.
// The narrow box holds tiles whose cells spread over 5 nodes, the wide one 6, and a
// tile that fits neither costs most where six CTAs leave the L1 28 KB.  So large
// displacements (Grid::wide, set by the context where |v| dt is more than kWideCfl
// cells somewhere) take the wide box and kernels compiled for its four CTAs.
// Four steps at 512^3, modes up to 24, share of tiles that overflow and time,
// narrow / wide: CFL 12: 13 % 5.3 ms / 1.4 % 5.2; CFL 16: 42 % 7.6 / 14 % 5.9;
// CFL 24: 74 % 15.2 / 54 % 7.4; CFL 41: 91 % 29.4 / 83 % 9.5.  Modes up to 6,
// CFL 12: 0.3 % 4.6 / 0 4.9; CFL 24: 19 % 5.7 / 7 % 5.4.  320^3, up to 24, CFL 10:
// 16 % 1.44 narrow; CFL 13: 46 % 2.15 / 11 % 1.49; CFL 15: 69 % 3.3 / 32 % 1.7.
// Half boxes of 16 columns for the tiles that overflow: 1.3 to 1.9 times the wide
// box's time.
constexpr int kBoxCapLinear = 9216;
template <int ORDER, int ES = 4>
__host__ __device__ __forceinline__ int box_cap(const Grid& g)
{
    return ORDER == 1 && ES == 4 && !g.wide ? kBoxCapLinear : kBoxCapFloats;
}
// WIDE: the kernel launched with the wide box, compiled for its four CTAs per SM (with
// the registers of six, 512^3 interpolation at no displacement took 0.88 ms
// instead of 0.75 behind the wide box).
template <int ORDER, int ES = 4, bool WIDE = false>
constexpr int tile_min_blocks()
{
    return ORDER == 1 && ES == 4 && !WIDE ? 6 : CLAIRE_TILE_MIN_BLOCKS;
}

__device__ __forceinline__ void cp_async_f32(float* smem_dst, const float* gmem_src)
{
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem_src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

template <int ORDER>
__device__ __forceinline__ void axis_weights(float t, float w[4])
{
    scheme_weights<ORDER>(t, w);
}

// Direct global-memory gather for tiles whose departure box does not fit
// (kept out of line so that it does not add to the register budget of the
// shared-memory path).
// Trilinear: the operations of tile_eval in its order, so that a value does not
// depend on whether the tile's box fits (Grid::wide chooses the box by speed alone).
template <int ORDER, class S>
__device__ __noinline__ float gather_global(const Grid g, const S* __restrict__ f, int i, int j,
                                            int k, float d1, float d2, float d3)
{
    Stencil<ORDER> s;
    s.build(g, i, j, k, d1, d2, d3);
    if constexpr (ORDER == 1) {
        float val = 0.0f;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            float acc[2];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const S* row = f + s.a1.idx[a] + s.a2.idx[b];
                acc[b] = __fmul_rn(__fmul_rn(s.a2.w[b], s.a3.w[0]), ldf<S>(row + s.a3.idx[0]));
                acc[b] = __fmaf_rn(__fmul_rn(s.a2.w[b], s.a3.w[1]), ldf<S>(row + s.a3.idx[1]), acc[b]);
            }
            val = fmaf(s.a1.w[a], __fadd_rn(acc[0], acc[1]), val);
        }
        return val;
    } else {
        return s.template eval<S>(f);
    }
}

// ---- building blocks of the tiled gathers ----

// Geometry of the CTA's stencil box, shared by all threads of the CTA.
struct BoxPar {
    int O1, O2, O3;  // first node (unwrapped grid coordinates)
    int E1, E2, E3;  // extents; E1 == 0 means "does not fit: gather from global memory"
    int S3;          // row stride, a multiple of 32
};

// The grid whose extents bound the box: an axis too short for a tile's usual
// box (32 columns, 8 rows or 4 planes, the stencil and some spread) counts
// double, since a field of period n also has period 2 n; the staging wraps
// such indices twice.  Without this every tile of a grid with n3 < 40 or so
// took the global-memory path (32^3 backtrace: 26 us against 13 us).
__host__ __device__ __forceinline__ Grid box_grid(Grid g)
{
    g.n1 = g.n1 < 16 ? 2 * g.n1 : g.n1;
    g.n2 = g.n2 < 24 ? 2 * g.n2 : g.n2;
    g.n3 = g.n3 < 64 ? 2 * g.n3 : g.n3;
    return g;
}

// Wrapped index of w + c for w in [0, n) and an offset c < 2 n inside a box.
__device__ __forceinline__ int box_wrap(int x, int n)
{
    x = x >= n ? x - n : x;
    return x >= n ? x - n : x;
}

// Box geometry from the bounds [a, z] (per axis) of the first-node cells
// (before the -OFF shift) of a tile's stencils: par[0..2] the first node
// (unwrapped grid coordinates), par[3..5] the extents and par[6] the row
// stride, with par[3..6] = 0 when the box does not fit the shared-memory cap
// or the grid, when the bounds are not ordered (z < a), or when `bad` says
// that a displacement of the tile failed disp_ok (non-finite or at least 2^20
// cells).  Such a tile is gathered from global memory with the clamped split,
// whose indices always wrap into range.
// The x3 origin and extent are rounded to the widest chunk the row length
// allows (16, 8 or 4 bytes), so that no chunk straddles the x3 wrap.
// ES: bytes per stored value of the field (4, or 2 for FP16 / BF16 storage,
// whose box is staged as raw 16-bit pairs before widening to FP32).
// Unsigned 32-bit arithmetic (every thread of a tile with a tile-bounds table
// runs this): spans are compared before anything is added to them.
template <int ORDER, int ES = 4>
__host__ __device__ __forceinline__ void box_geometry(const Grid& g, int a1, int a2, int a3, int z1, int z2, int z3,
                                                      bool bad, int par[7])
{
    constexpr unsigned M = Scheme<ORDER>::M;
    constexpr unsigned OFF = Scheme<ORDER>::OFF;
    constexpr unsigned WIDE = 16 / ES;  // values per 16-byte chunk
    const unsigned d1 = static_cast<unsigned>(z1) - static_cast<unsigned>(a1),
                   d2 = static_cast<unsigned>(z2) - static_cast<unsigned>(a2),
                   d3 = static_cast<unsigned>(z3) - static_cast<unsigned>(a3);
    const unsigned n1 = g.n1, n2 = g.n2, n3 = g.n3;
    // box of the stencils: cells [a - OFF, z - OFF + M); the tile always
    // holds at least one valid point
    bool fits = !bad && z1 >= a1 && z2 >= a2 && z3 >= a3 && d1 <= n1 - M && d2 <= n2 - M && d3 <= n3 - M;
    const unsigned e1 = d1 + M, e2 = d2 + M;
    unsigned o3 = static_cast<unsigned>(a3) - OFF, e3 = d3 + M;
    unsigned align = WIDE;
    while (align > 1 && (n3 & (align - 1))) align /= 2;
    const unsigned r = o3 & (align - 1);
    o3 -= r;
    e3 = (e3 + r + align - 1) & ~(align - 1);
    const unsigned s3 = (e3 + 31) & ~31u;  // bank-aligned row stride
    // FP32 box plus, for 16-bit storage, the staging copy (half its size)
    fits = fits && e3 <= n3 &&
           static_cast<unsigned long long>(e1 * e2) * s3 * (ES == 2 ? 3 : 2) <= 2ull * box_cap<ORDER, ES>(g);
    par[0] = fits ? static_cast<int>(static_cast<unsigned>(a1) - OFF) : 0;
    par[1] = fits ? static_cast<int>(static_cast<unsigned>(a2) - OFF) : 0;
    par[2] = fits ? static_cast<int>(o3) : 0;
    par[3] = fits ? static_cast<int>(e1) : 0;
    par[4] = fits ? static_cast<int>(e2) : 0;
    par[5] = fits ? static_cast<int>(e3) : 0;
    par[6] = fits ? static_cast<int>(s3) : 0;
}

// Fold one point's displacement (grid units) along an axis into the tile's
// bounds of first-node cells; `bad` records a displacement that fails disp_ok.
__host__ __device__ __forceinline__ void bounds_add(int node, float d, int& lo, int& hi, bool& bad)
{
#ifdef __CUDA_ARCH__
    // one floor conversion: for |d| < 2^20 it equals the clamped split; any
    // other value marks the tile bad, whose bounds are then not used
    const int b = node + __float2int_rd(d);
#else
    float t;
    const int b = node + split_disp(d, t);
#endif
    lo = lo < b ? lo : b;
    hi = hi > b ? hi : b;
    bad = bad || !disp_ok(d);
}

#ifdef __CUDACC__
// Block-wide bounds of the first-node cells [lo, hi] per axis and the vote on
// `bad` (any thread).  Thread 0 gets the tile's bounds in b = (a1, a2, a3, z1,
// z2, z3); every thread gets the vote.
__device__ __forceinline__ bool tile_bounds(int lo1, int lo2, int lo3, int hi1, int hi2, int hi3, bool bad,
                                            int (*red)[TILE2], int lane, int warp, int b[6])
{
    lo1 = __reduce_min_sync(0xffffffffu, lo1);
    lo2 = __reduce_min_sync(0xffffffffu, lo2);
    lo3 = __reduce_min_sync(0xffffffffu, lo3);
    hi1 = __reduce_max_sync(0xffffffffu, hi1);
    hi2 = __reduce_max_sync(0xffffffffu, hi2);
    hi3 = __reduce_max_sync(0xffffffffu, hi3);
    if (lane == 0) {
        red[0][warp] = lo1; red[1][warp] = lo2; red[2][warp] = lo3;
        red[3][warp] = hi1; red[4][warp] = hi2; red[5][warp] = hi3;
    }
    const bool any_bad = __syncthreads_or(bad) != 0;
    if (threadIdx.x == 0) {
        b[0] = b[1] = b[2] = INT_MAX;
        b[3] = b[4] = b[5] = INT_MIN;
#pragma unroll
        for (int w = 0; w < TILE2; ++w) {
            b[0] = min(b[0], red[0][w]); b[1] = min(b[1], red[1][w]); b[2] = min(b[2], red[2][w]);
            b[3] = max(b[3], red[3][w]); b[4] = max(b[4], red[4][w]); b[5] = max(b[5], red[5][w]);
        }
    }
    return any_bad;
}

// Block-wide box of the stencils whose first-node cells span [lo, hi] per
// axis, with the vote on `bad`; thread 0 publishes the box in par.
template <int ORDER, int ES = 4>
__device__ __forceinline__ BoxPar tile_box(const Grid& g, int lo1, int lo2, int lo3, int hi1, int hi2,
                                           int hi3, bool bad, int (*red)[TILE2], int* par, int lane, int warp)
{
    int b[6];
    const bool any_bad = tile_bounds(lo1, lo2, lo3, hi1, hi2, hi3, bad, red, lane, warp, b);
    if (threadIdx.x == 0) box_geometry<ORDER, ES>(box_grid(g), b[0], b[1], b[2], b[3], b[4], b[5], any_bad, par);
    __syncthreads();
    BoxPar bp;
    bp.O1 = par[0]; bp.O2 = par[1]; bp.O3 = par[2];
    bp.E1 = par[3]; bp.E2 = par[4]; bp.E3 = par[5]; bp.S3 = par[6];
    return bp;
}

// Tile-bounds table of a displacement field, written by the backtrace that
// produced the field: entry t (the CTA index of the tiled grid, x fastest) is
// tb[2t] = (a1, a2, a3, bad) and tb[2t + 1] = (z1, z2, z3, 0), the first-node
// cell bounds of the tile's points (before the -OFF shift) and whether a
// displacement failed disp_ok.
__device__ __forceinline__ unsigned tile_index()
{
    return (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
}
#endif

// Two 16-bit values packed in a word (low half first) widened to FP32.
template <class S>
__device__ __forceinline__ float2 widen2(uint32_t w)
{
    S lo, hi;
    const unsigned short ulo = static_cast<unsigned short>(w & 0xffffu);
    const unsigned short uhi = static_cast<unsigned short>(w >> 16);
    memcpy(&lo, &ulo, 2);
    memcpy(&hi, &uhi, 2);
    return make_float2(to_f32<S>(lo), to_f32<S>(hi));
}

// Bytes per copy with which the box of f is staged: the widest chunk that the
// x3 origin, the x3 extent, n3 and the address of f are all multiples of (a
// field passed by a caller may start at any 4-byte boundary); 0 when not even
// pairs of values line up (FP32 only: single values then).
template <class S>
__device__ __forceinline__ int box_chunk_bytes(const Grid& g, const S* f, const BoxPar& bp)
{
    const unsigned a = static_cast<unsigned>(bp.O3 | bp.E3 | g.n3) * static_cast<unsigned>(sizeof(S)) |
                       static_cast<unsigned>(reinterpret_cast<uintptr_t>(f));
    if ((a & 15u) == 0) return 16;
    if ((a & 7u) == 0) return 8;
    return sizeof(S) == 2 ? 4 : 0;  // 16-bit fields are the context's own: even rows at 4-byte boundaries
}

// Threads per box row when chunks of BYTES are staged by columns: a row of 64
// values (two bank rows, the usual box) in one pass.
template <class S, int BYTES>
struct ColumnMap {
    static constexpr int VPC = BYTES / static_cast<int>(sizeof(S));  // values per chunk
    static constexpr int LPR = 64 / VPC;                             // threads per row
};

// Origin of the box wrapped into the grid.
struct BoxOrigin {
    int w1, w2, w3;
    __device__ __forceinline__ BoxOrigin(const Grid& g, const BoxPar& bp)
        : w1(wrap_index(bp.O1, g.n1)), w2(wrap_index(bp.O2, g.n2)), w3(wrap_index(bp.O3, g.n3))
    {
    }
};

// Box staging by columns: thread t owns box row t / LPR (and every
// kTileThreads / LPR rows on) and chunk t % LPR (+ LPR) and copies that chunk
// of each of the E1 planes in turn, so the wrapped x2 / x3 indices and the row
// pointer are formed once per (row, chunk) and a plane costs one address step.
// dst0: the box (FP32) or the 16-bit staging area, whose rows are S3 values
// apart.  182 x 218 x 182 (n3 not a multiple of 4): 8-byte chunks of FP32 and
// 4-byte pairs of halves instead of value-wise row loops took the FP16 adjoint
// step from 171 to 111 us (the tile-bounds table included).
template <class S, int BYTES>
__device__ __forceinline__ void stage_box_columns(const Grid& g, const S* __restrict__ f, uint32_t dst0,
                                                  const BoxPar& bp, const BoxOrigin* origin)
{
    constexpr int VPC = ColumnMap<S, BYTES>::VPC, LPR = ColumnMap<S, BYTES>::LPR;
    const BoxOrigin w = origin ? *origin : BoxOrigin(g, bp);
    const int w1 = w.w1, w2 = w.w2, w3 = w.w3;
    const int nch = bp.E3 / VPC;
    const uint32_t row_bytes = static_cast<uint32_t>(bp.S3) * sizeof(S);
    const uint32_t plane_bytes = row_bytes * static_cast<uint32_t>(bp.E2);
    for (int b = threadIdx.x / LPR; b < bp.E2; b += kTileThreads / LPR) {
        const int gj = box_wrap(w2 + b, g.n2);
        for (int c = threadIdx.x % LPR; c < nch; c += LPR) {
            const int gk = box_wrap(w3 + VPC * c, g.n3);
            const S* src = f + static_cast<size_t>(gj) * g.n3 + gk;
            uint32_t dst = dst0 + static_cast<uint32_t>(b) * row_bytes + static_cast<uint32_t>(BYTES) * c;
            int gi = w1;
            for (int a = 0; a < bp.E1; ++a) {
                if constexpr (BYTES == 16)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst),
                                 "l"(src + static_cast<size_t>(gi) * g.n23)
                                 : "memory");
                else
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(dst),
                                 "l"(src + static_cast<size_t>(gi) * g.n23), "n"(BYTES)
                                 : "memory");
                dst += plane_bytes;
                gi = gi + 1 == g.n1 ? 0 : gi + 1;
            }
        }
    }
}

// Widen the chunks stage_box_columns copied from this thread, in its order.
template <class S, int BYTES>
__device__ __forceinline__ void widen_box_columns(const uint32_t* stage, float* box, const BoxPar& bp)
{
    constexpr int VPC = ColumnMap<S, BYTES>::VPC, LPR = ColumnMap<S, BYTES>::LPR;
    const int nch = bp.E3 / VPC;
    for (int b = threadIdx.x / LPR; b < bp.E2; b += kTileThreads / LPR)
        for (int c = threadIdx.x % LPR; c < nch; c += LPR)
            for (int a = 0; a < bp.E1; ++a) {
                const int r = a * bp.E2 + b;
                const uint32_t* sp = stage + r * (bp.S3 / 2) + c * (VPC / 2);
                float* dp = box + r * bp.S3 + c * VPC;
                if constexpr (BYTES == 16) {
                    const uint4 w = *reinterpret_cast<const uint4*>(sp);
                    const float2 p0 = widen2<S>(w.x), p1 = widen2<S>(w.y), p2 = widen2<S>(w.z), p3 = widen2<S>(w.w);
                    reinterpret_cast<float4*>(dp)[0] = make_float4(p0.x, p0.y, p1.x, p1.y);
                    reinterpret_cast<float4*>(dp)[1] = make_float4(p2.x, p2.y, p3.x, p3.y);
                } else if constexpr (BYTES == 8) {
                    const uint2 w = *reinterpret_cast<const uint2*>(sp);
                    const float2 p0 = widen2<S>(w.x), p1 = widen2<S>(w.y);
                    *reinterpret_cast<float4*>(dp) = make_float4(p0.x, p0.y, p1.x, p1.y);
                } else {
                    *reinterpret_cast<float2*>(dp) = widen2<S>(*sp);
                }
            }
}

// Copy the (periodically wrapped) box of f into shared memory asynchronously:
// FP32 fields into the box itself, 16-bit ones as raw values into a staging
// area behind it (tile_widen_box then fills the box).  origin: the wrapped origin,
// when the caller keeps it from field to field.
template <class S>
__device__ __forceinline__ void tile_load_box(const Grid& g, const S* __restrict__ f, float* box,
                                              const BoxPar& bp, int lane, int warp,
                                              const BoxOrigin* origin = nullptr)
{
    const int bytes = box_chunk_bytes<S>(g, f, bp);
    if constexpr (sizeof(S) == 4) {
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(box));
        if (bytes == 16) {
            stage_box_columns<S, 16>(g, f, dst, bp, origin);
        } else if (bytes == 8) {
            stage_box_columns<S, 8>(g, f, dst, bp, origin);
        } else {
            // a caller's field at an odd 4-byte boundary: value by value
            const int w1 = wrap_index(bp.O1, g.n1), w2 = wrap_index(bp.O2, g.n2), w3 = wrap_index(bp.O3, g.n3);
            for (int a = 0; a < bp.E1; ++a) {
                const S* plane = f + static_cast<size_t>(box_wrap(w1 + a, g.n1)) * g.n23;
                for (int b = warp; b < bp.E2; b += TILE2) {
                    const S* src = plane + box_wrap(w2 + b, g.n2) * g.n3;
                    float* row = box + (a * bp.E2 + b) * bp.S3;
                    for (int c = lane; c < bp.E3; c += 32)
                        cp_async_f32(row + c, reinterpret_cast<const float*>(src + box_wrap(w3 + c, g.n3)));
                }
            }
        }
    } else {
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(box + bp.E1 * bp.E2 * bp.S3));
        if (bytes == 16)
            stage_box_columns<S, 16>(g, f, dst, bp, origin);
        else if (bytes == 8)
            stage_box_columns<S, 8>(g, f, dst, bp, origin);
        else
            stage_box_columns<S, 4>(g, f, dst, bp, origin);
    }
}

// Completion of tile_load_box for 16-bit storage: every thread waits for its
// own copies and widens exactly the chunks it issued, in the same order, so no
// barrier separates the copy from the widening; the caller's barrier before
// the stencils publishes the box.  FP32 storage: nothing (the caller waits
// for the copies).
template <class S>
__device__ __forceinline__ void tile_widen_box(const Grid& g, const S* f, float* box, const BoxPar& bp)
{
    if constexpr (sizeof(S) == 2) {
        const uint32_t* stage = reinterpret_cast<const uint32_t*>(box + bp.E1 * bp.E2 * bp.S3);
        const int bytes = box_chunk_bytes<S>(g, f, bp);
        cp_async_wait_all();
        if (bytes == 16)
            widen_box_columns<S, 16>(stage, box, bp);
        else if (bytes == 8)
            widen_box_columns<S, 8>(stage, box, bp);
        else
            widen_box_columns<S, 4>(stage, box, bp);
    }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 32-bit shared-memory load at a byte address plus an immediate byte offset.
template <int BYTE_OFF>
__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];\n" : "=f"(v) : "r"(addr), "n"(BYTE_OFF));
    return v;
}

template <int ORDER>
__device__ __forceinline__ float row_dot(uint32_t addr, const float w[4])
{
    if constexpr (Scheme<ORDER>::M == 4) {
        float s = w[0] * lds_f32<0>(addr);
        s = fmaf(w[1], lds_f32<4>(addr), s);
        s = fmaf(w[2], lds_f32<8>(addr), s);
        return fmaf(w[3], lds_f32<12>(addr), s);
    } else {
        return fmaf(w[1], lds_f32<4>(addr), w[0] * lds_f32<0>(addr));
    }
}

// Split of a displacement inside a fitting box: floor and fraction.  Every
// displacement of a tile whose box fits passed disp_ok (finite, |d| < 2^20),
// where this floor equals the clamped split of the bounds pass; with a box
// from a tile-bounds table, every point also passed in_box.
__host__ __device__ __forceinline__ int split_in_box(float d, float& t)
{
#ifdef __CUDA_ARCH__
    const int fl = __float2int_rd(d);
#else
    // the device conversion: floor, saturated to the int range, NaN to 0
    const float f = floorf(d);
    const int fl = d != d ? 0 : (f >= 2147483648.0f ? INT_MAX : (f < -2147483648.0f ? INT_MIN : static_cast<int>(f)));
#endif
    t = d - static_cast<float>(fl);
    return fl;
}

// Offset in the box (floats) of the first stencil node of the point
// (i, j, k) + (d1, d2, d3), and the three fractions.
template <int ORDER>
__host__ __device__ __forceinline__ int tile_offset(const BoxPar& bp, int i, int j, int k, float d1, float d2,
                                                    float d3, float& t1, float& t2, float& t3)
{
    constexpr int OFF = Scheme<ORDER>::OFF;
    const int P = bp.E2 * bp.S3;
    return (i + split_in_box(d1, t1) - OFF - bp.O1) * P + (j + split_in_box(d2, t2) - OFF - bp.O2) * bp.S3 +
           (k + split_in_box(d3, t3) - OFF - bp.O3);
}

// Whether the stencil of (i, j, k) + (d1, d2, d3) lies inside the box: its
// first-node offsets along each axis in [0, E - M].  The floor saturates for
// |d| >= 2^31 and is 0 for NaN (as the device conversion does), and the
// offsets are formed in unsigned arithmetic, so no input reaches an index
// outside the box without failing this test.
template <int ORDER>
__host__ __device__ __forceinline__ bool in_box(const BoxPar& bp, int i, int j, int k, float d1, float d2, float d3)
{
    constexpr int M = Scheme<ORDER>::M;
    constexpr int OFF = Scheme<ORDER>::OFF;
    float t;
    const unsigned r1 = static_cast<unsigned>(i) - static_cast<unsigned>(OFF + bp.O1) +
                        static_cast<unsigned>(split_in_box(d1, t));
    const unsigned r2 = static_cast<unsigned>(j) - static_cast<unsigned>(OFF + bp.O2) +
                        static_cast<unsigned>(split_in_box(d2, t));
    const unsigned r3 = static_cast<unsigned>(k) - static_cast<unsigned>(OFF + bp.O3) +
                        static_cast<unsigned>(split_in_box(d3, t));
    return bp.E1 >= M && bp.E2 >= M && bp.E3 >= M && r1 <= static_cast<unsigned>(bp.E1 - M) &&
           r2 <= static_cast<unsigned>(bp.E2 - M) && r3 <= static_cast<unsigned>(bp.E3 - M);
}

template <int ORDER>
__device__ __forceinline__ float tile_eval(const float* box, const BoxPar& bp, int i, int j, int k, float d1,
                                           float d2, float d3)
{
    constexpr int M = Scheme<ORDER>::M;
    const int P = bp.E2 * bp.S3;
    float t1, t2, t3, w1[4], w2[4], w3[4];
    const int o = tile_offset<ORDER>(bp, i, j, k, d1, d2, d3, t1, t2, t3);
    axis_weights<ORDER>(t1, w1);
    axis_weights<ORDER>(t2, w2);
    axis_weights<ORDER>(t3, w3);
    float val = 0.0f;
#if CLAIRE_FFMA2
    // rows b and b+1 of plane a are contracted along x3 together in one
    // packed FMA per node; then the x2 weights pair up the same way
    // rows b and b+1 of plane a are contracted together, one packed FMA per
    // x3 node with the products w2[b] w3[c], w2[b+1] w3[c] formed once per point
    const uint32_t base = smem_u32(box) + 4u * static_cast<uint32_t>(o);
    const uint32_t P4 = 4u * static_cast<uint32_t>(P), S4 = 4u * static_cast<uint32_t>(bp.S3);
    float2 W[M / 2][M];
#pragma unroll
    for (int b = 0; b < M; b += 2)
#pragma unroll
        for (int c = 0; c < M; ++c) W[b / 2][c] = __fmul2_rn(make_float2(w2[b], w2[b + 1]), make_float2(w3[c], w3[c]));
#pragma unroll
    for (int a = 0; a < M; ++a) {
        const uint32_t r0a = base + a * P4;
        float2 acc = __fmul2_rn(W[0][0], make_float2(lds_f32<0>(r0a), lds_f32<0>(r0a + S4)));
#pragma unroll
        for (int b = 0; b < M; b += 2) {
            const uint32_t r0 = r0a + b * S4, r1 = r0 + S4;
            if (b > 0) acc = __ffma2_rn(W[b / 2][0], make_float2(lds_f32<0>(r0), lds_f32<0>(r1)), acc);
            acc = __ffma2_rn(W[b / 2][1], make_float2(lds_f32<4>(r0), lds_f32<4>(r1)), acc);
            if constexpr (Scheme<ORDER>::M == 4) {
                acc = __ffma2_rn(W[b / 2][2], make_float2(lds_f32<8>(r0), lds_f32<8>(r1)), acc);
                acc = __ffma2_rn(W[b / 2][3], make_float2(lds_f32<12>(r0), lds_f32<12>(r1)), acc);
            }
        }
        val = fmaf(w1[a], acc.x + acc.y, val);
    }
#elif CLAIRE_LDS_ASM
    const uint32_t base = smem_u32(box) + 4u * static_cast<uint32_t>(o);
    const uint32_t P4 = 4u * static_cast<uint32_t>(P), S4 = 4u * static_cast<uint32_t>(bp.S3);
#pragma unroll
    for (int a = 0; a < M; ++a) {
        float sa = 0.0f;
#pragma unroll
        for (int b = 0; b < M; ++b) sa = fmaf(w2[b], row_dot<ORDER>(base + a * P4 + b * S4, w3), sa);
        val = fmaf(w1[a], sa, val);
    }
#else
#pragma unroll
    for (int a = 0; a < M; ++a) {
        float sa = 0.0f;
#pragma unroll
        for (int b = 0; b < M; ++b) {
            const int row = o + a * P + b * bp.S3;
            float sb = 0.0f;
#pragma unroll
            for (int c = 0; c < M; ++c) sb = fmaf(w3[c], box[row + c], sb);
            sa = fmaf(w2[b], sb, sa);
        }
        val = fmaf(w1[a], sa, val);
    }
#endif
    return val;
}

// Gather f at x + d for the CTA's tile and hand each value to the epilogue.
//
// Shared-memory layout of the box: element (a, b, c) at (a E2 + b) S3 + c
// with the row stride S3 a multiple of 32 floats, so an element's bank is its
// column mod 32 whatever its row: the 32 lanes of a warp (consecutive x3
// arrivals, hence consecutive departure columns, but rows that vary with the
// x1/x2 displacement) read 32 different banks.  The epilogue's operands are
// requested (prefetch) while the box is in flight and consumed (finish) after
// the stencil is evaluated.
// FULL: the tiles cover the grid exactly (n3 % 32 = n2 % 8 = n1 % TILE1 = 0),
// so no point of a tile is out of range and the bounds tests compile away.
// TB: the box comes from the tile-bounds table tb that the
// backtrace wrote with d, so the CTA starts staging it at once, reads the
// displacements and the epilogue operands while it is in flight, and needs no
// block reduction.  Every point is checked against the box (in_box); if any
// fails, which a table written with this d never causes, the tile takes the
// global-memory path.
template <int ORDER, class Epi, class S, bool FULL, bool TB = false, bool WIDE = false>
__global__ void __launch_bounds__(kTileThreads, tile_min_blocks<ORDER, sizeof(S), WIDE>())
    k_gather_tiled(Grid g, const S* __restrict__ f, const float* __restrict__ d, Epi epi,
                   const int4* __restrict__ tb = nullptr)
{
    extern __shared__ float box[];
    __shared__ int red[6][TILE2];
    __shared__ int par[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * TILE3 + lane;
    const int j = blockIdx.y * TILE2 + warp;
    const int i0 = blockIdx.z * TILE1;
    const size_t N = g.N;
    const bool col_ok = FULL || ((k < g.n3) && (j < g.n2));
    const uint32_t p0 = static_cast<uint32_t>(i0) * g.n23 + j * g.n3 + k;
    auto valid = [&](int q) { return FULL || (col_ok && i0 + q < g.n1); };

    if constexpr (TB) {
        const unsigned t = tile_index();
        const int4 lo = __ldg(tb + 2 * t), hi = __ldg(tb + 2 * t + 1);
        int gp[7];
        box_geometry<ORDER, sizeof(S)>(box_grid(g), lo.x, lo.y, lo.z, hi.x, hi.y, hi.z, lo.w != 0, gp);
        BoxPar bp;
        bp.O1 = gp[0]; bp.O2 = gp[1]; bp.O3 = gp[2];
        bp.E1 = gp[3]; bp.E2 = gp[4]; bp.E3 = gp[5]; bp.S3 = gp[6];
        if (bp.E1 != 0) tile_load_box<S>(g, f, box, bp, lane, warp);  // E1 is the same in every thread
        float e1[TILE1], e2[TILE1], e3[TILE1];
        typename Epi::Pre pre[TILE1];
        bool out = bp.E1 == 0;
#pragma unroll
        for (int q = 0; q < TILE1; ++q) {
            if (!valid(q)) continue;
            const uint32_t p = p0 + q * g.n23;
            e1[q] = __ldg(d + p);
            e2[q] = __ldg(d + N + p);
            e3[q] = __ldg(d + 2 * N + p);
            pre[q] = epi.prefetch(p);
        }
#pragma unroll
        for (int q = 0; q < TILE1; ++q)
            if (valid(q)) out = out || !in_box<ORDER>(bp, i0 + q, j, k, e1[q], e2[q], e3[q]);
        if (bp.E1 != 0) tile_widen_box<S>(g, f, box, bp);
        cp_async_wait_all();
        if (__syncthreads_or(out)) {
            if (threadIdx.x == 0) atomicAdd(&g_gather_global_tiles, 1ull);
#pragma unroll
            for (int q = 0; q < TILE1; ++q)
                if (valid(q))
                    epi.finish(p0 + q * g.n23, gather_global<ORDER, S>(g, f, i0 + q, j, k, e1[q], e2[q], e3[q]),
                               pre[q]);
            return;
        }
#pragma unroll
        for (int q = 0; q < TILE1; ++q)
            if (valid(q))
                epi.finish(p0 + q * g.n23, tile_eval<ORDER>(box, bp, i0 + q, j, k, e1[q], e2[q], e3[q]), pre[q]);
        return;
    }
    float d1[TILE1], d2[TILE1], d3[TILE1];
    int lo1 = INT_MAX, lo2 = INT_MAX, lo3 = INT_MAX, hi1 = INT_MIN, hi2 = INT_MIN, hi3 = INT_MIN;
    bool bad = false;
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        if (valid(q)) {
            const uint32_t p = p0 + q * g.n23;
            d1[q] = __ldg(d + p);
            d2[q] = __ldg(d + N + p);
            d3[q] = __ldg(d + 2 * N + p);
            bounds_add(i0 + q, d1[q], lo1, hi1, bad);
            bounds_add(j, d2[q], lo2, hi2, bad);
            bounds_add(k, d3[q], lo3, hi3, bad);
        }
    }
    const BoxPar bp = tile_box<ORDER, sizeof(S)>(g, lo1, lo2, lo3, hi1, hi2, hi3, bad, red, par, lane, warp);
    if (bp.E1 == 0) {
        // the tile's box does not fit: gather it from global memory (kept out
        // of the shared-memory path, which then has no call in its loop)
        if (threadIdx.x == 0) atomicAdd(&g_gather_global_tiles, 1ull);
#pragma unroll
        for (int q = 0; q < TILE1; ++q) {
            if (!valid(q)) continue;
            const uint32_t p = p0 + q * g.n23;
            const typename Epi::Pre pr = epi.prefetch(p);
            epi.finish(p, gather_global<ORDER, S>(g, f, i0 + q, j, k, d1[q], d2[q], d3[q]), pr);
        }
        return;
    }
    tile_load_box<S>(g, f, box, bp, lane, warp);
    // epilogue operands of every point are requested while the box is in flight
    typename Epi::Pre pre[TILE1];
#pragma unroll
    for (int q = 0; q < TILE1; ++q)
        if (valid(q)) pre[q] = epi.prefetch(p0 + q * g.n23);
    tile_widen_box<S>(g, f, box, bp);
    cp_async_wait_all();
    __syncthreads();
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        if (!valid(q)) continue;
        const float val = tile_eval<ORDER>(box, bp, i0 + q, j, k, d1[q], d2[q], d3[q]);
        epi.finish(p0 + q * g.n23, val, pre[q]);
    }
}

// nf fields f + q N (q < nf) gathered at one displacement d into out + q N:
// the displacements, bounds and box geometry are taken once per tile, and the
// box of each field is staged into the same shared memory in turn.  Per point
// and field this moves (8 nf + 12) / nf bytes instead of 20.
// MAP: the step of the deformation map, f = u^j and out = u^{j+1} = u^j(X) +
// (X - x) in physical units, nf = 3.  It reads its 192 stencil values from the
// box as the gathers do; the per-point kernel it replaced fetched them through
// L1 (256^3, CFL 3.4: 0.80 ms per step; from the box 0.56 ms).
// Every order takes the wide box here (set by the launch): the displacements and bounds
// are read once for all fields, so that six CTAs gain nothing.
template <int ORDER, bool FULL, bool MAP>
__global__ void __launch_bounds__(kTileThreads, CLAIRE_TILE_MIN_BLOCKS)
    k_gather_tiled_fields(Grid g, const float* __restrict__ f, int nf, const float* __restrict__ d,
                          float* __restrict__ out)
{
    extern __shared__ float box[];
    __shared__ int red[6][TILE2];
    __shared__ int par[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * TILE3 + lane;
    const int j = blockIdx.y * TILE2 + warp;
    const int i0 = blockIdx.z * TILE1;
    const size_t N = g.N;
    const bool col_ok = FULL || ((k < g.n3) && (j < g.n2));
    const uint32_t p0 = static_cast<uint32_t>(i0) * g.n23 + j * g.n3 + k;
    auto valid = [&](int q) { return FULL || (col_ok && i0 + q < g.n1); };
    float d1[TILE1], d2[TILE1], d3[TILE1];
    int lo1 = INT_MAX, lo2 = INT_MAX, lo3 = INT_MAX, hi1 = INT_MIN, hi2 = INT_MIN, hi3 = INT_MIN;
    bool bad = false;
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        if (valid(q)) {
            const uint32_t p = p0 + q * g.n23;
            d1[q] = __ldg(d + p);
            d2[q] = __ldg(d + N + p);
            d3[q] = __ldg(d + 2 * N + p);
            bounds_add(i0 + q, d1[q], lo1, hi1, bad);
            bounds_add(j, d2[q], lo2, hi2, bad);
            bounds_add(k, d3[q], lo3, hi3, bad);
        }
    }
    auto moved = [&](int fld, int q, float val) {
        const float dc = fld == 0 ? d1[q] : (fld == 1 ? d2[q] : d3[q]);
        return fmaf(dc, fld == 0 ? g.h1 : (fld == 1 ? g.h2 : g.h3), val);
    };
    const BoxPar bp = tile_box<ORDER, 4>(g, lo1, lo2, lo3, hi1, hi2, hi3, bad, red, par, lane, warp);
    if (bp.E1 == 0) {
        if (threadIdx.x == 0) atomicAdd(&g_gather_global_tiles, 1ull);
        for (int fld = 0; fld < nf; ++fld)
#pragma unroll
            for (int q = 0; q < TILE1; ++q) {
                if (!valid(q)) continue;
                const uint32_t p = p0 + q * g.n23;
                const float val = gather_global<ORDER, float>(g, f + fld * N, i0 + q, j, k, d1[q], d2[q], d3[q]);
                out[fld * N + p] = MAP ? moved(fld, q, val) : val;
            }
        return;
    }
    // three divisions per thread and field otherwise (256^3, four trilinear fields at no
    // displacement: 255 -> 239 us); the other orders have no registers for them
    const BoxOrigin origin(g, bp);
    for (int fld = 0; fld < nf; ++fld) {
        // the weights and offsets of the four points are formed anew for each
        // field: kept across the loop they do not fit the 64 registers (the
        // compiler then spilled 240 bytes per thread; those of the trilinear
        // stencil do)
        if constexpr (ORDER != 1) {
#pragma unroll
            for (int q = 0; q < TILE1; ++q) asm volatile("" : "+f"(d1[q]), "+f"(d2[q]), "+f"(d3[q]));
        }
        tile_load_box<float>(g, f + fld * N, box, bp, lane, warp, ORDER == 1 ? &origin : nullptr);
        cp_async_wait_all();
        __syncthreads();
#pragma unroll
        for (int q = 0; q < TILE1; ++q) {
            if (!valid(q)) continue;
            const float val = tile_eval<ORDER>(box, bp, i0 + q, j, k, d1[q], d2[q], d3[q]);
            out[fld * N + p0 + q * g.n23] = MAP ? moved(fld, q, val) : val;
        }
        __syncthreads();  // every read of this field's box is done before the next staging
    }
}

inline bool tiles_cover_grid(const Grid& g)
{
    return g.n3 % TILE3 == 0 && g.n2 % TILE2 == 0 && g.n1 % TILE1 == 0;
}

inline dim3 tiled_grid(const Grid& g)
{
    return dim3((g.n3 + TILE3 - 1) / TILE3, (g.n2 + TILE2 - 1) / TILE2, (g.n1 + TILE1 - 1) / TILE1);
}

template <int ORDER, int ES = 4>
size_t tiled_smem_bytes(const Grid& g)
{
    return box_cap<ORDER, ES>(g) * sizeof(float);
}

template <int ORDER, class Epi, class S, bool FULL, bool TB>
inline void launch_tiled_as(const Grid& g, const S* f, const float* d, const Epi& e, cudaStream_t st, const int4* tb)
{
    const size_t smem = tiled_smem_bytes<ORDER, sizeof(S)>(g);
    auto launch = [&](auto kernel) {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        kernel<<<tiled_grid(g), kTileThreads, smem, st>>>(g, f, d, e, tb);
    };
    if constexpr (ORDER == 1 && sizeof(S) == 4) {
        if (g.wide) return launch(k_gather_tiled<ORDER, Epi, S, FULL, TB, true>);
    }
    launch(k_gather_tiled<ORDER, Epi, S, FULL, TB>);
}

template <int ORDER, class Epi, class S>
inline void launch_tiled(const Grid& g, const S* f, const float* d, const Epi& e, cudaStream_t st,
                         const int4* tb = nullptr)
{
    const bool full = tiles_cover_grid(g);
    if (tb && full)
        launch_tiled_as<ORDER, Epi, S, true, true>(g, f, d, e, st, tb);
    else if (tb)
        launch_tiled_as<ORDER, Epi, S, false, true>(g, f, d, e, st, tb);
    else if (full)
        launch_tiled_as<ORDER, Epi, S, true, false>(g, f, d, e, st, tb);
    else
        launch_tiled_as<ORDER, Epi, S, false, false>(g, f, d, e, st, tb);
}

// ---- epilogues: prefetch(p) loads the point's operands early, finish(p, v, pre)
// completes; S is the storage type of the fields they read and write ----

// plain interpolation / state step: out = f(X)
template <class S>
struct EpiStore {
    S* __restrict__ out;
    struct Pre {};
    __device__ __forceinline__ Pre prefetch(uint32_t) const { return Pre{}; }
    __device__ __forceinline__ void finish(uint32_t p, float v, const Pre&) const { stf<S>(out + p, v); }
};

// adjoint step (Eq. (4), Heun along X+): lambda^j from lambda^{j+1}(X+)
template <class S>
struct EpiAdjointOnly {
    const S* __restrict__ divv;
    const S* __restrict__ divXp;
    S* __restrict__ lam;
    float dt;
    struct Pre {
        float dX, dx;
    };
    __device__ __forceinline__ Pre prefetch(uint32_t p) const { return Pre{ldf<S>(divXp + p), ldf<S>(divv + p)}; }
    __device__ __forceinline__ void finish(uint32_t p, float a, const Pre& r) const
    {
        const float adX = a * r.dX;
        const float pred = fmaf(dt, adX, a);
        stf<S>(lam + p, fmaf(0.5f * dt, fmaf(pred, r.dx, adX), a));
    }
};

// incremental state with precomputed source: q = f(X) + coef F
template <class S>
struct EpiIncSource {
    const S* __restrict__ F;
    S* __restrict__ q;
    float coef;
    struct Pre {
        float f;
    };
    __device__ __forceinline__ Pre prefetch(uint32_t p) const { return Pre{ldf<S>(F + p)}; }
    __device__ __forceinline__ void finish(uint32_t p, float a, const Pre& r) const
    {
        stf<S>(q + p, fmaf(coef, r.f, a));
    }
};

// last incremental state step, start of the incremental adjoint: lt = -(f(X) + coef F)
template <class S>
struct EpiIncSourceLast {
    const S* F;  // may alias lam: each point reads its F before writing lam
    S* lam;
    float coef;
    struct Pre {
        float f;
    };
    __device__ __forceinline__ Pre prefetch(uint32_t p) const { return Pre{to_f32<S>(F[p])}; }
    __device__ __forceinline__ void finish(uint32_t p, float a, const Pre& r) const
    {
        stf<S>(lam + p, -fmaf(coef, r.f, a));
    }
};

// Incremental state step with its source formed in place (grad m^{j+1}
// stored): f = -vt . grad m^{j+1} at the arrival point, rounded to the
// storage type as a stored source would be, then q = f(X) + coef f.  It
// reads vt and grad m^{j+1} (24 B) instead of a precomputed source (4 B), so
// the pass that wrote every level's source is not needed.
template <class S>
__device__ __forceinline__ float inc_source_at(const float* __restrict__ vt, const S* __restrict__ gm, uint32_t N,
                                               uint32_t p)
{
    const float f = -(__ldg(vt + p) * ldf<S>(gm + p) + __ldg(vt + N + p) * ldf<S>(gm + N + p) +
                      __ldg(vt + 2 * N + p) * ldf<S>(gm + 2 * N + p));
    return to_f32<S>(from_f32<S>(f));
}

template <class S>
struct EpiIncGrad {
    const float* __restrict__ vt;
    const S* __restrict__ gm;  // grad m^{j+1}, 3N values
    S* __restrict__ q;
    float coef;
    uint32_t N;
    struct Pre {
        float f;
    };
    __device__ __forceinline__ Pre prefetch(uint32_t p) const { return Pre{inc_source_at<S>(vt, gm, N, p)}; }
    __device__ __forceinline__ void finish(uint32_t p, float a, const Pre& r) const
    {
        stf<S>(q + p, fmaf(coef, r.f, a));
    }
};

// last step with its source formed in place: lt = -(f(X) + coef f)
template <class S>
struct EpiIncGradLast {
    const float* __restrict__ vt;
    const S* __restrict__ gm;  // grad m^{nt}
    S* __restrict__ lam;
    float coef;
    uint32_t N;
    struct Pre {
        float f;
    };
    __device__ __forceinline__ Pre prefetch(uint32_t p) const { return Pre{inc_source_at<S>(vt, gm, N, p)}; }
    __device__ __forceinline__ void finish(uint32_t p, float a, const Pre& r) const
    {
        stf<S>(lam + p, -fmaf(coef, r.f, a));
    }
};

}  // namespace claire
