// Semi-Lagrangian kernels of libclaire (sm_103a): RK2 backtrace, off-grid
// gathers with the fused source terms of the state, adjoint and incremental
// solves, 8th-order finite differences, deformation-map transport and the
// Jacobian determinant.  Method: "CLAIRE at scale" (arXiv 2209.08189),
// Sec. 2.2 (SL with RK2, FD8) and Sec. 3 (IP and FD kernels).
#include "detj.cuh"
#include "internal.h"
#include "sl_tiled.cuh"

#include <type_traits>

namespace claire {

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(uint32_t n) { return (n + kThreads - 1) / kThreads; }

// ---------------------------------------------------------------------------
// gathers
// ---------------------------------------------------------------------------

// Heun characteristic: sign = +1 gives X = x - dt/2 [v(x) + v(x - dt v(x))],
// sign = -1 gives X+ = x + dt/2 [v(x) + v(x + dt v(x))]; d in grid units.
// The three velocity gathers at the predictor point are served from a
// shared-memory box per 4 x 8 x 32 tile (one box, staged once per component;
// the predictor points of a tile share its bounds).  TBW: also write the
// tile-bounds table of d (tile_index order), from the same FP32 values that
// are stored, for the gathers at d.
template <int ORDER, bool FULL, bool TBW, bool WIDE = false>
__global__ void __launch_bounds__(kTileThreads, tile_min_blocks<ORDER, 4, WIDE>())
    k_backtrace_tiled(Grid g, const float* __restrict__ v, const float* __restrict__ vc, float dt, float sign,
                      float* __restrict__ d, int4* __restrict__ tb)
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
    const float sdt = sign * dt;
    float u1[TILE1], u2[TILE1], u3[TILE1];
    int lo1 = INT_MAX, lo2 = INT_MAX, lo3 = INT_MAX, hi1 = INT_MIN, hi2 = INT_MIN, hi3 = INT_MIN;
    bool bad = false;
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        u1[q] = u2[q] = u3[q] = 0.0f;
        if (FULL || (col_ok && i0 + q < g.n1)) {
            const uint32_t p = p0 + q * g.n23;
            u1[q] = __ldg(v + p) * g.ih1;
            u2[q] = __ldg(v + N + p) * g.ih2;
            u3[q] = __ldg(v + 2 * N + p) * g.ih3;
            bounds_add(i0 + q, -sdt * u1[q], lo1, hi1, bad);
            bounds_add(j, -sdt * u2[q], lo2, hi2, bad);
            bounds_add(k, -sdt * u3[q], lo3, hi3, bad);
        }
    }
    // a non-finite or huge predictor displacement sends the tile to the
    // global-memory gather (clamped split, indices always in range)
    const BoxPar bp = tile_box<ORDER, 4>(g, lo1, lo2, lo3, hi1, hi2, hi3, bad, red, par, lane, warp);
    const bool use_box = bp.E1 != 0;
    if (!use_box && threadIdx.x == 0) atomicAdd(&g_gather_global_tiles, 1ull);
    const float cc = -0.5f * sdt;
    bool dbad = false;  // a component of the characteristic itself fails disp_ok (TBW)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float* f = vc + c * N;
        const float ih = c == 0 ? g.ih1 : (c == 1 ? g.ih2 : g.ih3);
        int lo = INT_MAX, hi = INT_MIN;  // bounds of the characteristic along axis c (TBW)
        // weights and offsets are formed anew per component: kept across the
        // three they do not fit the 64 registers
#pragma unroll
        for (int q = 0; q < TILE1; ++q) asm volatile("" : "+f"(u1[q]), "+f"(u2[q]), "+f"(u3[q]));
        if (use_box) {
            tile_load_box<float>(g, f, box, bp, lane, warp);
            cp_async_wait_all();
            __syncthreads();
        }
#pragma unroll
        for (int q = 0; q < TILE1; ++q) {
            const int i = i0 + q;
            if (!(FULL || (col_ok && i < g.n1))) continue;
            const float vsq = use_box
                                  ? tile_eval<ORDER>(box, bp, i, j, k, -sdt * u1[q], -sdt * u2[q], -sdt * u3[q])
                                  : gather_global<ORDER, float>(g, f, i, j, k, -sdt * u1[q], -sdt * u2[q],
                                                                -sdt * u3[q]);
            const float uc = c == 0 ? u1[q] : (c == 1 ? u2[q] : u3[q]);
            const float dc = cc * (uc + vsq * ih);
            d[c * N + p0 + q * g.n23] = dc;
            if constexpr (TBW) bounds_add(c == 0 ? i : (c == 1 ? j : k), dc, lo, hi, dbad);
        }
        if constexpr (TBW) {
            // reduced per component, so that two bounds are live at a time (red is
            // free again: tile_box read it before its last barrier)
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0) {
                red[c][warp] = lo;
                red[3 + c][warp] = hi;
            }
        }
        if (use_box) __syncthreads();  // every read of this component is done before the next staging
    }
    if constexpr (TBW) {
        const bool any_bad = __syncthreads_or(dbad) != 0;
        if (threadIdx.x < 6) {
            // thread c: lower bound of axis c, thread 3 + c: upper bound
            const int r = threadIdx.x;
            int x = red[r][0];
#pragma unroll
            for (int w = 1; w < TILE2; ++w) x = r < 3 ? min(x, red[r][w]) : max(x, red[r][w]);
            int* e = reinterpret_cast<int*>(tb + 2 * tile_index());
            e[r < 3 ? r : r + 1] = x;
            if (r == 0) {
                e[3] = any_bad ? 1 : 0;
                e[7] = 0;
            }
        }
    }
}

template <int ORDER, bool FULL, bool TBW>
void launch_backtrace_tiled_as(const Grid& g, const float* v, const float* vc, float dt, float sign, float* d,
                               int4* tb, cudaStream_t st)
{
    const size_t smem = tiled_smem_bytes<ORDER>(g);
    auto launch = [&](auto kernel) {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        kernel<<<tiled_grid(g), kTileThreads, smem, st>>>(g, v, vc, dt, sign, d, tb);
    };
    if constexpr (ORDER == 1) {
        if (g.wide) return launch(k_backtrace_tiled<ORDER, FULL, TBW, true>);
    }
    launch(k_backtrace_tiled<ORDER, FULL, TBW>);
}

template <int ORDER>
void launch_backtrace_tiled(const Grid& g, const float* v, const float* vc, float dt, float sign, float* d,
                            int4* tb, cudaStream_t st)
{
    const bool full = tiles_cover_grid(g);
    if (tb && full)
        launch_backtrace_tiled_as<ORDER, true, true>(g, v, vc, dt, sign, d, tb, st);
    else if (tb)
        launch_backtrace_tiled_as<ORDER, false, true>(g, v, vc, dt, sign, d, tb, st);
    else if (full)
        launch_backtrace_tiled_as<ORDER, true, false>(g, v, vc, dt, sign, d, nullptr, st);
    else
        launch_backtrace_tiled_as<ORDER, false, false>(g, v, vc, dt, sign, d, nullptr, st);
}

// Sources of the incremental state for every time level at once:
// f^j = -vt . grad m^j; q0 = coef0 f^0 starts the Heun recursion and
// f^1..f^nt go to F (slot j at F + j N).  S: storage of grad m, q0, F.
// ---------------------------------------------------------------------------
// 8th-order central finite differences
// ---------------------------------------------------------------------------

// The 8th-order central difference (grid units) from the values at +s and -s
// nodes, s = 1..4: sum_s c_s (f(+s) - f(-s)) with c_s = 4/5, -1/5, 4/105,
// -1/280 (the standard stencil), accumulated in this order.
__device__ __forceinline__ float fd8_combine(const float fp[4], const float fm[4])
{
    const float cs[4] = {0.8f, -0.2f, 0.0380952380952381f, -0.003571428571428571f};
    float acc = 0.0f;
#pragma unroll
    for (int s = 0; s < 4; ++s) acc = fmaf(cs[s], fp[s] - fm[s], acc);
    return acc;
}

template <class S = float>
__device__ __forceinline__ float fd8_axis(const S* __restrict__ f, uint32_t p, int idx, int n,
                                          int stride)
{
    const long base = static_cast<long>(p) - static_cast<long>(idx) * stride;
    float fp[4], fm[4];
#pragma unroll
    for (int s = 1; s <= 4; ++s) {
        int ip = idx + s;
        ip = ip >= n ? ip - n : ip;
        int im = idx - s;
        im = im < 0 ? im + n : im;
        fp[s - 1] = ldf<S>(f + base + static_cast<long>(ip) * stride);
        fm[s - 1] = ldf<S>(f + base + static_cast<long>(im) * stride);
    }
    return fd8_combine(fp, fm);
}

// FD8 gradient of f at node p = (i, j, k), physical units
template <class S>
__device__ __forceinline__ void fd8_grad_at(const Grid& g, const S* __restrict__ f, uint32_t p, int i, int j,
                                            int k, float& g0, float& g1, float& g2)
{
    g0 = fd8_axis<S>(f, p, i, g.n1, g.n23) * g.ih1;
    g1 = fd8_axis<S>(f, p, j, g.n2, g.n3) * g.ih2;
    g2 = fd8_axis<S>(f, p, k, g.n3, 1) * g.ih3;
}

// Incremental-state sources with grad m^j computed here (FD8 of the stored
// states, no stored gradients): f^j = -vt . grad m^j; q0 = coef0 f^0,
// F[j] = f^j for j = 1..nt.
template <class S>
__global__ void __launch_bounds__(kThreads) k_inc_sources_fd(Grid g, const float* __restrict__ vt,
                                                              const S* __restrict__ m, int nt, float coef0,
                                                              S* __restrict__ q0, S* __restrict__ F)
{
    const uint32_t p = blockIdx.x * kThreads + threadIdx.x;
    if (p >= g.N) return;
    int i, j, k;
    coords_of(g, p, i, j, k);
    const size_t N = g.N;
    const float v0 = __ldg(vt + p), v1 = __ldg(vt + N + p), v2 = __ldg(vt + 2 * N + p);
    for (int l = 0; l <= nt; ++l) {
        float g0, g1, g2;
        fd8_grad_at<S>(g, m + l * N, p, i, j, k, g0, g1, g2);
        const float f = -(v0 * g0 + v1 * g1 + v2 * g2);
        if (l == 0)
            stf<S>(q0 + p, coef0 * f);
        else
            stf<S>(F + l * N + p, f);
    }
}

// Gradient body with grad m^j computed here: out_c (+)= sum_j w_j lambda^j grad_c m^j.
template <class S>
__global__ void __launch_bounds__(kThreads) k_body_fd(Grid g, const S* __restrict__ lam, const S* __restrict__ m,
                                                       int nt, float w_end, float w_mid, int accumulate,
                                                       float* __restrict__ out)
{
    const uint32_t p = blockIdx.x * kThreads + threadIdx.x;
    if (p >= g.N) return;
    int i, j, k;
    coords_of(g, p, i, j, k);
    const size_t N = g.N;
    float b0 = 0.0f, b1 = 0.0f, b2 = 0.0f;
    for (int l = 0; l <= nt; ++l) {
        const float wl = (l == 0 || l == nt ? w_end : w_mid) * ldf<S>(lam + l * N + p);
        float g0, g1, g2;
        fd8_grad_at<S>(g, m + l * N, p, i, j, k, g0, g1, g2);
        b0 = fmaf(wl, g0, b0);
        b1 = fmaf(wl, g1, b1);
        b2 = fmaf(wl, g2, b2);
    }
    if (accumulate) {
        b0 += out[p];
        b1 += out[N + p];
        b2 += out[2 * N + p];
    }
    out[p] = b0;
    out[N + p] = b1;
    out[2 * N + p] = b2;
}

template <class S>
__global__ void __launch_bounds__(kThreads) k_inc_sources(Grid g, const float* __restrict__ vt,
                                                           const S* __restrict__ gm, int nt,
                                                           float coef0, S* __restrict__ q0,
                                                           S* __restrict__ F)
{
    const uint32_t p = blockIdx.x * kThreads + threadIdx.x;
    if (p >= g.N) return;
    const size_t N = g.N;
    const float v0 = __ldg(vt + p), v1 = __ldg(vt + N + p), v2 = __ldg(vt + 2 * N + p);
    for (int j = 0; j <= nt; ++j) {
        const S* gj = gm + 3 * j * N;
        const float f = -(v0 * ldf<S>(gj + p) + v1 * ldf<S>(gj + N + p) + v2 * ldf<S>(gj + 2 * N + p));
        if (j == 0)
            stf<S>(q0 + p, coef0 * f);
        else
            stf<S>(F + j * N + p, f);
    }
}

// q0 = coef0 f^0 with f^0 = -vt . grad m^0, the start of the incremental
// state when the later steps form their sources in place (EpiIncGrad).
template <class S>
__global__ void __launch_bounds__(kThreads) k_inc_source0(Grid g, const float* __restrict__ vt,
                                                          const S* __restrict__ gm, float coef0, S* __restrict__ q0)
{
    const uint32_t p = blockIdx.x * kThreads + threadIdx.x;
    if (p >= g.N) return;
    stf<S>(q0 + p, coef0 * inc_source_at<S>(vt, gm, g.N, p));
}

// Gradient body by trapezoid in time, added to out (FP32):
// out_c (+)= sum_j w_j lambda^j grad_c m^j, w_0 = w_nt = w_end, else w_mid.
template <class S>
__global__ void __launch_bounds__(kThreads) k_body(Grid g, const S* __restrict__ lam,
                                                    const S* __restrict__ gm, int nt, float w_end,
                                                    float w_mid, int accumulate, float* __restrict__ out)
{
    const uint32_t p = blockIdx.x * kThreads + threadIdx.x;
    if (p >= g.N) return;
    const size_t N = g.N;
    float b0 = 0.0f, b1 = 0.0f, b2 = 0.0f;
    for (int j = 0; j <= nt; ++j) {
        const float wl = (j == 0 || j == nt ? w_end : w_mid) * ldf<S>(lam + j * N + p);
        const S* gj = gm + 3 * j * N;
        b0 = fmaf(wl, ldf<S>(gj + p), b0);
        b1 = fmaf(wl, ldf<S>(gj + N + p), b1);
        b2 = fmaf(wl, ldf<S>(gj + 2 * N + p), b2);
    }
    if (accumulate) {
        b0 += out[p];
        b1 += out[N + p];
        b2 += out[2 * N + p];
    }
    out[p] = b0;
    out[N + p] = b1;
    out[2 * N + p] = b2;
}

// out = a - s in storage S (start of the adjoint: lambda^{nt} = m1 - m^{nt})
template <class S>
__global__ void __launch_bounds__(kThreads) k_sub(const S* __restrict__ a, const S* __restrict__ s,
                                                   S* __restrict__ out, uint32_t n)
{
    const uint32_t p = blockIdx.x * kThreads + threadIdx.x;
    if (p < n) stf<S>(out + p, ldf<S>(a + p) - ldf<S>(s + p));
}

// out = convert(in): FP32 <-> storage S
template <class Si, class So>
__global__ void __launch_bounds__(kThreads) k_convert(const Si* __restrict__ in, So* __restrict__ out,
                                                       uint32_t n)
{
    const uint32_t p = blockIdx.x * kThreads + threadIdx.x;
    if (p < n) stf<So>(out + p, ldf<Si>(in + p));
}

// ---- FD8 over 8 x 32 columns ----
// A CTA owns an 8 x 32 column of (x2, x3) nodes over zlen consecutive x1
// planes.  Each plane of the column, with the halo of 4 nodes that its
// differences need in x2 and x3 (periodically wrapped), is staged in shared
// memory (two buffers, one barrier per plane); every thread keeps the nine
// values of its own column along x1 in registers, loading one new value per
// plane.  A plane's values are requested one plane ahead, so their latency
// overlaps the differences of the plane before.  Each value crosses HBM about
// once and L2 about 2.5 times, instead of 24 neighbour loads per point and
// field through L1/L2; the arithmetic is fd8_combine in the same order
// whatever the split.  Bound: HBM (16 B per point for a gradient or a
// divergence).  The columns need not divide the grid: nodes past its end are
// staged from the last wrapped halo node and not written.
constexpr int kFdRows = 8 + 8, kFdCols = 32 + 8;  // staged plane with its halo of 4
constexpr int kFdPlane = kFdRows * kFdCols;

// Planes per column: 32 (a quarter of the x1 halo reads of 8 planes) when
// enough columns remain to fill the chip four times over, else 16, else 8.
inline int fd_zlen(const Grid& g)
{
    const long long cols = static_cast<long long>((g.n3 + 31) / 32) * ((g.n2 + 7) / 8);
    for (int z = 32; z > 8; z /= 2)
        if (cols * ((g.n1 + z - 1) / z) >= 4 * 152 * 4) return z;
    return 8;
}

inline dim3 fd_grid(const Grid& g, int zlen)
{
    return dim3((g.n3 + 31) / 32, (g.n2 + 7) / 8, (g.n1 + zlen - 1) / zlen);
}

// The nodes a thread stages and owns in the column (bx, by).
struct FdColumn {
    int soff[3];   // plane offsets of the up to three halo-plane nodes it stages
    bool s2;       // whether it stages the third
    uint32_t col;  // plane offset of its own node (clamped into the grid)
    bool ok;       // whether its own node exists
    __device__ __forceinline__ FdColumn(const Grid& g, int bx, int by)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int k = bx * 32 + lane, j = by * 8 + warp;
        ok = k < g.n3 && j < g.n2;
        col = static_cast<uint32_t>(min(j, g.n2 - 1)) * g.n3 + min(k, g.n3 - 1);
        s2 = threadIdx.x + 2 * kThreads < kFdPlane;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const int e = min(static_cast<int>(threadIdx.x) + u * kThreads, kFdPlane - 1);
            const int row = e / kFdCols, c = e - row * kFdCols;
            // at most n + 3 (the halo of the last node; n2, n3 >= 8 > 4, so one wrap suffices)
            int gj = min(by * 8 + row - 4, g.n2 + 3);
            gj = gj < 0 ? gj + g.n2 : (gj >= g.n2 ? gj - g.n2 : gj);
            int gk = min(bx * 32 + c - 4, g.n3 + 3);
            gk = gk < 0 ? gk + g.n3 : (gk >= g.n3 ? gk - g.n3 : gk);
            soff[u] = gj * g.n3 + gk;
        }
    }
};

__device__ __forceinline__ int fd_wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// x1 queue of one field: the column's values at planes i-4 .. i+4.
template <class S>
__device__ __forceinline__ void fd_queue_fill(const Grid& g, const S* __restrict__ f, uint32_t col, int i0, float q[9])
{
#pragma unroll
    for (int s = 0; s < 9; ++s) q[s] = ldf<S>(f + static_cast<size_t>(fd_wrap(i0 - 4 + s, g.n1)) * g.n23 + col);
}

__device__ __forceinline__ float fd_queue_diff(const float q[9])
{
    float fp[4], fm[4];
#pragma unroll
    for (int s = 1; s <= 4; ++s) {
        fp[s - 1] = q[4 + s];
        fm[s - 1] = q[4 - s];
    }
    return fd8_combine(fp, fm);
}

__device__ __forceinline__ void fd_queue_push(float q[9], float next)
{
#pragma unroll
    for (int s = 0; s < 8; ++s) q[s] = q[s + 1];
    q[8] = next;
}

// Difference at sh[0] along a shared-memory stride.
template <int STRIDE>
__device__ __forceinline__ float fd_sh_diff(const float* sh)
{
    float fp[4], fm[4];
#pragma unroll
    for (int s = 1; s <= 4; ++s) {
        fp[s - 1] = sh[s * STRIDE];
        fm[s - 1] = sh[-s * STRIDE];
    }
    return fd8_combine(fp, fm);
}

// FD8 gradient.  256^3 FP32: 71 us; 182 x 218 x 182 FP16, whose grid the
// columns do not cover: 36.5 us (the per-point kernel: 77 us).
template <class S>
__global__ void __launch_bounds__(kThreads) k_fd8_grad_tiled(Grid g, const S* __restrict__ f,
                                                              S* __restrict__ out, int zlen)
{
    __shared__ float sh[2][kFdPlane];
    const FdColumn t(g, blockIdx.x, blockIdx.y);
    const int own = (static_cast<int>(threadIdx.x >> 5) + 4) * kFdCols + (threadIdx.x & 31) + 4;
    const int i0 = blockIdx.z * zlen, i1 = min(i0 + zlen, g.n1);
    const size_t N = g.N;
    float q[9];
    fd_queue_fill<S>(g, f, t.col, i0, q);
    const S* plane = f + static_cast<size_t>(i0) * g.n23;
    float p0 = ldf<S>(plane + t.soff[0]), p1 = ldf<S>(plane + t.soff[1]), p2 = t.s2 ? ldf<S>(plane + t.soff[2]) : 0.0f;
    for (int i = i0; i < i1; ++i) {
        float* b = sh[(i - i0) & 1];
        b[threadIdx.x] = p0;
        b[threadIdx.x + kThreads] = p1;
        if (t.s2) b[threadIdx.x + 2 * kThreads] = p2;
        // the next plane's values, requested before the barrier
        const float qn = ldf<S>(f + static_cast<size_t>(fd_wrap(i + 5, g.n1)) * g.n23 + t.col);
        if (i + 1 < i1) {
            plane += g.n23;
            p0 = ldf<S>(plane + t.soff[0]);
            p1 = ldf<S>(plane + t.soff[1]);
            if (t.s2) p2 = ldf<S>(plane + t.soff[2]);
        }
        __syncthreads();
        const float d1 = fd_queue_diff(q), d2 = fd_sh_diff<kFdCols>(b + own), d3 = fd_sh_diff<1>(b + own);
        if (t.ok) {
            const size_t p = static_cast<size_t>(i) * g.n23 + t.col;
            stf<S>(out + p, d1 * g.ih1);
            stf<S>(out + N + p, d2 * g.ih2);
            stf<S>(out + 2 * N + p, d3 * g.ih3);
        }
        fd_queue_push(q, qn);
    }
}

// Divergence of an FP32 vector field, stored as S (256^3: 77 us, the per-point
// kernel 171 us): x1 differences of v_1 from
// the register queue, x2 differences of v_2 from a staged plane with the x2
// halo only (16 rows of 32), x3 differences of v_3 from one with the x3 halo
// only (8 rows of 40).
template <class S>
__global__ void __launch_bounds__(kThreads) k_fd8_div_tiled(Grid g, const float* __restrict__ v,
                                                             S* __restrict__ out, int zlen)
{
    __shared__ float sh2[2][kFdRows * 32], sh3[2][8 * kFdCols];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane, j = blockIdx.y * 8 + warp;
    const bool ok = k < g.n3 && j < g.n2;
    const int kc = min(k, g.n3 - 1), jc = min(j, g.n2 - 1);
    const uint32_t col = static_cast<uint32_t>(jc) * g.n3 + kc;
    // staged nodes: v_2 at rows warp and warp + 8 of the halo column; v_3 at
    // elements t and t + 256 (only 320) of the halo rows
    int o2[2], o3[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int gj = fd_wrap(min(static_cast<int>(blockIdx.y) * 8 + warp + 8 * u - 4, g.n2 + 3), g.n2);
        o2[u] = gj * g.n3 + kc;
        const int e = min(static_cast<int>(threadIdx.x) + u * kThreads, 8 * kFdCols - 1);
        const int row = e / kFdCols, c = e - row * kFdCols;
        const int gk = fd_wrap(min(static_cast<int>(blockIdx.x) * 32 + c - 4, g.n3 + 3), g.n3);
        o3[u] = min(static_cast<int>(blockIdx.y) * 8 + row, g.n2 - 1) * g.n3 + gk;
    }
    const bool s3 = threadIdx.x + kThreads < 8 * kFdCols;
    const int i0 = blockIdx.z * zlen, i1 = min(i0 + zlen, g.n1);
    const size_t N = g.N;
    float q[9];
    fd_queue_fill<float>(g, v, col, i0, q);
    const float* w2 = v + N + static_cast<size_t>(i0) * g.n23;
    const float* w3 = v + 2 * N + static_cast<size_t>(i0) * g.n23;
    float a0 = __ldg(w2 + o2[0]), a1 = __ldg(w2 + o2[1]), c0 = __ldg(w3 + o3[0]), c1 = s3 ? __ldg(w3 + o3[1]) : 0.0f;
    for (int i = i0; i < i1; ++i) {
        const int b = (i - i0) & 1;
        sh2[b][threadIdx.x] = a0;
        sh2[b][threadIdx.x + kThreads] = a1;
        sh3[b][threadIdx.x] = c0;
        if (s3) sh3[b][threadIdx.x + kThreads] = c1;
        const float qn = __ldg(v + static_cast<size_t>(fd_wrap(i + 5, g.n1)) * g.n23 + col);
        if (i + 1 < i1) {
            w2 += g.n23;
            w3 += g.n23;
            a0 = __ldg(w2 + o2[0]);
            a1 = __ldg(w2 + o2[1]);
            c0 = __ldg(w3 + o3[0]);
            if (s3) c1 = __ldg(w3 + o3[1]);
        }
        __syncthreads();
        const float d1 = fd_queue_diff(q), d2 = fd_sh_diff<32>(&sh2[b][(warp + 4) * 32 + lane]),
                    d3 = fd_sh_diff<1>(&sh3[b][warp * kFdCols + lane + 4]);
        // one order of rounding for all storage types and grids: a 16-bit div v
        // turns another order's last FP32 bit into 2^-11 of the value
        if (ok)
            stf<S>(out + static_cast<size_t>(i) * g.n23 + col,
                   fmaf(d3, g.ih3, fmaf(d1, g.ih1, __fmul_rn(d2, g.ih2))));
        fd_queue_push(q, qn);
    }
}

// Order-preserving map between floats (no NaN) and ints, for warp extrema.
__device__ __forceinline__ int ordered_int(float x)
{
    const int i = __float_as_int(x);
    return i ^ ((i >> 31) & 0x7fffffff);
}
constexpr int kOrderedInf = 0x7f800000;  // +infinity; ~kOrderedInf is -infinity
__device__ __forceinline__ float ordered_float(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// Extrema of det(I + grad u) in FP64.
//
// Bound: the nine FD8 differences per point.  The FP64 pipe of this part runs
// 2 operations per clock and SM, so the 30 FP64 operations of every point's
// determinant were most of the kernel (256^3: 933 us).  Each determinant is
// first formed in FP32 with an error bound E; only points that may be below
// the block's smallest or above its largest value so far are formed in FP64
// (det_bounds).  A NaN or an overflow fails both comparisons and is formed in
// FP64.  The extrema are the FP64 ones of the same FP32 differences, bit for bit.
// Columns are walked by a fixed number of CTAs (one partial each).  256^3: 330 us on a
// random velocity, 345 at the end of a registration.
__global__ void __launch_bounds__(kThreads) k_detj_minmax(Grid g, const float* __restrict__ u, int zlen, int ncol,
                                                           Reduction red)
{
    __shared__ float sh[2][3][kFdPlane];
    const int own = (static_cast<int>(threadIdx.x >> 5) + 4) * kFdCols + (threadIdx.x & 31) + 4;
    const int nx = (g.n3 + 31) / 32, ny = (g.n2 + 7) / 8;
    const size_t N = g.N;
    double lo = 1e300, hi = -1e300;
    __shared__ int blo, bhi;  // the block's bounds of lo and hi (ordered ints)
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        blo = kOrderedInf;
        bhi = ~kOrderedInf;
    }
    __syncthreads();
    int par = 0;
    for (int cb = blockIdx.x; cb < ncol; cb += gridDim.x) {
        const int bx = cb % nx, by = (cb / nx) % ny, bz = cb / (nx * ny);
        const FdColumn t(g, bx, by);
        const int i0 = bz * zlen, i1 = min(i0 + zlen, g.n1);
        float q[3][9], p[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            fd_queue_fill<float>(g, u + c * N, t.col, i0, q[c]);
            const float* plane = u + c * N + static_cast<size_t>(i0) * g.n23;
            p[c][0] = __ldg(plane + t.soff[0]);
            p[c][1] = __ldg(plane + t.soff[1]);
            p[c][2] = t.s2 ? __ldg(plane + t.soff[2]) : 0.0f;
        }
        for (int i = i0; i < i1; ++i, par ^= 1) {
            float qn[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float* b = sh[par][c];
                b[threadIdx.x] = p[c][0];
                b[threadIdx.x + kThreads] = p[c][1];
                if (t.s2) b[threadIdx.x + 2 * kThreads] = p[c][2];
                qn[c] = __ldg(u + c * N + static_cast<size_t>(fd_wrap(i + 5, g.n1)) * g.n23 + t.col);
                if (i + 1 < i1) {
                    const float* plane = u + c * N + static_cast<size_t>(i + 1) * g.n23;
                    p[c][0] = __ldg(plane + t.soff[0]);
                    p[c][1] = __ldg(plane + t.soff[1]);
                    if (t.s2) p[c][2] = __ldg(plane + t.soff[2]);
                }
            }
            __syncthreads();
            // any value a lane reads here bounds the block's extrema; the warp takes lane 0's
            float flo = ordered_float(__shfl_sync(0xffffffffu, *static_cast<volatile int*>(&blo), 0)),
                  fhi = ordered_float(__shfl_sync(0xffffffffu, *static_cast<volatile int*>(&bhi), 0));
            float e[3][3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                e[c][0] = __fmul_rn(fd_queue_diff(q[c]), g.ih1);
                e[c][1] = __fmul_rn(fd_sh_diff<kFdCols>(sh[par][c] + own), g.ih2);
                e[c][2] = __fmul_rn(fd_sh_diff<1>(sh[par][c] + own), g.ih3);
                fd_queue_push(q[c], qn[c]);
            }
            float dlo, dhi;
            det_bounds(e, dlo, dhi);
            // dhi bounds lo from above, dlo bounds hi from below (finite ones only);
            // the bounds are raised by the plane's own points before it is tested
            const bool fin = t.ok && fabsf(dlo) < 3e38f && fabsf(dhi) < 3e38f;
            if (!__any_sync(0xffffffffu, t.ok && !(dlo > flo && dhi < fhi))) continue;  // also NaN
            flo = fminf(flo, ordered_float(__reduce_min_sync(0xffffffffu, fin ? ordered_int(dhi) : kOrderedInf)));
            fhi = fmaxf(fhi, ordered_float(__reduce_max_sync(0xffffffffu, fin ? ordered_int(dlo) : ~kOrderedInf)));
            if (lane == 0) {
                atomicMin(&blo, ordered_int(flo));
                atomicMax(&bhi, ordered_int(fhi));
            }
            if (t.ok && !(dlo > flo && dhi < fhi)) {
                const double d = det_exact(e);
                lo = min_nan(lo, d);  // a NaN propagates to both extrema
                hi = max_nan(hi, d);
            }
        }
    }
    grid_minmax(lo, hi, red);
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

// tiled gathers: cubic B-spline (order 4) only for FP32 fields
#define CLAIRE_TILED(order, EPI, fs, d, e)                                        \
    do {                                                                          \
        if ((order) == 3)                                                         \
            launch_tiled<3, EPI<SType>, SType>(g, fs, d, e, st, tb);              \
        else if ((order) == 1)                                                    \
            launch_tiled<1, EPI<SType>, SType>(g, fs, d, e, st, tb);              \
        else if constexpr (std::is_same<SType, float>::value)                     \
            launch_tiled<4, EPI<SType>, SType>(g, fs, d, e, st, tb);              \
    } while (0)

void launch_interp(const Grid& g, int order, const void* f, const float* d, void* out, Storage sto,
                   cudaStream_t st, const int4* tb)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        EpiStore<SType> e{static_cast<SType*>(out)};
        const SType* fs = static_cast<const SType*>(f);
        CLAIRE_TILED(order, EpiStore, fs, d, e);
    });
}

template <int ORDER, bool FULL, bool MAP>
void launch_fields_tiles(Grid g, const float* f, int nf, const float* d, float* out, cudaStream_t st)
{
    g.wide = 1;
    const size_t smem = tiled_smem_bytes<ORDER>(g);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_gather_tiled_fields<ORDER, FULL, MAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem));
    k_gather_tiled_fields<ORDER, FULL, MAP><<<tiled_grid(g), kTileThreads, smem, st>>>(g, f, nf, d, out);
}

template <int ORDER, bool MAP>
void launch_fields_as(const Grid& g, const float* f, int nf, const float* d, float* out, cudaStream_t st)
{
    if (tiles_cover_grid(g))
        launch_fields_tiles<ORDER, true, MAP>(g, f, nf, d, out, st);
    else
        launch_fields_tiles<ORDER, false, MAP>(g, f, nf, d, out, st);
}

void launch_interp_fields(const Grid& g, int order, const float* f, int nf, const float* d, float* out,
                          cudaStream_t st)
{
    if (order == 3)
        launch_fields_as<3, false>(g, f, nf, d, out, st);
    else if (order == 4)
        launch_fields_as<4, false>(g, f, nf, d, out, st);
    else
        launch_fields_as<1, false>(g, f, nf, d, out, st);
}

size_t tiled_grid_tiles(int n1, int n2, int n3)
{
    Grid g{};
    g.n1 = n1;
    g.n2 = n2;
    g.n3 = n3;
    const dim3 t = tiled_grid(g);
    return static_cast<size_t>(t.x) * t.y * t.z;
}

cudaError_t gather_fallback_tiles(unsigned long long* count, bool reset)
{
    cudaError_t e = cudaMemcpyFromSymbol(count, g_gather_global_tiles, sizeof(unsigned long long));
    if (e != cudaSuccess || !reset) return e;
    const unsigned long long z = 0;
    return cudaMemcpyToSymbol(g_gather_global_tiles, &z, sizeof(z));
}

void launch_backtrace(const Grid& g, int order, const float* v, const float* vc, float dt, int sign, float* d,
                      cudaStream_t st, int4* tb)
{
    const float* f = vc ? vc : v;
    const float sg = static_cast<float>(sign);
    if (order == 3)
        launch_backtrace_tiled<3>(g, v, f, dt, sg, d, tb, st);
    else if (order == 4)
        launch_backtrace_tiled<4>(g, v, f, dt, sg, d, tb, st);
    else
        launch_backtrace_tiled<1>(g, v, f, dt, sg, d, tb, st);
}

void launch_adj_step(const Grid& g, int order, const void* lam_next, const float* dA, const void* divv,
                     const void* divXp, float dt, void* lam, Storage sto, cudaStream_t st, const int4* tb)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        EpiAdjointOnly<SType> e{static_cast<const SType*>(divv), static_cast<const SType*>(divXp),
                                static_cast<SType*>(lam), dt};
        const SType* fs = static_cast<const SType*>(lam_next);
        CLAIRE_TILED(order, EpiAdjointOnly, fs, dA, e);
    });
}

void launch_inc_sources(const Grid& g, const float* vt, const void* gm, int nt, float coef0, void* q0,
                        void* F, Storage sto, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_inc_sources<SType><<<blocks_for(g.N), kThreads, 0, st>>>(
            g, vt, static_cast<const SType*>(gm), nt, coef0, static_cast<SType*>(q0), static_cast<SType*>(F));
    });
}

void launch_inc_sources_fd(const Grid& g, const float* vt, const void* m, int nt, float coef0, void* q0, void* F,
                           Storage sto, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_inc_sources_fd<SType><<<blocks_for(g.N), kThreads, 0, st>>>(
            g, vt, static_cast<const SType*>(m), nt, coef0, static_cast<SType*>(q0), static_cast<SType*>(F));
    });
}

void launch_body_fd(const Grid& g, const void* lam, const void* m, int nt, float w_end, float w_mid, int accumulate,
                    float* out, Storage sto, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_body_fd<SType><<<blocks_for(g.N), kThreads, 0, st>>>(g, static_cast<const SType*>(lam),
                                                              static_cast<const SType*>(m), nt, w_end, w_mid,
                                                              accumulate, out);
    });
}

void launch_body(const Grid& g, const void* lam, const void* gm, int nt, float w_end, float w_mid,
                 int accumulate, float* out, Storage sto, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_body<SType><<<blocks_for(g.N), kThreads, 0, st>>>(g, static_cast<const SType*>(lam),
                                                           static_cast<const SType*>(gm), nt, w_end, w_mid,
                                                           accumulate, out);
    });
}

void launch_inc_step_src(const Grid& g, int order, const void* q_prev, const float* d, const void* F,
                         float coef, void* q, Storage sto, cudaStream_t st, const int4* tb)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        EpiIncSource<SType> e{static_cast<const SType*>(F), static_cast<SType*>(q), coef};
        const SType* fs = static_cast<const SType*>(q_prev);
        CLAIRE_TILED(order, EpiIncSource, fs, d, e);
    });
}

void launch_inc_last_src(const Grid& g, int order, const void* q_prev, const float* d, const void* F,
                         float coef, void* lam, Storage sto, cudaStream_t st, const int4* tb)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        EpiIncSourceLast<SType> e{static_cast<const SType*>(F), static_cast<SType*>(lam), coef};
        const SType* fs = static_cast<const SType*>(q_prev);
        CLAIRE_TILED(order, EpiIncSourceLast, fs, d, e);
    });
}

void launch_inc_source0(const Grid& g, const float* vt, const void* gm, float coef0, void* q0, Storage sto,
                        cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_inc_source0<SType><<<blocks_for(g.N), kThreads, 0, st>>>(g, vt, static_cast<const SType*>(gm), coef0,
                                                                   static_cast<SType*>(q0));
    });
}

void launch_inc_step_grad(const Grid& g, int order, const void* q_prev, const float* d, const float* vt,
                          const void* gm, float coef, void* q, Storage sto, cudaStream_t st, const int4* tb)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        EpiIncGrad<SType> e{vt, static_cast<const SType*>(gm), static_cast<SType*>(q), coef, g.N};
        const SType* fs = static_cast<const SType*>(q_prev);
        CLAIRE_TILED(order, EpiIncGrad, fs, d, e);
    });
}

void launch_inc_last_grad(const Grid& g, int order, const void* q_prev, const float* d, const float* vt,
                          const void* gm, float coef, void* lam, Storage sto, cudaStream_t st, const int4* tb)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        EpiIncGradLast<SType> e{vt, static_cast<const SType*>(gm), static_cast<SType*>(lam), coef, g.N};
        const SType* fs = static_cast<const SType*>(q_prev);
        CLAIRE_TILED(order, EpiIncGradLast, fs, d, e);
    });
}

void launch_sub(const void* a, const void* b, void* out, size_t n, Storage sto, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_sub<SType><<<blocks_for(static_cast<uint32_t>(n)), kThreads, 0, st>>>(
            static_cast<const SType*>(a), static_cast<const SType*>(b), static_cast<SType*>(out),
            static_cast<uint32_t>(n));
    });
}

void launch_to_storage(const float* in, void* out, size_t n, Storage sto, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_convert<float, SType><<<blocks_for(static_cast<uint32_t>(n)), kThreads, 0, st>>>(
            in, static_cast<SType*>(out), static_cast<uint32_t>(n));
    });
}

void launch_from_storage(const void* in, float* out, size_t n, Storage sto, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_convert<SType, float><<<blocks_for(static_cast<uint32_t>(n)), kThreads, 0, st>>>(
            static_cast<const SType*>(in), out, static_cast<uint32_t>(n));
    });
}

void launch_map_step(const Grid& g, int order, const float* u_prev, const float* d, float* u,
                     cudaStream_t st)
{
    if (order == 3)
        launch_fields_as<3, true>(g, u_prev, 3, d, u, st);
    else if (order == 4)
        launch_fields_as<4, true>(g, u_prev, 3, d, u, st);
    else
        launch_fields_as<1, true>(g, u_prev, 3, d, u, st);
}

void launch_fd8_grad(const Grid& g, const void* f, void* out, Storage sto, cudaStream_t st)
{
    const int z = fd_zlen(g);
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_fd8_grad_tiled<SType><<<fd_grid(g, z), kThreads, 0, st>>>(g, static_cast<const SType*>(f),
                                                                    static_cast<SType*>(out), z);
    });
}

void launch_fd8_div(const Grid& g, const float* v, void* out, Storage sto, cudaStream_t st)
{
    const int z = fd_zlen(g);
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_fd8_div_tiled<SType><<<fd_grid(g, z), kThreads, 0, st>>>(g, v, static_cast<SType*>(out), z);
    });
}

void launch_detj_minmax(const Grid& g, const float* u, const Reduction& red, cudaStream_t st)
{
    const int z = fd_zlen(g);
    const dim3 cols = fd_grid(g, z);
    k_detj_minmax<<<red.nblocks, kThreads, 0, st>>>(g, u, z, static_cast<int>(cols.x * cols.y * cols.z), red);
}

}  // namespace claire
