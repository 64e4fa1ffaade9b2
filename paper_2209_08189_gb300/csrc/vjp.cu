// Reverse-mode derivative of the discrete semi-Lagrangian transport
// (discretise-then-differentiate) for sm_103a.
//
// Forward map (grid units, u = v / h, per node x): predictor y = x - dt u(x),
// U = I[u](y), displacement d = -dt/2 (u(x) + U), X = x + d,
// m^{j+1}(x) = I[m^j](X(x)), j = 0..nt-1 (Sec. 2.2: SL with RK2).
// Given gbar = dL/dm^{nt} the kernels below produce dL/dm^0 and dL/dv:
//   dbar_c  += mbar^{j+1} d_c I[m^j](X)        (interpolant gradient at X)
//   mbar^j   = W(X)^T mbar^{j+1}               (scatter transpose)
//   Ubar     = -dt/2 dbar,  ubar = -dt/2 dbar - dt sum_c Ubar_c grad I[u_c](y)
//              + W(y)^T Ubar                   (through the predictor)
//   vbar     = ubar / h.
// The scatter transposes accumulate 64-bit fixed-point integers, so their
// sums do not depend on the order of the atomic additions: the result is
// bitwise deterministic.
#include "internal.h"
#include "sl_tiled.cuh"

#include <climits>
#include <cmath>

namespace claire {

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(size_t n) { return static_cast<unsigned>((n + kThreads - 1) / kThreads); }

// 1-D basis and its t-derivative.
template <int ORDER>
__device__ __forceinline__ void basis_and_deriv(float t, float w[4], float dw[4])
{
    if constexpr (ORDER == 4) {
        bspline_weights(t, w);
        const float s = 1.0f - t;
        dw[0] = -0.5f * s * s;
        dw[1] = 1.5f * t * t - 2.0f * t;
        dw[2] = -1.5f * t * t + t + 0.5f;
        dw[3] = 0.5f * t * t;
    } else if constexpr (ORDER == 3) {
        cubic_weights(t, w);
        const float t2 = t * t;
        dw[0] = -(1.0f / 6.0f) * (3.0f * t2 - 6.0f * t + 2.0f);
        dw[1] = 0.5f * (3.0f * t2 - 4.0f * t - 1.0f);
        dw[2] = -0.5f * (3.0f * t2 - 2.0f * t - 2.0f);
        dw[3] = (1.0f / 6.0f) * (3.0f * t2 - 1.0f);
    } else {
        w[0] = 1.0f - t;
        w[1] = t;
        dw[0] = -1.0f;
        dw[1] = 1.0f;
    }
}

// Wrapped node offsets and weights (plus derivatives) of one axis.
template <int ORDER>
struct DAxis {
    static constexpr int M = Scheme<ORDER>::M;
    int idx[M];
    float w[4], dw[4];
    __device__ __forceinline__ void build(int node, float disp, int n, int stride)
    {
        float t;
        const int b = wrap_index(node + split_disp(disp, t) - Scheme<ORDER>::OFF, n);
#pragma unroll
        for (int a = 0; a < M; ++a) {
            const int q = b + a;
            idx[a] = (q >= n ? q - n : q) * stride;
        }
        basis_and_deriv<ORDER>(t, w, dw);
    }
};

// Gradient of the interpolant of f at node (i,j,k) + (d1,d2,d3), grid units.
template <int ORDER>
__device__ __forceinline__ void interp_gradient(const Grid& g, const float* __restrict__ f, int i, int j,
                                                int k, float d1, float d2, float d3, float grad[3])
{
    constexpr int M = DAxis<ORDER>::M;
    DAxis<ORDER> a1, a2, a3;
    a1.build(i, d1, g.n1, g.n23);
    a2.build(j, d2, g.n2, g.n3);
    a3.build(k, d3, g.n3, 1);
    float g0 = 0.f, g1 = 0.f, g2 = 0.f;
#pragma unroll
    for (int a = 0; a < M; ++a) {
        float s0 = 0.f, s1 = 0.f, s2 = 0.f;  // d1-weighted, plain for d2 and d3 paths
#pragma unroll
        for (int b = 0; b < M; ++b) {
            const float* row = f + a1.idx[a] + a2.idx[b];
            float r = 0.f, rd = 0.f;
#pragma unroll
            for (int c = 0; c < M; ++c) {
                const float fv = __ldg(row + a3.idx[c]);
                r = fmaf(a3.w[c], fv, r);
                rd = fmaf(a3.dw[c], fv, rd);
            }
            s0 = fmaf(a2.w[b], r, s0);
            s1 = fmaf(a2.dw[b], r, s1);
            s2 = fmaf(a2.w[b], rd, s2);
        }
        g0 = fmaf(a1.dw[a], s0, g0);
        g1 = fmaf(a1.w[a], s1, g1);
        g2 = fmaf(a1.w[a], s2, g2);
    }
    grad[0] = g0;
    grad[1] = g1;
    grad[2] = g2;
}

// interp_gradient out of line: the path of tiles whose box does not fit.
template <int ORDER>
__device__ __noinline__ float3 interp_gradient_global(const Grid g, const float* __restrict__ f, int i, int j, int k,
                                                      float d1, float d2, float d3)
{
    float gr[3];
    interp_gradient<ORDER>(g, f, i, j, k, d1, d2, d3, gr);
    return make_float3(gr[0], gr[1], gr[2]);
}

// Gradient of the interpolant from the tile's shared-memory box.  Each node
// is read once for the value and the derivative along x3, which one packed
// FMA per node accumulates together.
template <int ORDER>
__device__ __forceinline__ void tile_gradient(const float* box, const BoxPar& bp, int i, int j, int k, float d1,
                                              float d2, float d3, float grad[3])
{
    constexpr int M = Scheme<ORDER>::M;
    float t1, t2, t3, w1[4], w2[4], w3[4], dw1[4], dw2[4], dw3[4];
    const int o = tile_offset<ORDER>(bp, i, j, k, d1, d2, d3, t1, t2, t3);
    basis_and_deriv<ORDER>(t1, w1, dw1);
    basis_and_deriv<ORDER>(t2, w2, dw2);
    basis_and_deriv<ORDER>(t3, w3, dw3);
    const uint32_t base = smem_u32(box) + 4u * static_cast<uint32_t>(o);
    const uint32_t P4 = 4u * static_cast<uint32_t>(bp.E2 * bp.S3), S4 = 4u * static_cast<uint32_t>(bp.S3);
    float g0 = 0.0f, g1 = 0.0f, g2 = 0.0f;
#pragma unroll
    for (int a = 0; a < M; ++a) {
        float2 s = make_float2(0.0f, 0.0f);  // w2-weighted (value, x3 derivative)
        float s1 = 0.0f;                     // dw2-weighted value
#pragma unroll
        for (int b = 0; b < M; ++b) {
            const uint32_t row = base + a * P4 + b * S4;
            auto pair = [&](int c, float f, float2 acc) {
                return __ffma2_rn(make_float2(w3[c], dw3[c]), make_float2(f, f), acc);
            };
            float2 r = make_float2(0.0f, 0.0f);
            r = pair(0, lds_f32<0>(row), r);
            r = pair(1, lds_f32<4>(row), r);
            if constexpr (M == 4) {
                r = pair(2, lds_f32<8>(row), r);
                r = pair(3, lds_f32<12>(row), r);
            }
            s = __ffma2_rn(make_float2(w2[b], w2[b]), r, s);
            s1 = fmaf(dw2[b], r.x, s1);
        }
        g0 = fmaf(dw1[a], s.x, g0);
        g1 = fmaf(w1[a], s1, g1);
        g2 = fmaf(w1[a], s.y, g2);
    }
    grad[0] = g0;
    grad[1] = g1;
    grad[2] = g2;
}

// dbar_c(p) (+)= mbar(p) * d_c I[m](X(p)); FIRST: dbar is written, not added to.
//
// The 64 stencil values of a point come from the tile's shared-memory box, as
// in the gathers; bound: the shared-memory pipe (64 reads per point) beside 44 B
// per point of HBM traffic.  128^3, cubic: the per-point kernel it replaced,
// whose reads went through L1, took 71 us; this one 42 us.
template <int ORDER, bool FULL, bool FIRST>
__global__ void __launch_bounds__(kTileThreads, 3)
    k_grad_accum(Grid g, const float* __restrict__ m, const float* __restrict__ d, const float* __restrict__ mbar,
                 float* __restrict__ dbar)
{
    extern __shared__ float box[];
    __shared__ int red[6][TILE2];
    __shared__ int par[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * TILE3 + lane, j = blockIdx.y * TILE2 + warp, i0 = blockIdx.z * TILE1;
    const size_t N = g.N;
    const bool col_ok = FULL || (k < g.n3 && j < g.n2);
    const uint32_t p0 = static_cast<uint32_t>(i0) * g.n23 + j * g.n3 + k;
    auto valid = [&](int q) { return FULL || (col_ok && i0 + q < g.n1); };
    float d1[TILE1], d2[TILE1], d3[TILE1], mb[TILE1];
    int lo1 = INT_MAX, lo2 = INT_MAX, lo3 = INT_MAX, hi1 = INT_MIN, hi2 = INT_MIN, hi3 = INT_MIN;
    bool bad = false;
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        if (!valid(q)) continue;
        const uint32_t p = p0 + q * g.n23;
        d1[q] = __ldg(d + p);
        d2[q] = __ldg(d + N + p);
        d3[q] = __ldg(d + 2 * N + p);
        bounds_add(i0 + q, d1[q], lo1, hi1, bad);
        bounds_add(j, d2[q], lo2, hi2, bad);
        bounds_add(k, d3[q], lo3, hi3, bad);
    }
    const BoxPar bp = tile_box<ORDER, 4>(g, lo1, lo2, lo3, hi1, hi2, hi3, bad, red, par, lane, warp);
    const bool use_box = bp.E1 != 0;
    if (use_box) tile_load_box<float>(g, m, box, bp, lane, warp);
#pragma unroll
    for (int q = 0; q < TILE1; ++q)
        if (valid(q)) mb[q] = __ldg(mbar + p0 + q * g.n23);
    cp_async_wait_all();
    __syncthreads();
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        if (!valid(q)) continue;
        const uint32_t p = p0 + q * g.n23;
        float o[3] = {0.0f, 0.0f, 0.0f}, gr[3];
        if constexpr (!FIRST) {
#pragma unroll
            for (int c = 0; c < 3; ++c) o[c] = dbar[c * N + p];
        }
        if (use_box)
            tile_gradient<ORDER>(box, bp, i0 + q, j, k, d1[q], d2[q], d3[q], gr);
        else {
            const float3 t = interp_gradient_global<ORDER>(g, m, i0 + q, j, k, d1[q], d2[q], d3[q]);
            gr[0] = t.x; gr[1] = t.y; gr[2] = t.z;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) dbar[c * N + p] = fmaf(mb[q], gr[c], o[c]);
    }
}

// Fixed-point scale 2^(48 - e) with max|y| <= 2^e, so every scaled term
// stays below 2^48 in magnitude and a node can receive 2^14 full-size terms
// before the 64-bit sum could overflow.  kind 0: y = 0 (nothing to add);
// kind 2: max|y| is not finite (the maximum kernel maps NaN to infinity),
// every output is NaN.  The scale is applied as two FP32 factors up and down
// (2^(48-e) itself may lie outside the FP32 range): both are powers of two, so
// the products are exact.
struct FixedScale {
    int kind;
    float up0, up1;      // 2^(48 - e) = up0 up1
    float down0, down1;  // 2^(e - 48) = down0 down1
};

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }  // -126 <= e <= 127

__device__ __forceinline__ FixedScale fixed_scale_of(double mx)
{
    FixedScale s{0, 0.f, 0.f, 0.f, 0.f};
    const long long b = __double_as_longlong(mx) & 0x7fffffffffffffffll;
    if (b == 0) return s;
    if (b >= 0x7ff0000000000000ll) {
        s.kind = 2;
        return s;
    }
    // max|y| is an FP32 value held as a double, so normal: exponent field - 1022 is frexp's
    const int k = 48 - (static_cast<int>(b >> 52) - 1022);  // -80 .. 197
    s.kind = 1;
    const int h = k / 2;
    s.up0 = pow2f(h);
    s.up1 = pow2f(k - h);
    s.down0 = pow2f(-h);
    s.down1 = pow2f(h - k);
    return s;
}

// Displacement of point p (grid units): d if given, else the RK2 predictor -sdt v / h.
__device__ __forceinline__ void scatter_disp(const Grid& g, const float* __restrict__ d,
                                             const float* __restrict__ v, float sdt, uint32_t p, float& d1,
                                             float& d2, float& d3)
{
    const size_t N = g.N;
    if (d) {
        d1 = __ldg(d + p); d2 = __ldg(d + N + p); d3 = __ldg(d + 2 * N + p);
    } else {
        d1 = -sdt * __ldg(v + p) * g.ih1;
        d2 = -sdt * __ldg(v + N + p) * g.ih2;
        d3 = -sdt * __ldg(v + 2 * N + p) * g.ih3;
    }
}

// Fixed-point contribution of (scale y w_a w_b) w_c, |.| <= 2^48: the product p is
// formed in FP32 and rounded to the integer grid, so every term is a
// deterministic integer and the sums do not depend on their order.  64-bit
// conversions run on the FP64 pipe of this part (2 lanes per clock and SM, 64
// terms per point), so the integer is assembled from h ~ p 2^-27, |h| <= 2^21 + 1,
// read off the mantissa of (w_ab 2^-27) w_c + 1.5 2^23, and the remainder
// p - h 2^27, at most a little over 2^26 in magnitude, which FP32 holds
// exactly (a multiple of ulp(p)); h 2^27 is an even integer, so rounding the
// remainder rounds the sum the same way.
constexpr float kFixMagic = 12582912.0f;             // 1.5 2^23, bits 0x4b400000
constexpr float kFixDown = 7.450580596923828125e-9f;  // 2^-27

// The term as two words, its h biased by the magic's bits: term + kFixBias 2^32
// mod 2^64 (the bias 0x4b400000 2^27 has only a high word).  The carries are in PTX
// here and in add_high: written in C++ (64-bit sum, old + lo < old) the bits are the
// same and the reverse pass takes longer (128^3 2.23 ms against 2.16, 182 x 218 x 182
// 6.8 against 6.45).
constexpr unsigned kFixBias = 0x4b400000u >> 5;

struct FixedTerm {
    unsigned lo, hi;
};

__device__ __forceinline__ FixedTerm fixed_term_biased(float wab, float wab_down, float wc)
{
    const float p = wab * wc;
    const float x = fmaf(wab_down, wc, kFixMagic);
    const int r = __float2int_rn(fmaf(__fsub_rn(x, kFixMagic), -134217728.0f, p));
    FixedTerm t;
    asm("{\n .reg .u32 a, b, s;\n shl.b32 a, %2, 27;\n add.cc.u32 %0, a, %3;\n shr.u32 b, %2, 5;\n"
        " shr.s32 s, %3, 31;\n addc.u32 %1, b, s;\n}\n"
        : "=r"(t.lo), "=r"(t.hi)
        : "r"(__float_as_int(x)), "r"(r));
    return t;
}

__device__ __forceinline__ unsigned long long fixed_term(float wab, float wc)
{
    const FixedTerm t = fixed_term_biased(wab, wab * kFixDown, wc);
    return (static_cast<unsigned long long>(t.hi - kFixBias) << 32) | t.lo;
}

// 64-bit addition of a biased term into shared memory as two 32-bit additions:
// the low words first, whose returned old value tells the carry into the high
// word, then the high word less the bias.  (A 64-bit shared-memory atomic is a
// compare-and-swap loop on this part.)  The sum of all additions is exact
// whatever their order.
template <int BYTE_OFF>
__device__ __forceinline__ unsigned add_low(uint32_t lo, const FixedTerm& t)
{
    unsigned old;
    asm volatile("atom.shared.add.u32 %0, [%1+%2], %3;" : "=r"(old) : "r"(lo), "n"(BYTE_OFF), "r"(t.lo) : "memory");
    return old;
}
template <int BYTE_OFF>
__device__ __forceinline__ void add_high(uint32_t hi, const FixedTerm& t, unsigned old)
{
    asm volatile("{\n .reg .u32 a, b;\n add.cc.u32 a, %2, %3;\n addc.u32 b, %4, %5;\n red.shared.add.u32 [%0+%1], b;\n}\n"
                 ::"r"(hi), "n"(BYTE_OFF), "r"(old), "r"(t.lo), "r"(t.hi), "n"(0u - kFixBias) : "memory");
}

// Scatter-transpose tiles: a CTA owns a 4 x 8 x 32 tile of source points
// (256 threads, 4 points each along x1), like the gather tiles.  The
// destination stencils of the tile span a box that is accumulated in shared
// memory and flushed with one global atomic per touched node, instead of 64
// global atomics per point.  Boxes larger than kScatterCap nodes fall back to
// global atomics.  Integer sums do not depend on the order of additions, so
// either path gives the same bits.
//
// Bound: instruction issue (68 % of the slots, 112 M warp instructions at 128^3) beside
// the shared-memory data pipe (55 %: 128 atomics per point, 8.4 M warp
// instructions of 2.8 wavefronts).  128^3, cubic: 326 us with 64-bit conversions
// and 64-bit shared atomics, 139 us.
constexpr int kST1 = 4, kST2 = 8, kST3 = 32;
constexpr int kScatterCap = 6976;  // nodes of 8 B: four CTAs of 54.5 KB per SM

template <int ORDER>
__global__ void __launch_bounds__(kThreads, 4) k_scatter_tiled(Grid g, const float* __restrict__ yv,
                                                             const float* __restrict__ d,
                                                             const float* __restrict__ v, float sdt,
                                                             const double* __restrict__ maxabs,
                                                             unsigned long long* __restrict__ acc)
{
    extern __shared__ uint4 sbox4[];
    unsigned* slo = reinterpret_cast<unsigned*>(sbox4);  // low words, then the high words
    __shared__ int red[6][kST2];
    __shared__ int par[7];
    constexpr int M = DAxis<ORDER>::M;
    constexpr int OFF = Scheme<ORDER>::OFF;
    const FixedScale sc = fixed_scale_of(*maxabs);
    if (sc.kind != 1) return;  // uniform: zero or non-finite cotangent
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j = blockIdx.y * kST2 + warp, k = blockIdx.x * kST3 + lane, i0 = blockIdx.z * kST1;
    const bool col_ok = j < g.n2 && k < g.n3;
    float dd[kST1][3], yy[kST1];
    int lo1 = INT_MAX, lo2 = INT_MAX, lo3 = INT_MAX, hi1 = INT_MIN, hi2 = INT_MIN, hi3 = INT_MIN;
#pragma unroll
    for (int q = 0; q < kST1; ++q) {
        yy[q] = 0.0f;
        const int i = i0 + q;
        if (!(col_ok && i < g.n1)) continue;
        const uint32_t p = (static_cast<uint32_t>(i) * g.n2 + j) * g.n3 + k;
        yy[q] = __ldg(yv + p);
        if (yy[q] == 0.0f) continue;
        scatter_disp(g, d, v, sdt, p, dd[q][0], dd[q][1], dd[q][2]);
        float t;
        const int b1 = i + split_disp(dd[q][0], t) - OFF;
        const int b2 = j + split_disp(dd[q][1], t) - OFF;
        const int b3 = k + split_disp(dd[q][2], t) - OFF;
        lo1 = min(lo1, b1); hi1 = max(hi1, b1);
        lo2 = min(lo2, b2); hi2 = max(hi2, b2);
        lo3 = min(lo3, b3); hi3 = max(hi3, b3);
    }
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
    __syncthreads();
    if (threadIdx.x == 0) {
        int a[3] = {INT_MAX, INT_MAX, INT_MAX}, z[3] = {INT_MIN, INT_MIN, INT_MIN}, e[3];
        for (int w = 0; w < kST2; ++w)
            for (int c = 0; c < 3; ++c) {
                a[c] = min(a[c], red[c][w]);
                z[c] = max(z[c], red[3 + c][w]);
            }
        par[0] = a[0]; par[1] = a[1]; par[2] = a[2];
        if (a[0] > z[0]) {
            par[6] = 0;  // no non-zero point in the tile
        } else {
            par[6] = scatter_box_fits(a, z, M, kScatterCap, e) ? 1 : 2;
            par[3] = e[0]; par[4] = e[1]; par[5] = e[2];
        }
    }
    __syncthreads();
    const int mode = par[6];
    if (mode == 0) return;
    const int o1 = par[0], o2 = par[1], o3 = par[2];
    const int e1 = par[3], e2 = par[4], e3 = par[5];
    const int half = mode == 1 ? (e1 * e2 * e3 + 3) & ~3 : 0;  // words of the low half (16-byte multiples)
    unsigned* shi = slo + half;
    const uint32_t lo_s = smem_u32(slo), hi_off = 4u * static_cast<uint32_t>(half);
    if (mode == 1)
        for (int t = threadIdx.x; t < half / 2; t += kThreads) sbox4[t] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (mode == 2) {
#pragma unroll
        for (int q = 0; q < kST1; ++q) {
            if (yy[q] == 0.0f) continue;
            const float ys = sc.up1 * (sc.up0 * yy[q]);
            DAxis<ORDER> a1x, a2x, a3x;
            a1x.build(i0 + q, dd[q][0], g.n1, g.n23);
            a2x.build(j, dd[q][1], g.n2, g.n3);
            a3x.build(k, dd[q][2], g.n3, 1);
#pragma unroll 1
            for (int a = 0; a < M; ++a)
#pragma unroll
                for (int b = 0; b < M; ++b) {
                    const float wab = ys * (a1x.w[a] * a2x.w[b]);
                    const size_t row = static_cast<size_t>(a1x.idx[a]) + a2x.idx[b];
#pragma unroll
                    for (int c = 0; c < M; ++c)
                        atomicAdd(acc + row + a3x.idx[c],
                                  fixed_term(wab, a3x.w[c]));
                }
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < kST1; ++q) {
        if (yy[q] == 0.0f) continue;
        const float ys = sc.up1 * (sc.up0 * yy[q]);
        // box-relative stencil: unwrapped first node minus the box origin
        float t1, t2, t3;
        const int r1 = i0 + q + split_disp(dd[q][0], t1) - OFF - o1;
        const int r2 = j + split_disp(dd[q][1], t2) - OFF - o2;
        const int r3 = k + split_disp(dd[q][2], t3) - OFF - o3;
        float w1[4], w2[4], w3[4];
        scheme_weights<ORDER>(t1, w1);
        scheme_weights<ORDER>(t2, w2);
        scheme_weights<ORDER>(t3, w3);
        const int first = (r1 * e2 + r2) * e3 + r3;
#pragma unroll
        for (int a = 0; a < M; ++a)
#pragma unroll
            for (int b = 0; b < M; ++b) {
                const float wab = ys * (w1[a] * w2[b]), wd = wab * kFixDown;
                const uint32_t lo = lo_s + 4u * static_cast<uint32_t>(first + (a * e2 + b) * e3);
                const uint32_t hi = lo + hi_off;
                FixedTerm t[M];
                unsigned old[M];
#pragma unroll
                for (int c = 0; c < M; ++c) t[c] = fixed_term_biased(wab, wd, w3[c]);
                old[0] = add_low<0>(lo, t[0]);
                old[1] = add_low<4>(lo, t[1]);
                if constexpr (M == 4) {
                    old[2] = add_low<8>(lo, t[2]);
                    old[3] = add_low<12>(lo, t[3]);
                }
                add_high<0>(hi, t[0], old[0]);
                add_high<4>(hi, t[1], old[1]);
                if constexpr (M == 4) {
                    add_high<8>(hi, t[2], old[2]);
                    add_high<12>(hi, t[3], old[3]);
                }
            }
    }
    __syncthreads();
    // flush by rows: a warp per (c1, c2), its lanes along x3
    const int rows = e1 * e2;
    for (int r = warp; r < rows; r += kThreads / 32) {
        const int c1 = r / e2, c2 = r - c1 * e2;
        const size_t base = (static_cast<size_t>(wrap_index(o1 + c1, g.n1)) * g.n2 + wrap_index(o2 + c2, g.n2)) * g.n3;
        for (int c3 = lane; c3 < e3; c3 += 32) {
            const int t = r * e3 + c3;
            const unsigned long long val = (static_cast<unsigned long long>(shi[t]) << 32) | slo[t];
            if (val) atomicAdd(acc + base + wrap_index(o3 + c3, g.n3), val);
        }
    }
}

// The 64-bit integer a as (f1 + f2 + f3) 2^e, exactly: f1 its leading 24 bits, f2 the
// next 24, f3 the last 16.  (The 64-bit conversion instructions run on the
// FP64 pipe, at some 300 cycles per warp and SM: at 128^3 they alone were 60 us
// of the 69 us of this kernel.)
__device__ __forceinline__ void ll_split(long long a, float& f1, float& f2, float& f3, int& e)
{
    const unsigned long long m = static_cast<unsigned long long>(a < 0 ? -a : a);
    if (m == 0) {
        f1 = f2 = f3 = 0.0f;
        e = 0;
        return;
    }
    const int z = __clzll(static_cast<long long>(m));
    const unsigned long long n = m << z;  // top bit set
    f1 = static_cast<float>(static_cast<unsigned>(n >> 40));
    f2 = static_cast<float>(static_cast<unsigned>(n >> 16) & 0xffffffu) * 5.9604644775390625e-8f;  // 2^-24
    f3 = static_cast<float>(static_cast<unsigned>(n) & 0xffffu) * 9.094947017729282379e-13f;       // 2^-40
    if (a < 0) {
        f1 = -f1;
        f2 = -f2;
        f3 = -f3;
    }
    e = 40 - z;
}

// a + b as s + r, exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& r)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    r = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// out = mult ((accumulate ? out : 0) + acc / scale); acc is cleared for reuse.
// Bound: HBM (20 B per point, 24 when accumulating).  The scaling is by powers of
// two, and the sum with out carries its rounding errors (two-sums), so the 64
// bits enter it whole; it is rounded to FP32, then the product with mult.  Four
// points per thread when the arrays are 16-byte aligned.  128^3: 10 us; 81 us
// with 64-bit conversions and FP64 sums.
__device__ __forceinline__ float fixed_value(long long a, const FixedScale& s, int accumulate, float mult, float old)
{
    if (s.kind == 2) return __int_as_float(0x7fffffff);  // non-finite cotangent: propagate NaN
    float f1, f2, f3;
    int e;
    ll_split(a, f1, f2, f3, e);
    const float pe = pow2f(e);  // -23 <= e <= 40
    f1 = s.down1 * (s.down0 * (f1 * pe));
    f2 = s.down1 * (s.down0 * (f2 * pe));
    f3 = s.down1 * (s.down0 * (f3 * pe));
    if (!accumulate) return mult * (f1 + (f2 + f3));
    float t, u, v, w, hi, lo;
    two_sum(old, f1, t, u);
    if (!(fabsf(t) < INFINITY)) return mult * t;  // the error terms would make a NaN of an infinity
    two_sum(u, f2, v, w);
    two_sum(t, v, hi, lo);
    if (!(fabsf(hi) < INFINITY)) return mult * hi;
    return mult * __fadd_rn(hi, __fadd_rn(lo, __fadd_rn(w, f3)));
}

__global__ void __launch_bounds__(kThreads) k_fixed_to_float(unsigned long long* __restrict__ acc,
                                                              const double* __restrict__ maxabs,
                                                              int accumulate, float mult,
                                                              float* __restrict__ out, size_t n)
{
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    const size_t t0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x;
    const FixedScale s = fixed_scale_of(*maxabs);
    size_t done = 0;
    if (((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(acc)) & 15u) == 0) {
        ulonglong2* a2 = reinterpret_cast<ulonglong2*>(acc);
        float4* o4 = reinterpret_cast<float4*>(out);
        const size_t n4 = n / 4;
        for (size_t i = t0; i < n4; i += stride) {
            const ulonglong2 u = a2[2 * i], w = a2[2 * i + 1];
            float4 o = accumulate ? o4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            a2[2 * i] = make_ulonglong2(0ull, 0ull);
            a2[2 * i + 1] = make_ulonglong2(0ull, 0ull);
            o.x = fixed_value(static_cast<long long>(u.x), s, accumulate, mult, o.x);
            o.y = fixed_value(static_cast<long long>(u.y), s, accumulate, mult, o.y);
            o.z = fixed_value(static_cast<long long>(w.x), s, accumulate, mult, o.z);
            o.w = fixed_value(static_cast<long long>(w.y), s, accumulate, mult, o.w);
            o4[i] = o;
        }
        done = 4 * n4;
    }
    for (size_t i = done + t0; i < n; i += stride) {
        const long long a = static_cast<long long>(acc[i]);
        acc[i] = 0ull;
        out[i] = fixed_value(a, s, accumulate, mult, accumulate ? out[i] : 0.0f);
    }
}

// Predictor terms: Ubar = -dt/2 dbar; ubar(x) = -dt/2 dbar(x) - dt sum_c Ubar_c grad I[u_c](y)
// with y = x - dt u(x); writes ubar (grid units) and Ubar.
// vc: the field the predictor interpolates (v itself, or its cubic B-spline
// coefficients); v gives the predictor displacement at the node.
// One tile box per component, staged in turn, as in the backtrace: the
// predictor points of a tile share its bounds (128^3: 130 -> 107 us).
template <int ORDER, bool FULL>
__global__ void __launch_bounds__(kTileThreads, 3)
    k_predictor_terms(Grid g, const float* __restrict__ v, const float* __restrict__ vc, float dt,
                      const float* __restrict__ dbar, float* __restrict__ ubar, float* __restrict__ Ubar)
{
    extern __shared__ float box[];
    __shared__ int red[6][TILE2];
    __shared__ int par[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * TILE3 + lane, j = blockIdx.y * TILE2 + warp, i0 = blockIdx.z * TILE1;
    const size_t N = g.N;
    const bool col_ok = FULL || (k < g.n3 && j < g.n2);
    const uint32_t p0 = static_cast<uint32_t>(i0) * g.n23 + j * g.n3 + k;
    auto valid = [&](int q) { return FULL || (col_ok && i0 + q < g.n1); };
    float e1[TILE1], e2[TILE1], e3[TILE1], yb[TILE1][3];
    int lo1 = INT_MAX, lo2 = INT_MAX, lo3 = INT_MAX, hi1 = INT_MIN, hi2 = INT_MIN, hi3 = INT_MIN;
    bool bad = false;
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        yb[q][0] = yb[q][1] = yb[q][2] = 0.0f;
        if (!valid(q)) continue;
        const uint32_t p = p0 + q * g.n23;
        e1[q] = -dt * __ldg(v + p) * g.ih1;
        e2[q] = -dt * __ldg(v + N + p) * g.ih2;
        e3[q] = -dt * __ldg(v + 2 * N + p) * g.ih3;
        bounds_add(i0 + q, e1[q], lo1, hi1, bad);
        bounds_add(j, e2[q], lo2, hi2, bad);
        bounds_add(k, e3[q], lo3, hi3, bad);
    }
    const BoxPar bp = tile_box<ORDER, 4>(g, lo1, lo2, lo3, hi1, hi2, hi3, bad, red, par, lane, warp);
    const bool use_box = bp.E1 != 0;
    for (int c = 0; c < 3; ++c) {
        // weights are formed anew per component (kept, they spill)
#pragma unroll
        for (int q = 0; q < TILE1; ++q) asm volatile("" : "+f"(e1[q]), "+f"(e2[q]), "+f"(e3[q]));
        if (use_box) {
            tile_load_box<float>(g, vc + c * N, box, bp, lane, warp);
            cp_async_wait_all();
            __syncthreads();
        }
        const float ih = c == 0 ? g.ih1 : (c == 1 ? g.ih2 : g.ih3);
#pragma unroll
        for (int q = 0; q < TILE1; ++q) {
            if (!valid(q)) continue;
            const uint32_t p = p0 + q * g.n23;
            const float Ub = -0.5f * dt * __ldg(dbar + c * N + p);
            float gr[3];  // gradient of v_c; u_c = v_c ih_c
            if (use_box)
                tile_gradient<ORDER>(box, bp, i0 + q, j, k, e1[q], e2[q], e3[q], gr);
            else {
                const float3 t = interp_gradient_global<ORDER>(g, vc + c * N, i0 + q, j, k, e1[q], e2[q], e3[q]);
                gr[0] = t.x; gr[1] = t.y; gr[2] = t.z;
            }
#pragma unroll
            for (int e = 0; e < 3; ++e) yb[q][e] = fmaf(Ub * ih, gr[e], yb[q][e]);
            Ubar[c * N + p] = Ub;
        }
        if (use_box) __syncthreads();  // every read of this component is done before the next staging
    }
#pragma unroll
    for (int q = 0; q < TILE1; ++q) {
        if (!valid(q)) continue;
        const uint32_t p = p0 + q * g.n23;
#pragma unroll
        for (int c = 0; c < 3; ++c) ubar[c * N + p] = -0.5f * dt * __ldg(dbar + c * N + p) - dt * yb[q][c];
    }
}

// y = a (y + x): the unit factor that k_fixed_to_float applies when it
// accumulates, for a term added after a prefilter.
__global__ void __launch_bounds__(kThreads) k_scale_add(float* __restrict__ y, float a, const float* __restrict__ x,
                                                         size_t n)
{
    const size_t p = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x;
    if (p < n) y[p] = a * (y[p] + x[p]);
}

// max |x| over n values (as a double).  The
// maximum is taken on the FP32 bit patterns, which order like the magnitudes;
// NaN becomes infinity, which the reductions keep.
__global__ void __launch_bounds__(kThreads) k_maxabs(const float* __restrict__ x, size_t n, Reduction red)
{
    unsigned hi = 0;
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    const size_t t0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x;
    size_t done = 0;
    if ((reinterpret_cast<uintptr_t>(x) & 15u) == 0) {
        const uint4* x4 = reinterpret_cast<const uint4*>(x);
        const size_t n4 = n / 4;
        for (size_t i = t0; i < n4; i += stride) {
            const uint4 u = __ldg(x4 + i);
            hi = max(hi, max(max(u.x & 0x7fffffffu, u.y & 0x7fffffffu), max(u.z & 0x7fffffffu, u.w & 0x7fffffffu)));
        }
        done = 4 * n4;
    }
    for (size_t i = done + t0; i < n; i += stride) hi = max(hi, __float_as_uint(x[i]) & 0x7fffffffu);
    const double m = __uint_as_float(min(hi, 0x7f800000u));
    grid_max_bits(static_cast<unsigned long long>(__double_as_longlong(m)), red);
}

}  // namespace

template <int ORDER, bool FULL>
void launch_grad_accum_as(const Grid& g, const float* m, const float* d, const float* mbar, float* dbar, bool first,
                          cudaStream_t st)
{
    if (first)
        k_grad_accum<ORDER, FULL, true><<<tiled_grid(g), kTileThreads, tiled_smem_bytes<ORDER>(g), st>>>(g, m, d, mbar, dbar);
    else
        k_grad_accum<ORDER, FULL, false><<<tiled_grid(g), kTileThreads, tiled_smem_bytes<ORDER>(g), st>>>(g, m, d, mbar, dbar);
}

static_assert(kBoxCapFloats * sizeof(float) <= 48 * 1024, "the kernels of this file launch with the default shared-memory limit");

void launch_grad_accum(const Grid& g, int order, const float* m, const float* d, const float* mbar, float* dbar,
                       bool first, cudaStream_t st)
{
    const bool full = tiles_cover_grid(g);
    if (order == 3)
        full ? launch_grad_accum_as<3, true>(g, m, d, mbar, dbar, first, st)
             : launch_grad_accum_as<3, false>(g, m, d, mbar, dbar, first, st);
    else if (order == 4)
        full ? launch_grad_accum_as<4, true>(g, m, d, mbar, dbar, first, st)
             : launch_grad_accum_as<4, false>(g, m, d, mbar, dbar, first, st);
    else
        full ? launch_grad_accum_as<1, true>(g, m, d, mbar, dbar, first, st)
             : launch_grad_accum_as<1, false>(g, m, d, mbar, dbar, first, st);
}

template <int ORDER>
cudaError_t launch_scatter_as(const Grid& g, const float* yv, const float* d, const float* v, float sdt,
                              const double* maxabs, unsigned long long* acc, cudaStream_t st)
{
    const dim3 grid((g.n3 + kST3 - 1) / kST3, (g.n2 + kST2 - 1) / kST2, (g.n1 + kST1 - 1) / kST1);
    const int smem = kScatterCap * static_cast<int>(sizeof(unsigned long long));
    const cudaError_t e =
        cudaFuncSetAttribute(k_scatter_tiled<ORDER>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_scatter_tiled<ORDER><<<grid, kThreads, smem, st>>>(g, yv, d, v, sdt, maxabs, acc);
    return cudaSuccess;
}

cudaError_t launch_scatter_fixed(const Grid& g, int order, const float* yv, const float* d, const float* v, float sdt,
                                 const double* maxabs, unsigned long long* acc, cudaStream_t st)
{
    if (order == 3) return launch_scatter_as<3>(g, yv, d, v, sdt, maxabs, acc, st);
    if (order == 4) return launch_scatter_as<4>(g, yv, d, v, sdt, maxabs, acc, st);
    return launch_scatter_as<1>(g, yv, d, v, sdt, maxabs, acc, st);
}

void launch_fixed_to_float(unsigned long long* acc, const double* maxabs, int accumulate, float mult, float* out,
                           size_t n, cudaStream_t st)
{
    const unsigned blocks = blocks_for((n + 3) / 4);
    k_fixed_to_float<<<blocks < 152 * 16 ? blocks : 152 * 16, kThreads, 0, st>>>(acc, maxabs, accumulate, mult, out, n);
}

template <int ORDER>
void launch_predictor_as(const Grid& g, const float* v, const float* vc, float dt, const float* dbar, float* ubar,
                         float* Ubar, cudaStream_t st)
{
    if (tiles_cover_grid(g))
        k_predictor_terms<ORDER, true><<<tiled_grid(g), kTileThreads, tiled_smem_bytes<ORDER>(g), st>>>(g, v, vc, dt, dbar, ubar,
                                                                                             Ubar);
    else
        k_predictor_terms<ORDER, false><<<tiled_grid(g), kTileThreads, tiled_smem_bytes<ORDER>(g), st>>>(g, v, vc, dt, dbar, ubar,
                                                                                              Ubar);
}

void launch_predictor_terms(const Grid& g, int order, const float* v, const float* vc, float dt, const float* dbar,
                            float* ubar, float* Ubar, cudaStream_t st)
{
    if (order == 3)
        launch_predictor_as<3>(g, v, vc, dt, dbar, ubar, Ubar, st);
    else if (order == 4)
        launch_predictor_as<4>(g, v, vc, dt, dbar, ubar, Ubar, st);
    else
        launch_predictor_as<1>(g, v, vc, dt, dbar, ubar, Ubar, st);
}

void launch_scale_add(float* y, float a, const float* x, size_t n, cudaStream_t st)
{
    k_scale_add<<<blocks_for(n), kThreads, 0, st>>>(y, a, x, n);
}

void launch_maxabs(const float* x, size_t n, const Reduction& red, cudaStream_t st)
{
    k_maxabs<<<red.nblocks, kThreads, 0, st>>>(x, n, red);
}

}  // namespace claire
