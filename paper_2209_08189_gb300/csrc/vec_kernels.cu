// Spectral scaling, FP64 reductions and vector updates of libclaire (sm_103a).
// The spectral kernel applies the per-wavenumber 3x3 symbols of the
// regularisation operator, its inverse (the PCG preconditioner) and the
// paper's K operator in one pass over the three half-spectra (Sec. 2.2:
// "two FFTs and one Hadamard product"); cuFFT does the transforms.
#include "internal.h"

namespace claire {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float2 cmul(float s, float2 z) { return make_float2(s * z.x, s * z.y); }

// Per-mode pieces of the symbol S(k) = a I + c u u^T on the half spectrum:
// a = beta_v |k|^2 (H1) or beta_v |k|^4 (H2), c = beta_w (1 + |k|^2), u = k
// with Nyquist components set to zero; wt = multiplicity of the mode in the
// full spectrum (1 on the x3 = 0 and Nyquist planes, else 2).
struct Mode {
    float u1, u2, u3, a, c, kk, wt;
};

// idx: index of the mode on the half spectrum (below 2^31: 32-bit divisions).
__device__ __forceinline__ Mode mode_of(const Grid& g, uint32_t idx, int n3h, const RegParams& rp)
{
    Mode m;
    const uint32_t r = idx / static_cast<uint32_t>(n3h);
    const int k3i = static_cast<int>(idx - r * static_cast<uint32_t>(n3h));
    const int i = static_cast<int>(r / static_cast<uint32_t>(g.n2));
    const int j = static_cast<int>(r) - i * g.n2;
    const float k1 = static_cast<float>(i <= g.n1 / 2 ? i : i - g.n1);
    const float k2 = static_cast<float>(j <= g.n2 / 2 ? j : j - g.n2);
    const float k3 = static_cast<float>(k3i);
    m.kk = k1 * k1 + k2 * k2 + k3 * k3;
    m.u1 = (2 * i == g.n1) ? 0.0f : k1;
    m.u2 = (2 * j == g.n2) ? 0.0f : k2;
    m.u3 = (2 * k3i == g.n3) ? 0.0f : k3;
    m.a = rp.beta_v * (rp.reg == 2 ? m.kk * m.kk : m.kk);
    m.c = rp.beta_w * (1.0f + m.kk);
    m.wt = (k3i == 0 || 2 * k3i == g.n3) ? 1.0f : 2.0f;
    return m;
}

// The symbols of one mode.  Their roundings are written out: H p~ and the
// preconditioned residual are formed in one kernel for their inner products and again
// in the next for the update, and the recurrences need the same bits of both; the
// compiler may fuse products differently from kernel to kernel.  The two-level
// preconditioner's error against 64 bits is then that of recurrences that store
// both: 1.01 times in the geometric mean of 144 inputs at 256^3 (0.25 to 4.1 on
// single ones: roundoff in a few low modes decides it), 0.99 to 1.00 at 128^3 and
// 96 x 112 x 80, 64 inputs each.

// u . x
__device__ __forceinline__ float2 mode_div(const Mode& m, float2 x0, float2 x1, float2 x2)
{
    return make_float2(fmaf(m.u3, x2.x, fmaf(m.u2, x1.x, __fmul_rn(m.u1, x0.x))),
                       fmaf(m.u3, x2.y, fmaf(m.u2, x1.y, __fmul_rn(m.u1, x0.y))));
}

// x + f u ud
__device__ __forceinline__ float2 mode_add(float f, float u, float2 ud, float2 x)
{
    const float fu = __fmul_rn(f, u);
    return make_float2(fmaf(fu, ud.x, x.x), fmaf(fu, ud.y, x.y));
}

__device__ __forceinline__ float2 mode_mul(float a, float2 x) { return make_float2(__fmul_rn(a, x.x), __fmul_rn(a, x.y)); }

__device__ __forceinline__ float2 mode_axpy(float a, float2 x, float2 y)
{
    return make_float2(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y));
}

// -c / (a + c |u|^2)
__device__ __forceinline__ float mode_leray(const Mode& m)
{
    const float uu = fmaf(m.u3, m.u3, fmaf(m.u2, m.u2, __fmul_rn(m.u1, m.u1)));
    return -__fdiv_rn(m.c, fmaf(m.c, uu, m.a));
}

// y = S x for one mode
__device__ __forceinline__ void apply_S(const Mode& m, float2 x0, float2 x1, float2 x2, float2& y0,
                                        float2& y1, float2& y2)
{
    const float2 ud = mode_div(m, x0, x1, x2);
    y0 = mode_axpy(m.a, x0, mode_mul(__fmul_rn(m.c, m.u1), ud));
    y1 = mode_axpy(m.a, x1, mode_mul(__fmul_rn(m.c, m.u2), ud));
    y2 = mode_axpy(m.a, x2, mode_mul(__fmul_rn(m.c, m.u3), ud));
}

// y = S^{-1} x (op SPEC_INV) or (a I)^{-1} x (op SPEC_AINV); identity at k = 0
__device__ __forceinline__ void apply_inv(const Mode& m, int op, float2 x0, float2 x1, float2 x2,
                                          float2& y0, float2& y1, float2& y2)
{
    if (m.kk == 0.0f) {
        y0 = x0; y1 = x1; y2 = x2;
        return;
    }
    const float ia = __fdiv_rn(1.0f, m.a);
    if (op == SPEC_AINV) {
        y0 = mode_mul(ia, x0); y1 = mode_mul(ia, x1); y2 = mode_mul(ia, x2);
        return;
    }
    const float2 ud = mode_div(m, x0, x1, x2);
    const float f = mode_leray(m);
    y0 = mode_mul(ia, mode_add(f, m.u1, ud, x0));
    y1 = mode_mul(ia, mode_add(f, m.u2, ud, x1));
    y2 = mode_mul(ia, mode_add(f, m.u3, ud, x2));
}

// y = M x for one mode and any of the operators.
__device__ __forceinline__ void apply_op(const Mode& m, int op, float2 x0, float2 x1, float2 x2, float2& y0,
                                         float2& y1, float2& y2)
{
    if (op == SPEC_REG) {
        apply_S(m, x0, x1, x2, y0, y1, y2);
    } else if (op != SPEC_K) {
        apply_inv(m, op, x0, x1, x2, y0, y1, y2);
    } else if (m.kk == 0.0f) {
        y0 = x0; y1 = x1; y2 = x2;
    } else {
        // K = I - c u u^T / (a + c |u|^2);  S^{-1} = K / a  (Sherman-Morrison)
        const float2 ud = mode_div(m, x0, x1, x2);
        const float f = mode_leray(m);
        y0 = mode_add(f, m.u1, ud, x0);
        y1 = mode_add(f, m.u2, ud, x1);
        y2 = mode_add(f, m.u3, ud, x2);
    }
}

// One mode of a vector's three half-spectra.  An in-place kernel loads all three
// before its first store: a load behind a store to the same array waits for it
// (the compiler cannot tell that their components differ).  256^3: 119 -> 112 us
// per direction; a registration of ten PCG iterations 43.85 -> 43.72 ms.
__device__ __forceinline__ void load3(const float2* a, size_t cs, uint32_t idx, float2 (&out)[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = a[c * cs + idx];
}

// PCG direction in Fourier space: z~ = M r~ (recomputed from r~, not
// stored), p~ = z~ + beta p~ (p~ = z~ when first), copied to cp for the
// inverse FFT that yields p (it overwrites its input).
__global__ void __launch_bounds__(kThreads) k_spectral_direction(Grid g, const float2* __restrict__ rh,
                                                                  float2* __restrict__ ph,
                                                                  float2* __restrict__ cp, size_t cs,
                                                                  const double* __restrict__ sc, int first, int op,
                                                                  RegParams rp)
{
    const float beta = first ? 0.0f : static_cast<float>(sc[kPcgBeta]);
    const int n3h = g.n3 / 2 + 1;
    const uint32_t M = static_cast<uint32_t>(g.n1) * g.n2 * n3h;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        const Mode m = mode_of(g, idx, n3h, rp);
        float2 z[3], o[3] = {};
        if (!first) load3(ph, cs, idx, o);
        apply_inv(m, op, rh[idx], rh[cs + idx], rh[2 * cs + idx], z[0], z[1], z[2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 p = z[c];
            if (!first) p = make_float2(fmaf(beta, o[c].x, z[c].x), fmaf(beta, o[c].y, z[c].y));
            ph[c * cs + idx] = p;
            cp[c * cs + idx] = p;
        }
    }
}

// ---- PCG carried entirely in Fourier space ----
// Vectors are scaled half-spectra u~ = F[u] / N, so that the unnormalised
// inverse FFT returns u and sum_x u(x) w(x) = N sum_k wt Re(conj(u~) w~)
// (Parseval on the half spectrum; wt = multiplicity of the mode).

// Grid-wide sums of a and b (grid_sums).
__device__ __forceinline__ bool grid_sum2(double a, double b, const Reduction& r, double (&tot)[2])
{
    const double v[2] = {a, b};
    return grid_sums<2>(v, r, tot);
}

__device__ __forceinline__ float cdot3(float2 a0, float2 a1, float2 a2, float2 b0, float2 b1, float2 b2)
{
    return a0.x * b0.x + a0.y * b0.y + a1.x * b1.x + a1.y * b1.y + a2.x * b2.x + a2.y * b2.y;
}

// yh = scale * M(k) xh for the three half-spectra (in place when yh = xh); with
// ENERGY also the total of sum_k wt Re(conj(xh) M xh), the quadratic form of
// the operator (Parseval), so that no pass over the physical fields forms it.
template <bool ENERGY>
__global__ void __launch_bounds__(kThreads) k_spectral(Grid g, const float2* xh, float2* yh, size_t cs, int op,
                                                        RegParams rp, float scale, Reduction red)
{
    const int n3h = g.n3 / 2 + 1;
    const uint32_t M = static_cast<uint32_t>(g.n1) * g.n2 * n3h;
    double acc = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        const Mode m = mode_of(g, idx, n3h, rp);
        const float2 x0 = xh[idx], x1 = xh[cs + idx], x2 = xh[2 * cs + idx];
        float2 y0, y1, y2;
        apply_op(m, op, x0, x1, x2, y0, y1, y2);
        yh[idx] = cmul(scale, y0);
        yh[cs + idx] = cmul(scale, y1);
        yh[2 * cs + idx] = cmul(scale, y2);
        if constexpr (ENERGY) acc += static_cast<double>(m.wt * cdot3(x0, x1, x2, y0, y1, y2));
    }
    if constexpr (ENERGY) grid_sum(acc, red);
}

// Total of sum_k wt Re(conj(w) S w) for w = vh + alpha xh (xh may be null): the
// regularisation energy of a trial velocity from the spectra the solver
// carries, without transforming it.
__global__ void __launch_bounds__(kThreads) k_reg_energy(Grid g, const float2* __restrict__ vh,
                                                          const float2* __restrict__ xh, size_t cs, float alpha,
                                                          RegParams rp, Reduction red)
{
    const int n3h = g.n3 / 2 + 1;
    const uint32_t M = static_cast<uint32_t>(g.n1) * g.n2 * n3h;
    double acc = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        float2 w[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            w[c] = vh[c * cs + idx];
            if (xh) {
                const float2 x = xh[c * cs + idx];
                w[c] = make_float2(fmaf(alpha, x.x, w[c].x), fmaf(alpha, x.y, w[c].y));
            }
        }
        const Mode m = mode_of(g, idx, n3h, rp);
        float2 y0, y1, y2;
        apply_S(m, w[0], w[1], w[2], y0, y1, y2);
        acc += static_cast<double>(m.wt * cdot3(w[0], w[1], w[2], y0, y1, y2));
    }
    grid_sum(acc, red);
}

// Start: r~ = -scale g^ (spec holds F[g]), x~ = 0; partials of |r~|^2 and
// <r~, z~> with z~ = M r~ (recomputed by the direction kernel).
__global__ void __launch_bounds__(kThreads) k_fs_start(Grid g, float2* __restrict__ spec,
                                                        float2* __restrict__ rh, float2* __restrict__ xh,
                                                        size_t cs, int op, RegParams rp, float scale,
                                                        double* __restrict__ sc, Reduction red)
{
    const int n3h = g.n3 / 2 + 1;
    const uint32_t M = static_cast<uint32_t>(g.n1) * g.n2 * n3h;
    double arr = 0.0, arz = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        const Mode m = mode_of(g, idx, n3h, rp);
        const float2 r0 = cmul(-scale, spec[idx]), r1 = cmul(-scale, spec[cs + idx]),
                     r2 = cmul(-scale, spec[2 * cs + idx]);
        float2 z0, z1, z2;
        apply_inv(m, op, r0, r1, r2, z0, z1, z2);
        rh[idx] = r0; rh[cs + idx] = r1; rh[2 * cs + idx] = r2;
        xh[idx] = make_float2(0.f, 0.f); xh[cs + idx] = make_float2(0.f, 0.f); xh[2 * cs + idx] = make_float2(0.f, 0.f);
        arr += static_cast<double>(m.wt * cdot3(r0, r1, r2, r0, r1, r2));
        arz += static_cast<double>(m.wt * cdot3(r0, r1, r2, z0, z1, z2));
    }
    double tot[2];
    if (grid_sum2(arr, arz, red, tot)) sc[kPcgRz] = tot[1];
}

// h = S p~ + scale F[body] (T holds F[body]), or K of that for the paper's
// gradient form: one mode of H p~.
__device__ __forceinline__ void hp_mode(const Mode& m, const float2 p[3], const float2* __restrict__ T, size_t cs,
                                        uint32_t idx, int kform, float scale, float2 h[3])
{
    apply_S(m, p[0], p[1], p[2], h[0], h[1], h[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 b = T[c * cs + idx];
        h[c] = make_float2(fmaf(scale, b.x, h[c].x), fmaf(scale, b.y, h[c].y));
    }
    if (kform && m.kk != 0.0f) {
        const float2 ud = mode_div(m, h[0], h[1], h[2]);
        const float f = mode_leray(m);
        h[0] = mode_add(f, m.u1, ud, h[0]);
        h[1] = mode_add(f, m.u2, ud, h[1]);
        h[2] = mode_add(f, m.u3, ud, h[2]);
    }
}

// Step length of a CG iteration from its curvature pq: alpha = rz / pq, or 0
// when pq <= 0 or NaN (the caller sees pq).  FP64, as the host would do it.
__device__ __forceinline__ double cg_alpha(double rz, double pq) { return pq > 0.0 ? rz / pq : 0.0; }

// Total of <p~, H p~>, then alpha.  H p~ is not stored: the update forms it again
// from p~ and T, the same reads as of a stored H p~ (256^3: 30 us less per
// iteration than writing it).
__global__ void __launch_bounds__(kThreads) k_fs_hp(Grid g, const float2* __restrict__ T,
                                                     const float2* __restrict__ ph, size_t cs, int kform,
                                                     RegParams rp, float scale, double* __restrict__ sc, Reduction red)
{
    const int n3h = g.n3 / 2 + 1;
    const uint32_t M = static_cast<uint32_t>(g.n1) * g.n2 * n3h;
    double acc = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        const Mode m = mode_of(g, idx, n3h, rp);
        const float2 p[3] = {ph[idx], ph[cs + idx], ph[2 * cs + idx]};
        float2 h[3];
        hp_mode(m, p, T, cs, idx, kform, scale, h);
        acc += static_cast<double>(m.wt * cdot3(p[0], p[1], p[2], h[0], h[1], h[2]));
    }
    double pq;
    if (grid_sum(acc, red, &pq)) {
        sc[kPcgAlpha] = cg_alpha(sc[kPcgRz], pq);
        put_result(red, 1, sc[kPcgAlpha]);
    }
}

// x~ += alpha p~, r~ -= alpha H p~; totals |r~|^2 and <r~, z~> with z~ = M r~
// (recomputed by the next direction kernel), or, when a stored preconditioned
// residual zc is given, <H p~, zc> instead.  Without zc also beta and the new
// rz for the next direction.
__global__ void __launch_bounds__(kThreads) k_fs_update(Grid g, const float2* __restrict__ T,
                                                         const float2* __restrict__ ph,
                                                         float2* __restrict__ xh, float2* __restrict__ rh,
                                                         const float2* __restrict__ zc, size_t cs, int kform, int op,
                                                         RegParams rp, float scale, double* __restrict__ sc,
                                                         Reduction red)
{
    const float alpha = static_cast<float>(sc[kPcgAlpha]);
    const int n3h = g.n3 / 2 + 1;
    const uint32_t M = static_cast<uint32_t>(g.n1) * g.n2 * n3h;
    double arr = 0.0, arz = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        const Mode m = mode_of(g, idx, n3h, rp);
        const float2 p[3] = {ph[idx], ph[cs + idx], ph[2 * cs + idx]};
        float2 h[3], x[3], r[3];
        load3(xh, cs, idx, x);
        load3(rh, cs, idx, r);
        hp_mode(m, p, T, cs, idx, kform, scale, h);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            r[c] = make_float2(fmaf(-alpha, h[c].x, r[c].x), fmaf(-alpha, h[c].y, r[c].y));
            xh[c * cs + idx] = make_float2(fmaf(alpha, p[c].x, x[c].x), fmaf(alpha, p[c].y, x[c].y));
            rh[c * cs + idx] = r[c];
        }
        arr += static_cast<double>(m.wt * cdot3(r[0], r[1], r[2], r[0], r[1], r[2]));
        if (zc) {
            arz += static_cast<double>(m.wt * cdot3(h[0], h[1], h[2], zc[idx], zc[cs + idx], zc[2 * cs + idx]));
        } else {
            float2 z0, z1, z2;
            apply_inv(m, op, r[0], r[1], r[2], z0, z1, z2);
            arz += static_cast<double>(m.wt * cdot3(r[0], r[1], r[2], z0, z1, z2));
        }
    }
    double tot[2];
    if (grid_sum2(arr, arz, red, tot) && !zc) {
        sc[kPcgBeta] = tot[1] / sc[kPcgRz];
        sc[kPcgRz] = tot[1];
    }
}

__device__ __forceinline__ bool aligned16(const void* p)
{
    return (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
}

__global__ void __launch_bounds__(kThreads) k_dot(const float* __restrict__ x, const float* __restrict__ y, size_t n,
                                                   Reduction red)
{
    double acc = 0.0;
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    const size_t t0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x;
    size_t done = 0;
    if (aligned16(x) && aligned16(y)) {
        const size_t n4 = n / 4;
        const float4* x4 = reinterpret_cast<const float4*>(x);
        const float4* y4 = reinterpret_cast<const float4*>(y);
        for (size_t i = t0; i < n4; i += stride) {
            const float4 a = __ldg(x4 + i), b = __ldg(y4 + i);
            acc += static_cast<double>(a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w);
        }
        done = n4 * 4;
    }
    for (size_t i = done + t0; i < n; i += stride) acc += static_cast<double>(x[i] * y[i]);
    grid_sum(acc, red);
}

template <class S>
__global__ void __launch_bounds__(kThreads) k_sqdiff(const S* __restrict__ a, const S* __restrict__ b, size_t n,
                                                      Reduction red)
{
    double acc = 0.0;
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    const size_t t0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x;
    size_t done = 0;
    if constexpr (sizeof(S) == 4) {
        if (aligned16(a) && aligned16(b)) {
            const size_t n4 = n / 4;
            const float4* a4 = reinterpret_cast<const float4*>(a);
            const float4* b4 = reinterpret_cast<const float4*>(b);
            for (size_t i = t0; i < n4; i += stride) {
                const float4 p = __ldg(a4 + i), q = __ldg(b4 + i);
                const float d0 = p.x - q.x, d1 = p.y - q.y, d2 = p.z - q.z, d3 = p.w - q.w;
                acc += static_cast<double>(d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3);
            }
            done = n4 * 4;
        }
    }
    for (size_t i = done + t0; i < n; i += stride) {
        const float d = ldf<S>(a + i) - ldf<S>(b + i);
        acc += static_cast<double>(d * d);
    }
    grid_sum(acc, red);
}

// max over points of |v|_2^2 in FP64.
//
// Bound: one pass over v (12 B per point, HBM).  The FP64 pipe of this part
// runs 2 operations per clock and SM, so forming every |v|^2 in FP64 cost ten
// times the pass (256^3: 336 us; 512^3: 2567 us).  Each point is first
// formed in FP32 (relative error below 2^-22: three roundings of non-negative
// terms); only points that can reach the block's largest value so far are
// formed in FP64, a few per warp.  thr is that value lowered by 2^-20, so a
// point below it is below the FP64 maximum too; it is raised by a batch's own
// largest point before the batch is tested, and it stays 0 (every point is
// formed) until the maximum is normal.  Non-finite points always compare above
// it (bit patterns of non-negative floats, NaN on top).  The result is the
// FP64 maximum, bit for bit, and keeps a NaN; maxima are taken on the bit
// patterns (integers), which order non-negative doubles the same way.
__device__ __forceinline__ unsigned norm3_bits(float a, float b, float c)
{
    return __float_as_uint(fmaf(c, c, fmaf(b, b, a * a)));
}

__device__ __forceinline__ void norm3_fold(float a, float b, float c, unsigned s, unsigned thr,
                                           unsigned long long& hi)
{
    if (s < thr) return;
    const double x = a, y = b, z = c;
    const unsigned long long t =
        static_cast<unsigned long long>(__double_as_longlong(x * x + y * y + z * z)) & 0x7fffffffffffffffull;
    hi = t > hi ? t : hi;
}

__device__ __forceinline__ void norm3_fold4(const float4& a, const float4& b, const float4& c, const uint4& s,
                                            unsigned thr, unsigned long long& hi)
{
    norm3_fold(a.x, b.x, c.x, s.x, thr, hi);
    norm3_fold(a.y, b.y, c.y, s.y, thr, hi);
    norm3_fold(a.z, b.z, c.z, s.z, thr, hi);
    norm3_fold(a.w, b.w, c.w, s.w, thr, hi);
}

__device__ __forceinline__ uint4 norm3_bits4(const float4& a, const float4& b, const float4& c)
{
    return make_uint4(norm3_bits(a.x, b.x, c.x), norm3_bits(a.y, b.y, c.y), norm3_bits(a.z, b.z, c.z),
                      norm3_bits(a.w, b.w, c.w));
}

__device__ __forceinline__ unsigned max4(const uint4& s) { return max(max(s.x, s.y), max(s.z, s.w)); }

// Whether any component of the points is non-zero.
__device__ __forceinline__ bool norm3_any4(const float4& a, const float4& b, const float4& c)
{
    return fabsf(a.x) + fabsf(a.y) + fabsf(a.z) + fabsf(a.w) + fabsf(b.x) + fabsf(b.y) + fabsf(b.z) + fabsf(b.w) +
               fabsf(c.x) + fabsf(c.y) + fabsf(c.z) + fabsf(c.w) !=
           0.0f;
}

// The threshold raised by a batch of points of which m is the warp's largest
// FP32 value.
__device__ __forceinline__ unsigned norm3_threshold(unsigned m, unsigned thr)
{
    const float f = __uint_as_float(m);
    if (m >= 0x7f800000u || !(f > 1e-30f)) return thr;  // non-finite, or rounding not relative
    return max(thr, __float_as_uint(f * (1.0f - 9.5367431640625e-07f)));
}

__global__ void __launch_bounds__(kThreads) k_maxnorm3(const float* __restrict__ v, size_t N, Reduction out)
{
    __shared__ unsigned bthr;                       // the block's threshold (only ever rises)
    unsigned long long hi = 0;                      // bits of the FP64 maximum
    if (threadIdx.x == 0) bthr = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    const size_t t0 = blockIdx.x * static_cast<size_t>(kThreads) + (threadIdx.x & ~31u);  // uniform in the warp
    auto raise = [&](unsigned m, unsigned thr) {
        const unsigned t = norm3_threshold(m, thr);
        if (t > thr && lane == 0) atomicMax(&bthr, t);
        return t;
    };
    if (aligned16(v) && (N & 3) == 0) {
        const size_t n4 = N / 4;
        const float4* v4 = reinterpret_cast<const float4*>(v);
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        for (size_t base = t0; base < n4; base += 2 * stride) {
            const size_t i = base + lane, j = i + stride;
            const bool in = i < n4, jn = j < n4;
            const float4 a = in ? __ldg(v4 + i) : zero, b = in ? __ldg(v4 + n4 + i) : zero,
                         c = in ? __ldg(v4 + 2 * n4 + i) : zero;
            const float4 d = jn ? __ldg(v4 + j) : zero, e = jn ? __ldg(v4 + n4 + j) : zero,
                         f = jn ? __ldg(v4 + 2 * n4 + j) : zero;
            unsigned thr = *static_cast<volatile unsigned*>(&bthr);
            thr = __shfl_sync(0xffffffffu, thr, 0);
            const uint4 s = norm3_bits4(a, b, c), u = norm3_bits4(d, e, f);
            const unsigned m = __reduce_max_sync(0xffffffffu, max(max4(s), max4(u)));
            // FP32 squares of zeros, or of values below 1e-22 or so: only the latter go on
            if (m == 0u && !__any_sync(0xffffffffu, norm3_any4(a, b, c) || norm3_any4(d, e, f))) continue;
            if (m >= thr) {
                thr = raise(m, thr);
                norm3_fold4(a, b, c, s, thr, hi);
                norm3_fold4(d, e, f, u, thr, hi);
            }
        }
    } else {
        for (size_t base = t0; base < N; base += stride) {
            const size_t i = base + lane;
            const bool in = i < N;
            const float a = in ? v[i] : 0.0f, b = in ? v[N + i] : 0.0f, c = in ? v[2 * N + i] : 0.0f;
            unsigned thr = *static_cast<volatile unsigned*>(&bthr);
            thr = __shfl_sync(0xffffffffu, thr, 0);
            const unsigned s = norm3_bits(a, b, c);
            const unsigned m = __reduce_max_sync(0xffffffffu, s);
            if (m == 0u && !__any_sync(0xffffffffu, fabsf(a) + fabsf(b) + fabsf(c) != 0.0f)) continue;
            if (m >= thr) {
                thr = raise(m, thr);
                norm3_fold(a, b, c, s, thr, hi);
            }
        }
    }
    grid_max_bits(hi, out);
}

// Dice counts (Sec. 4.1): both = 0 counts a >= t and b >= t into totals 0 and
// 1; both = 1 counts (a >= t) and (b >= t) into total 0 (1 is zero).
// FP64 partial sums of integers: exact below 2^53.
__global__ void __launch_bounds__(kThreads) k_count(const float* __restrict__ a, const float* __restrict__ b, size_t n,
                                                     float t, int both, Reduction red)
{
    unsigned long long ca = 0, cb = 0;
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    for (size_t i = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; i < n; i += stride) {
        const bool ia = a[i] >= t, ib = b[i] >= t;
        if (both) {
            ca += (ia && ib) ? 1u : 0u;
        } else {
            ca += ia ? 1u : 0u;
            cb += ib ? 1u : 0u;
        }
    }
    double tot[2];
    grid_sum2(static_cast<double>(ca), static_cast<double>(cb), red, tot);
}

// The vector updates take a float4 path when every pointer is 16-byte aligned
// (the context's buffers always are) and a scalar loop for the tail.
__global__ void __launch_bounds__(kThreads) k_axpy(float a, const float* __restrict__ x,
                                                    float* __restrict__ y, size_t n)
{
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    const size_t t0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x;
    size_t done = 0;
    if (aligned16(x) && aligned16(y)) {
        const size_t n4 = n / 4;
        const float4* x4 = reinterpret_cast<const float4*>(x);
        float4* y4 = reinterpret_cast<float4*>(y);
        for (size_t i = t0; i < n4; i += stride) {
            const float4 u = __ldg(x4 + i);
            float4 w = y4[i];
            w.x = fmaf(a, u.x, w.x); w.y = fmaf(a, u.y, w.y); w.z = fmaf(a, u.z, w.z); w.w = fmaf(a, u.w, w.w);
            y4[i] = w;
        }
        done = n4 * 4;
    }
    for (size_t i = done + t0; i < n; i += stride) y[i] = fmaf(a, x[i], y[i]);
}

__global__ void __launch_bounds__(kThreads) k_xpay(const float* __restrict__ x, float a,
                                                    const float* y, float* z, size_t n)
{
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    const size_t t0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x;
    size_t done = 0;
    if (aligned16(x) && aligned16(y) && aligned16(z)) {
        const size_t n4 = n / 4;
        const float4* x4 = reinterpret_cast<const float4*>(x);
        const float4* y4 = reinterpret_cast<const float4*>(y);
        float4* z4 = reinterpret_cast<float4*>(z);
        for (size_t i = t0; i < n4; i += stride) {
            const float4 u = __ldg(x4 + i);
            const float4 v = y4[i];
            z4[i] = make_float4(fmaf(a, v.x, u.x), fmaf(a, v.y, u.y), fmaf(a, v.z, u.z), fmaf(a, v.w, u.w));
        }
        done = n4 * 4;
    }
    for (size_t i = done + t0; i < n; i += stride) z[i] = fmaf(a, y[i], x[i]);
}

unsigned stream_blocks(size_t n)
{
    size_t b = (n + kThreads - 1) / kThreads;
    const size_t cap = 152 * 16;  // enough resident blocks to cover the GPU, grid-stride beyond
    return static_cast<unsigned>(b < cap ? (b ? b : 1) : cap);
}


// B-spline prefilter in Fourier space: every mode of ncomp half spectra is
// divided by N prod_axes (2 + cos(k_a h_a)) / 3 (the sampled cubic B-spline),
// so that the inverse transform gives the interpolating spline's coefficients.
__global__ void k_bspline_scale(Grid g, cufftComplex* __restrict__ spec, size_t M, int ncomp, float invN)
{
    const size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
    if (e >= M * ncomp) return;
    const size_t m = e % M;
    const int n3h = g.n3 / 2 + 1;
    const int j3 = static_cast<int>(m % n3h);
    const int j2 = static_cast<int>((m / n3h) % g.n2);
    const int j1 = static_cast<int>(m / (static_cast<size_t>(n3h) * g.n2));
    const float two_pi = 6.283185307179586f;
    const float s1 = (2.0f + cosf(two_pi * j1 / g.n1)) * (1.0f / 3.0f);
    const float s2 = (2.0f + cosf(two_pi * j2 / g.n2)) * (1.0f / 3.0f);
    const float s3 = (2.0f + cosf(two_pi * j3 / g.n3)) * (1.0f / 3.0f);
    const float f = invN / (s1 * s2 * s3);
    spec[e].x *= f;
    spec[e].y *= f;
}
// out = w_end (m^0 + m^nt) + w_mid (m^1 + ... + m^{nt-1}) (trapezoid over the
// stored levels; N is a multiple of 8 and the levels are the context's own, so
// four points go together).
template <class S>
__device__ __forceinline__ float4 load4(const S* p)
{
    if constexpr (sizeof(S) == 4) {
        return __ldg(reinterpret_cast<const float4*>(p));
    } else {
        const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
        S v[4];
        memcpy(v, &u, 8);
        return make_float4(to_f32<S>(v[0]), to_f32<S>(v[1]), to_f32<S>(v[2]), to_f32<S>(v[3]));
    }
}

template <class S>
__global__ void __launch_bounds__(kThreads) k_mean_levels(const S* __restrict__ m, int nt, float w_end,
                                                           float w_mid, size_t N, float* __restrict__ out)
{
    for (size_t i = 4 * (blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x); i < N;
         i += static_cast<size_t>(gridDim.x) * (4 * kThreads)) {
        const float4 a = load4(m + i), b = load4(m + static_cast<size_t>(nt) * N + i);
        float4 acc = make_float4(w_end * (a.x + b.x), w_end * (a.y + b.y), w_end * (a.z + b.z), w_end * (a.w + b.w));
#pragma unroll 4
        for (int j = 1; j < nt; ++j) {
            const float4 v = load4(m + static_cast<size_t>(j) * N + i);
            acc.x = fmaf(w_mid, v.x, acc.x);
            acc.y = fmaf(w_mid, v.y, acc.y);
            acc.z = fmaf(w_mid, v.z, acc.z);
            acc.w = fmaf(w_mid, v.w, acc.w);
        }
        *reinterpret_cast<float4*>(out + i) = acc;
    }
}

__global__ void __launch_bounds__(kThreads) k_cscale(float2* __restrict__ x, size_t n, float s)
{
    for (size_t i = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; i < n;
         i += static_cast<size_t>(gridDim.x) * kThreads)
        x[i] = cmul(s, x[i]);
}

// ---- two-level zero-velocity preconditioner (Sec. 2.2) ----
// The coarse grid gc keeps the modes |k_i| < gc.n_i / 2 of the fine grid gf
// (its Nyquist planes are dropped); the inner PCG runs on those modes without
// the mean (k = 0), the "kept" modes, in the same scaled half-spectrum
// convention as the outer PCG (coefficients are resolution independent, so
// restriction and prolongation copy them).

// Wavenumbers of half-spectrum mode idx of grid g.
__device__ __forceinline__ void wavenumbers(const Grid& g, uint32_t idx, int& k1, int& k2, int& k3)
{
    const uint32_t n3h = g.n3 / 2 + 1;
    const uint32_t r = idx / n3h;
    k3 = static_cast<int>(idx - r * n3h);
    const int i = static_cast<int>(r / static_cast<uint32_t>(g.n2));
    const int j = static_cast<int>(r) - i * g.n2;
    k1 = i <= g.n1 / 2 ? i : i - g.n1;
    k2 = j <= g.n2 / 2 ? j : j - g.n2;
}

// |k_i| < n_i / 2 on every axis of grid g (no Nyquist plane)
__device__ __forceinline__ bool below_nyquist(const Grid& g, int k1, int k2, int k3)
{
    return 2 * abs(k1) < g.n1 && 2 * abs(k2) < g.n2 && 2 * k3 < g.n3;
}

// Half-spectrum index of wavenumber k on grid g (k assumed representable).
__device__ __forceinline__ size_t mode_index(const Grid& g, int k1, int k2, int k3)
{
    const int i = k1 >= 0 ? k1 : k1 + g.n1;
    const int j = k2 >= 0 ? k2 : k2 + g.n2;
    return (static_cast<size_t>(i) * g.n2 + j) * (g.n3 / 2 + 1) + k3;
}

// Coarse spectrum of a fine field given by its unnormalised R2C transform F
// (scaled by 1/N here): every coarse mode below the coarse Nyquist, mean
// included (the restriction R of the mean state gradient).
__global__ void __launch_bounds__(kThreads) k_tl_restrict(Grid gf, const float2* __restrict__ F, size_t csf,
                                                           Grid gc, float2* __restrict__ out, size_t csc,
                                                           float invN)
{
    const size_t Mc = static_cast<size_t>(gc.n1) * gc.n2 * (gc.n3 / 2 + 1);
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < Mc; idx += gridDim.x * kThreads) {
        int k1, k2, k3;
        wavenumbers(gc, idx, k1, k2, k3);
        const bool keep = below_nyquist(gc, k1, k2, k3);
        const size_t f = keep ? mode_index(gf, k1, k2, k3) : 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) out[c * csc + idx] = keep ? cmul(invN, F[c * csf + f]) : make_float2(0.f, 0.f);
    }
}

// Start of the inner PCG: r = Q R (rscale rf) (kept modes of the fine residual),
// x = 0, z = M r, p = z (and its copy cp for the inverse transform); totals
// |r|^2 and <r, z>.
__global__ void __launch_bounds__(kThreads) k_tl_start(Grid gf, const float2* __restrict__ rf, size_t csf,
                                                        Grid gc, float2* __restrict__ rh, float2* __restrict__ xh,
                                                        float2* __restrict__ ph, float2* __restrict__ cp, size_t cs,
                                                        int op, RegParams rp, float rscale, double* __restrict__ sc,
                                                        Reduction red)
{
    const int n3h = gc.n3 / 2 + 1;
    const uint32_t Mc = static_cast<uint32_t>(gc.n1) * gc.n2 * n3h;
    double arr = 0.0, arz = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < Mc; idx += gridDim.x * kThreads) {
        int k1, k2, k3;
        wavenumbers(gc, idx, k1, k2, k3);
        const bool keep = below_nyquist(gc, k1, k2, k3) && (k1 | k2 | k3) != 0;
        const size_t f = keep ? mode_index(gf, k1, k2, k3) : 0;
        const float2 zero = make_float2(0.f, 0.f);
        float2 r[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) r[c] = keep ? cmul(rscale, rf[c * csf + f]) : zero;
        const Mode m = mode_of(gc, idx, n3h, rp);
        float2 z[3];
        apply_inv(m, op, r[0], r[1], r[2], z[0], z[1], z[2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            rh[c * cs + idx] = r[c];
            xh[c * cs + idx] = zero;
            ph[c * cs + idx] = z[c];
            cp[c * cs + idx] = z[c];
        }
        arr += static_cast<double>(m.wt * cdot3(r[0], r[1], r[2], r[0], r[1], r[2]));
        arz += static_cast<double>(m.wt * cdot3(r[0], r[1], r[2], z[0], z[1], z[2]));
    }
    double tot[2];
    if (grid_sum2(arr, arz, red, tot)) sc[kPcgRz] = tot[1];
}

// In place on the coarse real fields: p <- gbar (gbar . p).
__global__ void __launch_bounds__(kThreads) k_tl_rank1(const float* __restrict__ gbar, float* __restrict__ p,
                                                        size_t Nc)
{
    for (size_t i = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; i < Nc;
         i += static_cast<size_t>(gridDim.x) * kThreads) {
        const float g0 = gbar[i], g1 = gbar[Nc + i], g2 = gbar[2 * Nc + i];
        const float s = g0 * p[i] + g1 * p[Nc + i] + g2 * p[2 * Nc + i];
        p[i] = s * g0;
        p[Nc + i] = s * g1;
        p[2 * Nc + i] = s * g2;
    }
}

// One mode of q = Q (S p + scale T) (K of the sum for the paper's gradient
// form), T the unnormalised transform of gbar (gbar . p).
__device__ __forceinline__ void tl_q(const Grid& gc, uint32_t idx, const Mode& m, const float2 p[3],
                                     const float2* __restrict__ T, size_t cs, int kform, float scale, float2 h[3])
{
    hp_mode(m, p, T, cs, idx, kform, scale, h);
    int k1, k2, k3;
    wavenumbers(gc, idx, k1, k2, k3);
    if (!(below_nyquist(gc, k1, k2, k3) && (k1 | k2 | k3) != 0)) h[0] = h[1] = h[2] = make_float2(0.f, 0.f);
}

// Total of <p, q>, then alpha.  Neither q nor the preconditioned residual is
// stored in the inner PCG: the update and the direction form them again from
// what they read anyway, and T lives where the copy of p was, so that an
// iteration's five coarse arrays (26 MB each at 128^3) stay near the L2 size
// instead of eight.
__global__ void __launch_bounds__(kThreads) k_tl_hp(Grid gc, const float2* __restrict__ T,
                                                     const float2* __restrict__ ph, size_t cs, int kform,
                                                     RegParams rp, float scale, double* __restrict__ sc, Reduction red)
{
    const int n3h = gc.n3 / 2 + 1;
    const uint32_t Mc = static_cast<uint32_t>(gc.n1) * gc.n2 * n3h;
    double acc = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < Mc; idx += gridDim.x * kThreads) {
        const Mode m = mode_of(gc, idx, n3h, rp);
        const float2 p[3] = {ph[idx], ph[cs + idx], ph[2 * cs + idx]};
        float2 h[3];
        tl_q(gc, idx, m, p, T, cs, kform, scale, h);
        acc += static_cast<double>(m.wt * cdot3(p[0], p[1], p[2], h[0], h[1], h[2]));
    }
    double pq;
    if (grid_sum(acc, red, &pq)) {
        sc[kPcgAlpha] = cg_alpha(sc[kPcgRz], pq);
        put_result(red, 1, pq > 0.0 ? 0.0 : (pq == pq ? 1.0 : 2.0));  // breakdown flag; 2: pq is NaN
    }
}

// x += alpha p, r -= alpha q; totals |r|^2 and <r, z> with z = M r, then beta =
// rz_new / rz and rz <- rz_new for the next direction.
__global__ void __launch_bounds__(kThreads) k_tl_update(Grid gc, const float2* __restrict__ T,
                                                         const float2* __restrict__ ph, float2* __restrict__ xh,
                                                         float2* __restrict__ rh, size_t cs, int kform, int op,
                                                         RegParams rp, float scale, double* __restrict__ sc,
                                                         Reduction red)
{
    const float alpha = static_cast<float>(sc[kPcgAlpha]);
    const int n3h = gc.n3 / 2 + 1;
    const uint32_t Mc = static_cast<uint32_t>(gc.n1) * gc.n2 * n3h;
    double arr = 0.0, arz = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < Mc; idx += gridDim.x * kThreads) {
        const Mode m = mode_of(gc, idx, n3h, rp);
        const float2 p[3] = {ph[idx], ph[cs + idx], ph[2 * cs + idx]};
        float2 h[3], x[3], r[3];
        load3(xh, cs, idx, x);
        load3(rh, cs, idx, r);
        tl_q(gc, idx, m, p, T, cs, kform, scale, h);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            r[c] = make_float2(fmaf(-alpha, h[c].x, r[c].x), fmaf(-alpha, h[c].y, r[c].y));
            xh[c * cs + idx] = make_float2(fmaf(alpha, p[c].x, x[c].x), fmaf(alpha, p[c].y, x[c].y));
            rh[c * cs + idx] = r[c];
        }
        float2 z0, z1, z2;
        apply_inv(m, op, r[0], r[1], r[2], z0, z1, z2);
        arr += static_cast<double>(m.wt * cdot3(r[0], r[1], r[2], r[0], r[1], r[2]));
        arz += static_cast<double>(m.wt * cdot3(r[0], r[1], r[2], z0, z1, z2));
    }
    double tot[2];
    if (grid_sum2(arr, arz, red, tot)) {
        sc[kPcgBeta] = tot[1] / sc[kPcgRz];
        sc[kPcgRz] = tot[1];
    }
}

// p = z + beta p (p = z when first) and its copy cp for the inverse transform:
// the outer PCG when z is stored.
__global__ void __launch_bounds__(kThreads) k_dir_stored(Grid g, const float2* __restrict__ zh,
                                                          float2* __restrict__ ph, float2* __restrict__ cp, size_t cs,
                                                          float beta, int first)
{
    const uint32_t M = static_cast<uint32_t>(g.n1) * g.n2 * (g.n3 / 2 + 1);
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        float2 z[3], o[3] = {};
        load3(zh, cs, idx, z);
        if (!first) load3(ph, cs, idx, o);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 p = z[c];
            if (!first) p = make_float2(fmaf(beta, o[c].x, z[c].x), fmaf(beta, o[c].y, z[c].y));
            ph[c * cs + idx] = p;
            cp[c * cs + idx] = p;
        }
    }
}

// Outer preconditioned residual of r = rscale rf: z = E x (kept coarse modes), r
// on the mean, M r on every other mode; total <r, z> (also the outer PCG's rz).
__global__ void __launch_bounds__(kThreads) k_tl_finish(Grid gf, const float2* __restrict__ rf,
                                                         float2* __restrict__ zf, size_t csf, Grid gc,
                                                         const float2* __restrict__ xc, size_t csc, int op,
                                                         RegParams rp, float rscale, double* __restrict__ sc,
                                                         Reduction red)
{
    const int n3h = gf.n3 / 2 + 1;
    const uint32_t M = static_cast<uint32_t>(gf.n1) * gf.n2 * n3h;
    double az = 0.0;
    for (uint32_t idx = blockIdx.x * kThreads + threadIdx.x; idx < M; idx += gridDim.x * kThreads) {
        int k1, k2, k3;
        wavenumbers(gf, idx, k1, k2, k3);
        const bool low = below_nyquist(gc, k1, k2, k3) && (k1 | k2 | k3) != 0;
        const Mode m = mode_of(gf, idx, n3h, rp);
        const float2 r0 = cmul(rscale, rf[idx]), r1 = cmul(rscale, rf[csf + idx]), r2 = cmul(rscale, rf[2 * csf + idx]);
        float2 z[3];
        if (low) {
            const size_t ci = mode_index(gc, k1, k2, k3);
#pragma unroll
            for (int c = 0; c < 3; ++c) z[c] = xc[c * csc + ci];
        } else {
            apply_inv(m, op, r0, r1, r2, z[0], z[1], z[2]);  // identity at k = 0
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) zf[c * csf + idx] = z[c];
        az += static_cast<double>(m.wt * cdot3(r0, r1, r2, z[0], z[1], z[2]));
    }
    double rz;
    if (grid_sum(az, red, &rz)) sc[kPcgRz] = rz;
}

}  // namespace

void launch_spectral(const Grid& g, const cufftComplex* xh, cufftComplex* yh, size_t cstride, SpectralOp op,
                     RegParams rp, float scale, const Reduction* energy, cudaStream_t st)
{
    const size_t M = static_cast<size_t>(g.n1) * g.n2 * (g.n3 / 2 + 1);
    auto x = reinterpret_cast<const float2*>(xh);
    auto y = reinterpret_cast<float2*>(yh);
    if (energy)
        k_spectral<true><<<energy->nblocks, kThreads, 0, st>>>(g, x, y, cstride, static_cast<int>(op), rp, scale, *energy);
    else
        k_spectral<false><<<stream_blocks(M), kThreads, 0, st>>>(g, x, y, cstride, static_cast<int>(op), rp, scale,
                                                                Reduction{});
}

void launch_reg_energy(const Grid& g, const cufftComplex* vh, const cufftComplex* xh, size_t cs, float alpha,
                       RegParams rp, const Reduction& red, cudaStream_t st)
{
    k_reg_energy<<<red.nblocks, kThreads, 0, st>>>(g, reinterpret_cast<const float2*>(vh),
                                                   reinterpret_cast<const float2*>(xh), cs, alpha, rp, red);
}

void launch_spectral_direction(const Grid& g, const cufftComplex* rh, cufftComplex* ph, cufftComplex* cp,
                               size_t cstride, const double* sc, int first, SpectralOp op, RegParams rp,
                               cudaStream_t st)
{
    const size_t M = static_cast<size_t>(g.n1) * g.n2 * (g.n3 / 2 + 1);
    k_spectral_direction<<<stream_blocks(M), kThreads, 0, st>>>(
        g, reinterpret_cast<const float2*>(rh), reinterpret_cast<float2*>(ph), reinterpret_cast<float2*>(cp),
        cstride, sc, first, static_cast<int>(op), rp);
}

void launch_fs_start(const Grid& g, cufftComplex* spec, cufftComplex* rh, cufftComplex* xh, size_t cs,
                     SpectralOp op, RegParams rp, float scale, double* sc, const Reduction& red, cudaStream_t st)
{
    k_fs_start<<<red.nblocks, kThreads, 0, st>>>(g, reinterpret_cast<float2*>(spec), reinterpret_cast<float2*>(rh),
                                                 reinterpret_cast<float2*>(xh), cs, static_cast<int>(op), rp, scale,
                                                 sc, red);
}

void launch_fs_hp(const Grid& g, const cufftComplex* T, const cufftComplex* ph, size_t cs, int kform, RegParams rp,
                  float scale, double* sc, const Reduction& red, cudaStream_t st)
{
    k_fs_hp<<<red.nblocks, kThreads, 0, st>>>(g, reinterpret_cast<const float2*>(T),
                                              reinterpret_cast<const float2*>(ph), cs, kform, rp, scale, sc, red);
}

void launch_fs_update(const Grid& g, const cufftComplex* T, const cufftComplex* ph, cufftComplex* xh,
                      cufftComplex* rh, const cufftComplex* zc, size_t cs, int kform, SpectralOp op, RegParams rp,
                      float scale, double* sc, const Reduction& red, cudaStream_t st)
{
    k_fs_update<<<red.nblocks, kThreads, 0, st>>>(g, reinterpret_cast<const float2*>(T),
                                                  reinterpret_cast<const float2*>(ph), reinterpret_cast<float2*>(xh),
                                                  reinterpret_cast<float2*>(rh), reinterpret_cast<const float2*>(zc),
                                                  cs, kform, static_cast<int>(op), rp, scale, sc, red);
}

void launch_mean_levels(const void* m, int nt, float w_end, float w_mid, size_t N, float* out, Storage sto,
                        cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_mean_levels<SType><<<stream_blocks(N / 4), kThreads, 0, st>>>(static_cast<const SType*>(m), nt, w_end, w_mid,
                                                                    N, out);
    });
}

// Coarse preconditioner correction: gbar_c <- sqrt(max(w, 0)) gbar_c on the
// coarse grid (three components of n values), so that the zero-velocity
// operator of the result is S + gbar_c w gbar_c^T.
__global__ void k_tl_weight(float* __restrict__ g, const float* __restrict__ w, size_t n)
{
    for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < n;
         e += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const float s = sqrtf(fmaxf(w[e], 0.0f));
        g[e] *= s;
        g[n + e] *= s;
        g[2 * n + e] *= s;
    }
}

void launch_tl_weight(float* gbar_c, const float* w, size_t n, cudaStream_t st)
{
    k_tl_weight<<<stream_blocks(n), kThreads, 0, st>>>(gbar_c, w, n);
}

void launch_cscale(cufftComplex* x, size_t n, float s, cudaStream_t st)
{
    k_cscale<<<stream_blocks(n), kThreads, 0, st>>>(reinterpret_cast<float2*>(x), n, s);
}

void launch_tl_restrict(const Grid& gf, const cufftComplex* F, size_t csf, const Grid& gc, cufftComplex* out,
                        size_t csc, float invN, cudaStream_t st)
{
    const size_t Mc = static_cast<size_t>(gc.n1) * gc.n2 * (gc.n3 / 2 + 1);
    k_tl_restrict<<<stream_blocks(Mc), kThreads, 0, st>>>(gf, reinterpret_cast<const float2*>(F), csf, gc,
                                                          reinterpret_cast<float2*>(out), csc, invN);
}

void launch_tl_start(const Grid& gf, const cufftComplex* rf, size_t csf, const Grid& gc, cufftComplex* rh,
                     cufftComplex* xh, cufftComplex* ph, cufftComplex* cp, size_t cs, SpectralOp op, RegParams rp,
                     float rscale, double* sc, const Reduction& red, cudaStream_t st)
{
    k_tl_start<<<red.nblocks, kThreads, 0, st>>>(gf, reinterpret_cast<const float2*>(rf), csf, gc,
                                                 reinterpret_cast<float2*>(rh), reinterpret_cast<float2*>(xh),
                                                 reinterpret_cast<float2*>(ph), reinterpret_cast<float2*>(cp), cs,
                                                 static_cast<int>(op), rp, rscale, sc, red);
}

void launch_tl_rank1(const float* gbar, float* p, size_t Nc, cudaStream_t st)
{
    k_tl_rank1<<<stream_blocks(Nc), kThreads, 0, st>>>(gbar, p, Nc);
}

void launch_tl_hp(const Grid& gc, const cufftComplex* T, const cufftComplex* ph, size_t cs, int kform, RegParams rp,
                  float scale, double* sc, const Reduction& red, cudaStream_t st)
{
    k_tl_hp<<<red.nblocks, kThreads, 0, st>>>(gc, reinterpret_cast<const float2*>(T),
                                              reinterpret_cast<const float2*>(ph), cs, kform, rp, scale, sc, red);
}

void launch_tl_update(const Grid& gc, const cufftComplex* T, const cufftComplex* ph, cufftComplex* xh,
                      cufftComplex* rh, size_t cs, int kform, SpectralOp op, RegParams rp, float scale, double* sc,
                      const Reduction& red, cudaStream_t st)
{
    k_tl_update<<<red.nblocks, kThreads, 0, st>>>(gc, reinterpret_cast<const float2*>(T),
                                                  reinterpret_cast<const float2*>(ph), reinterpret_cast<float2*>(xh),
                                                  reinterpret_cast<float2*>(rh), cs, kform, static_cast<int>(op), rp,
                                                  scale, sc, red);
}

void launch_dir_stored(const Grid& g, const cufftComplex* zh, cufftComplex* ph, cufftComplex* cp, size_t cs,
                       float beta, int first, cudaStream_t st)
{
    const size_t M = static_cast<size_t>(g.n1) * g.n2 * (g.n3 / 2 + 1);
    k_dir_stored<<<stream_blocks(M), kThreads, 0, st>>>(g, reinterpret_cast<const float2*>(zh),
                                                        reinterpret_cast<float2*>(ph), reinterpret_cast<float2*>(cp),
                                                        cs, beta, first);
}

void launch_tl_finish(const Grid& gf, const cufftComplex* rf, cufftComplex* zf, size_t csf, const Grid& gc,
                      const cufftComplex* xc, size_t csc, SpectralOp op, RegParams rp, float rscale, double* sc,
                      const Reduction& red, cudaStream_t st)
{
    k_tl_finish<<<red.nblocks, kThreads, 0, st>>>(gf, reinterpret_cast<const float2*>(rf),
                                                  reinterpret_cast<float2*>(zf), csf, gc,
                                                  reinterpret_cast<const float2*>(xc), csc, static_cast<int>(op), rp,
                                                  rscale, sc, red);
}

void launch_dot(const float* x, const float* y, size_t n, const Reduction& red, cudaStream_t st)
{
    k_dot<<<red.nblocks, kThreads, 0, st>>>(x, y, n, red);
}

void launch_sqdiff(const void* a, const void* b, size_t n, Storage sto, const Reduction& red, cudaStream_t st)
{
    CLAIRE_STORAGE_DISPATCH(sto, {
        k_sqdiff<SType><<<red.nblocks, kThreads, 0, st>>>(static_cast<const SType*>(a), static_cast<const SType*>(b), n,
                                                          red);
    });
}

void launch_maxnorm3(const float* v, size_t N, const Reduction& red, cudaStream_t st)
{
    k_maxnorm3<<<red.nblocks, kThreads, 0, st>>>(v, N, red);
}

void launch_count(const float* a, const float* b, size_t n, float t, int both, const Reduction& red, cudaStream_t st)
{
    k_count<<<red.nblocks, kThreads, 0, st>>>(a, b, n, t, both, red);
}

void launch_axpy(float a, const float* x, float* y, size_t n, cudaStream_t st)
{
    k_axpy<<<stream_blocks(n), kThreads, 0, st>>>(a, x, y, n);
}

void launch_xpay(const float* x, float a, const float* y, float* z, size_t n, cudaStream_t st)
{
    k_xpay<<<stream_blocks(n), kThreads, 0, st>>>(x, a, y, z, n);
}

}  // namespace claire

namespace claire {
void launch_bspline_scale(const Grid& g, cufftComplex* spec, size_t M, int ncomp, cudaStream_t st)
{
    const size_t n = M * ncomp;
    k_bspline_scale<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(g, spec, M, ncomp,
                                                                          1.0f / static_cast<float>(g.N));
}
}  // namespace claire
