// Internal declarations of libclaire: kernel launchers (one per kernel) and
// block-level reduction helpers.  Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <cufft.h>

#include <cstddef>
#include <cstdint>

#include "claire.h"
#include "common.cuh"

namespace claire {

// ---- reductions (256-thread blocks, fixed order: deterministic) ----

// A grid-wide FP64 reduction in one launch: every block writes its partial (one
// or two arrays of nblocks doubles), and the block that finishes last adds
// them up in a fixed order and stores the scaled totals at out (device) and
// host (their mirror in mapped pinned memory, read after the stream has been
// synchronised).  `ticket` counts finished blocks and is left at 0; launches
// that share it must be ordered (one stream).  A separate one-block kernel and
// a copy of the scalars, which this replaces, cost 4 and 3 us per reduction.
struct Reduction {
    double* partials;  // 2 nblocks doubles
    int nblocks;
    double scale;
    double* out;
    double* host;
    unsigned* ticket;
};

#ifdef __CUDACC__
__device__ __forceinline__ double warp_sum(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    return x;
}

// Block sums of K values per thread, in a fixed order: valid in lane 0 of warp k
// for value k.  An FP64 warp addition occupies the FP64 pipe for 16 cycles here,
// so the 256 values go through shared memory and one warp each adds them (13
// additions) instead of a shuffle tree in every warp (45 additions per block,
// 2.8 us per SM and pair of sums with four resident blocks).
template <int K>
__device__ __forceinline__ double block_sums(const double (&x)[K])
{
    __shared__ double sh[K][256];
#pragma unroll
    for (int k = 0; k < K; ++k) sh[k][threadIdx.x] = x[k];
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double y = 0.0;
    if (wid < K) {
#pragma unroll
        for (int i = 0; i < 8; ++i) y += sh[wid][lane + 32 * i];
        y = warp_sum(y);
    }
    return y;
}

// Whether this block is the last of the grid to get here; lane 0 of the first K
// warps has written the block's partials.  Same answer in every thread.
__device__ __forceinline__ bool last_block(unsigned* ticket)
{
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

__device__ __forceinline__ void put_result(const Reduction& r, int slot, double v)
{
    r.out[slot] = v;
    if (r.host) r.host[slot] = v;
}

// Grid-wide sums of K (1 or 2) values per thread.  True, with the scaled totals
// stored and returned in tot, in thread 0 of the block that finished last.
template <int K>
__device__ __forceinline__ bool grid_sums(const double (&x)[K], const Reduction& r, double (&tot)[K])
{
    __shared__ double fin[K];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double y = block_sums<K>(x);
    if (lane == 0 && wid < K) r.partials[wid * r.nblocks + blockIdx.x] = y;
    if (!last_block(r.ticket)) return false;
    // 256 / K threads per total, up to four loads in flight each
    constexpr int W = 256 / K;
    const int k = threadIdx.x / W, t = threadIdx.x % W;
    const double* p = r.partials + k * r.nblocks;
    double s = 0.0;
    for (int i = t; i < r.nblocks; i += 4 * W) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = i + u * W < r.nblocks ? __ldcg(p + i + u * W) : 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u) s += v[u];
    }
    // a thread holds a share of one total only: the other totals' shares are 0
    double z[K];
#pragma unroll
    for (int c = 0; c < K; ++c) z[c] = c == k ? s : 0.0;
    __syncthreads();  // block_sums' shared memory is read again below
    const double all = block_sums<K>(z);
    if (lane == 0 && wid < K) fin[wid] = all * r.scale;
    __syncthreads();
    if (threadIdx.x != 0) return false;
#pragma unroll
    for (int c = 0; c < K; ++c) {
        tot[c] = fin[c];
        put_result(r, c, tot[c]);
    }
    return true;
}

// One sum.
__device__ __forceinline__ bool grid_sum(double x, const Reduction& r, double* total = nullptr)
{
    const double v[1] = {x};
    double tot[1];
    if (!grid_sums<1>(v, r, tot)) return false;
    if (total) *total = tot[0];
    return true;
}

// Block maximum of non-negative doubles given by their bit patterns (integers
// order them the same way, NaN on top), then over the grid: result at out[0].
__device__ __forceinline__ unsigned long long block_max_bits(unsigned long long hi)
{
    __shared__ unsigned long long sh[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, hi, o);
        hi = t > hi ? t : hi;
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = hi;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) hi = sh[w] > hi ? sh[w] : hi;
    }
    __syncthreads();
    return hi;  // thread 0
}

__device__ __forceinline__ void grid_max_bits(unsigned long long hi, const Reduction& r)
{
    hi = block_max_bits(hi);
    if (threadIdx.x == 0) r.partials[blockIdx.x] = __longlong_as_double(static_cast<long long>(hi));
    if (!last_block(r.ticket)) return;
    hi = 0;
    for (int i = threadIdx.x; i < r.nblocks; i += 256) {
        const unsigned long long t = static_cast<unsigned long long>(__double_as_longlong(__ldcg(r.partials + i)));
        hi = t > hi ? t : hi;
    }
    hi = block_max_bits(hi);
    if (threadIdx.x == 0) put_result(r, 0, __longlong_as_double(static_cast<long long>(hi)));
}

// min / max that keep a NaN operand (fmin / fmax return the other operand),
// so that a NaN anywhere in a reduction reaches its result
__device__ __forceinline__ double min_nan(double a, double b) { return (a != a || b != b) ? a + b : fmin(a, b); }
__device__ __forceinline__ double max_nan(double a, double b) { return (a != a || b != b) ? a + b : fmax(a, b); }

// Block minimum of lo and maximum of hi into pmin / pmax[blockIdx.x]; a NaN
// in either propagates to that result.
__device__ __forceinline__ void block_minmax(double lo, double hi, double* pmin, double* pmax)
{
    __shared__ double slo[32], shi[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min_nan(lo, __shfl_down_sync(0xffffffffu, lo, o));
        hi = max_nan(hi, __shfl_down_sync(0xffffffffu, hi, o));
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        slo[wid] = lo;
        shi[wid] = hi;
    }
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        double a = lane < nw ? slo[lane] : 1e300;
        double b = lane < nw ? shi[lane] : -1e300;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a = min_nan(a, __shfl_down_sync(0xffffffffu, a, o));
            b = max_nan(b, __shfl_down_sync(0xffffffffu, b, o));
        }
        if (lane == 0) {
            pmin[blockIdx.x] = a;
            pmax[blockIdx.x] = b;
        }
    }
}

// Grid-wide minimum (out[0]) and maximum (out[1]); partial maxima first.
__device__ __forceinline__ void grid_minmax(double lo, double hi, const Reduction& r)
{
    __shared__ double fin[16];
    block_minmax(lo, hi, r.partials + r.nblocks, r.partials);
    if (!last_block(r.ticket)) return;
    lo = 1e300;
    hi = -1e300;
    for (int i = threadIdx.x; i < r.nblocks; i += 256) {
        lo = min_nan(lo, __ldcg(r.partials + r.nblocks + i));
        hi = max_nan(hi, __ldcg(r.partials + i));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min_nan(lo, __shfl_down_sync(0xffffffffu, lo, o));
        hi = max_nan(hi, __shfl_down_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        fin[threadIdx.x >> 5] = lo;
        fin[8 + (threadIdx.x >> 5)] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            lo = min_nan(lo, fin[w]);
            hi = max_nan(hi, fin[8 + w]);
        }
        put_result(r, 0, lo);
        put_result(r, 1, hi);
    }
}
#endif

// ---- semi-Lagrangian and FD kernels (sl_kernels.cu) ----
// CTAs of the tiled gathers on an n1 x n2 x n3 grid (entries of a tile-bounds table)
size_t tiled_grid_tiles(int n1, int n2, int n3);
// Pointers typed void* hold scalar fields in the storage type `sto` (FP32,
// FP16 or BF16); float* ones are always FP32 (displacements, velocities,
// vector work fields).
// tb: the tile-bounds table of d written by launch_backtrace (or null: the
// gathers reduce the bounds themselves)
void launch_interp(const Grid& g, int order, const void* f, const float* d, void* out, Storage sto,
                   cudaStream_t st, const int4* tb = nullptr);
// nf FP32 fields [nf][N] at one displacement into out [nf][N]
void launch_interp_fields(const Grid& g, int order, const float* f, int nf, const float* d, float* out,
                          cudaStream_t st);
// CTAs of the tiled gathers that took the global-memory path (device-wide counter)
cudaError_t gather_fallback_tiles(unsigned long long* count, bool reset);
// tb (may be null): also write the tile-bounds table of d (2 int4 per tile of
// the tiled grid)
void launch_backtrace(const Grid& g, int order, const float* v, const float* vc, float dt, int sign, float* d,
                      cudaStream_t st, int4* tb = nullptr);
// One SL step of Eq. (4): lam = Heun(lam_next(X+), div v(X+), div v).
void launch_adj_step(const Grid& g, int order, const void* lam_next, const float* dA, const void* divv,
                     const void* divXp, float dt, void* lam, Storage sto, cudaStream_t st,
                     const int4* tb = nullptr);
// f^j = -vt . grad m^j for j = 0..nt: q0 = coef0 f^0, F + j N <- f^j (j >= 1).
void launch_inc_sources(const Grid& g, const float* vt, const void* gm, int nt, float coef0, void* q0,
                        void* F, Storage sto, cudaStream_t st);
// out (+)= sum_j w_j lam^j grad m^j (lam slots j N, trapezoid weights w_end / w_mid).
// as launch_inc_sources / launch_body, with grad m^j computed from the stored states m (FD8)
void launch_inc_sources_fd(const Grid& g, const float* vt, const void* m, int nt, float coef0, void* q0, void* F,
                           Storage sto, cudaStream_t st);
void launch_body_fd(const Grid& g, const void* lam, const void* m, int nt, float w_end, float w_mid, int accumulate,
                    float* out, Storage sto, cudaStream_t st);
void launch_body(const Grid& g, const void* lam, const void* gm, int nt, float w_end, float w_mid,
                 int accumulate, float* out, Storage sto, cudaStream_t st);
// q = q_prev(X) + coef F;   lam = -(q_prev(X) + coef F)  (F may alias lam)
void launch_inc_step_src(const Grid& g, int order, const void* q_prev, const float* d, const void* F,
                         float coef, void* q, Storage sto, cudaStream_t st, const int4* tb = nullptr);
void launch_inc_last_src(const Grid& g, int order, const void* q_prev, const float* d, const void* F,
                         float coef, void* lam, Storage sto, cudaStream_t st, const int4* tb = nullptr);
#ifndef CLAIRE_INC_FUSED
#define CLAIRE_INC_FUSED 1  // incremental state steps form their sources in place when grad m^j is stored
#endif
// With grad m^j stored: q0 = coef0 f^0, and the steps above with the source
// f^{j+1} = -vt . grad m^{j+1} formed at each arrival point (gm: grad m^{j+1},
// 3N values in `sto`), so no pass writes the sources of every level.
void launch_inc_source0(const Grid& g, const float* vt, const void* gm, float coef0, void* q0, Storage sto,
                        cudaStream_t st);
void launch_inc_step_grad(const Grid& g, int order, const void* q_prev, const float* d, const float* vt,
                          const void* gm, float coef, void* q, Storage sto, cudaStream_t st, const int4* tb = nullptr);
void launch_inc_last_grad(const Grid& g, int order, const void* q_prev, const float* d, const float* vt,
                          const void* gm, float coef, void* lam, Storage sto, cudaStream_t st,
                          const int4* tb = nullptr);
// out = a - b; conversions FP32 <-> storage
void launch_sub(const void* a, const void* b, void* out, size_t n, Storage sto, cudaStream_t st);
void launch_to_storage(const float* in, void* out, size_t n, Storage sto, cudaStream_t st);
void launch_from_storage(const void* in, float* out, size_t n, Storage sto, cudaStream_t st);
void launch_map_step(const Grid& g, int order, const float* u_prev, const float* d, float* u,
                     cudaStream_t st);
void launch_fd8_grad(const Grid& g, const void* f, void* out, Storage sto, cudaStream_t st);
void launch_fd8_div(const Grid& g, const float* v, void* out, Storage sto, cudaStream_t st);
// totals: minimum at red.out[0], maximum at red.out[1] (scale unused)
void launch_detj_minmax(const Grid& g, const float* u, const Reduction& red, cudaStream_t st);

// Whether a context of GPU `device` may form a result of n floats at dst itself
// (a: dst's pointer attributes): managed memory or memory of that GPU (kernels of
// this GPU cannot store to another's unless peer access happens to be enabled, a
// copy can), at a 16-byte boundary (what the transforms and the vector loads
// need), sharing no byte with the input of m floats.
inline bool forms_in_place(const cudaPointerAttributes& a, int device, const void* dst, size_t n, const void* in,
                           size_t m)
{
    const uintptr_t d = reinterpret_cast<uintptr_t>(dst), i = reinterpret_cast<uintptr_t>(in);
    if ((d & 15u) || (d < i + m * sizeof(float) && i < d + n * sizeof(float))) return false;
    return a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == device);
}

// ---- context accessors for host-side drivers in other units (engine.cu) ----
cudaStream_t ctx_stream(const claire_ctx* c);
size_t ctx_points(const claire_ctx* c);
claire_status ctx_fail(claire_ctx* c, claire_status st, const char* msg);

// spectra of ncomp fields divided by N times the sampled cubic B-spline symbol (vec_kernels.cu)
void launch_bspline_scale(const Grid& g, cufftComplex* spec, size_t M, int ncomp, cudaStream_t st);

// ---- reverse-mode transport (vjp.cu) ----
// dbar_c += mbar * d_c I[m](X)   (interpolant gradient at x + d, grid units);
// first: dbar is written instead of added to
void launch_grad_accum(const Grid& g, int order, const float* m, const float* d, const float* mbar, float* dbar,
                       bool first, cudaStream_t st);
// Whether the scatter-transpose of a tile fits its shared-memory box: first nodes
// of the points' stencils in [a, z] per axis, stencils of m nodes, cap nodes in
// the box.  Displacements are clamped to 2^20 cells only, so an extent may reach
// 2^21: each is compared before they are multiplied (the product of three would
// not fit 63 bits).
__host__ __device__ inline bool scatter_box_fits(const int a[3], const int z[3], int m, int cap, int e[3])
{
    bool fits = true;
    for (int c = 0; c < 3; ++c) {
        e[c] = z[c] - a[c] + m;  // |a|, |z| below 2^30
        fits = fits && e[c] >= m && e[c] <= cap;
    }
    return fits && static_cast<long long>(e[0]) * e[1] * e[2] <= cap;
}

// acc += fixed-point(W(x + disp)^T yv), scale from *maxabs = max |yv| (device);
// disp = d, or -sdt v / h when d is null
cudaError_t launch_scatter_fixed(const Grid& g, int order, const float* yv, const float* d, const float* v, float sdt,
                                 const double* maxabs, unsigned long long* acc, cudaStream_t st);
// out = mult ((accumulate ? out : 0) + acc / scale); clears acc
void launch_fixed_to_float(unsigned long long* acc, const double* maxabs, int accumulate, float mult, float* out,
                           size_t n, cudaStream_t st);
// predictor terms of the velocity cotangent (grid units): ubar, Ubar from dbar
// y = a (y + x)
void launch_scale_add(float* y, float a, const float* x, size_t n, cudaStream_t st);
void launch_predictor_terms(const Grid& g, int order, const float* v, const float* vc, float dt, const float* dbar,
                            float* ubar, float* Ubar, cudaStream_t st);
// out[0] = max |x| (NaN: infinity)
void launch_maxabs(const float* x, size_t n, const Reduction& r, cudaStream_t st);

// ---- spectral scaling, vector ops and reductions (vec_kernels.cu) ----
enum SpectralOp { SPEC_REG = 0, SPEC_INV = 1, SPEC_K = 2, SPEC_AINV = 3 };

struct RegParams {
    float beta_v, beta_w;
    int reg;  // 1 = H1 seminorm, 2 = H2 seminorm
};

// Scaling of the three half-spectra xh[c] into yh[c] (may be xh), c = 0..2 (each
// n1 * n2 * (n3/2+1) complex values, stride cstride) by the 3x3 symbol of op,
// times scale (the 1/N of the unnormalised inverse transform); energy (may be
// null): also the total of the quadratic form of the operator.
void launch_spectral(const Grid& g, const cufftComplex* xh, cufftComplex* yh, size_t cstride, SpectralOp op,
                     RegParams rp, float scale, const Reduction* energy, cudaStream_t st);
// total of sum_k wt Re(conj(w) S w), w = vh + alpha xh (xh may be null)
void launch_reg_energy(const Grid& g, const cufftComplex* vh, const cufftComplex* xh, size_t cs, float alpha,
                       RegParams rp, const Reduction& red, cudaStream_t st);

// Device scalars sc of a PCG iteration (FP64).  The kernel that ends a reduction
// also forms what follows from it: start (and the two-level finish) store rz;
// hp forms alpha = rz / pq (0 when pq <= 0 or NaN); update forms beta = rz_new /
// rz and moves rz_new to rz.
constexpr int kPcgRz = 0, kPcgAlpha = 1, kPcgBeta = 2, kPcgSlots = 4;

// PCG direction in Fourier space: ph = z~ + beta ph (first: ph = z~), z~ = M rh, cp = ph.
void launch_spectral_direction(const Grid& g, const cufftComplex* rh, cufftComplex* ph, cufftComplex* cp,
                               size_t cstride, const double* sc, int first, SpectralOp op, RegParams rp,
                               cudaStream_t st);

// Fourier-space PCG (vectors are half spectra scaled by 1/N; totals are
// of sum_k wt Re(conj(a) b), wt the multiplicity of the mode; H p~ = S p~ + scale T, K
// of it if kform, is formed where it is used):
//   start:  r~ = -scale spec, x~ = 0;  totals |r~|^2, <r~, M r~>
//   hp:     totals <p~, H p~> and (second result) alpha
//   update: x~ += alpha p~, r~ -= alpha H p~;  totals as in start, or with zc |r~|^2, <H p~, zc>
void launch_fs_start(const Grid& g, cufftComplex* spec, cufftComplex* rh, cufftComplex* xh, size_t cs,
                     SpectralOp op, RegParams rp, float scale, double* sc, const Reduction& red, cudaStream_t st);
void launch_fs_hp(const Grid& g, const cufftComplex* T, const cufftComplex* ph, size_t cs, int kform, RegParams rp,
                  float scale, double* sc, const Reduction& red, cudaStream_t st);
void launch_fs_update(const Grid& g, const cufftComplex* T, const cufftComplex* ph, cufftComplex* xh,
                      cufftComplex* rh, const cufftComplex* zc, size_t cs, int kform, SpectralOp op, RegParams rp,
                      float scale, double* sc, const Reduction& red, cudaStream_t st);

// two-level zero-velocity preconditioner (coarse grid gc of the fine grid gf; cs* = component strides)
void launch_mean_levels(const void* m, int nt, float w_end, float w_mid, size_t N, float* out, Storage sto,
                        cudaStream_t st);
void launch_cscale(cufftComplex* x, size_t n, float s, cudaStream_t st);
void launch_tl_restrict(const Grid& gf, const cufftComplex* F, size_t csf, const Grid& gc, cufftComplex* out,
                        size_t csc, float invN, cudaStream_t st);
// coarse preconditioner correction: gbar_c [3][n] <- sqrt(max(w, 0)) gbar_c
void launch_tl_weight(float* gbar_c, const float* w, size_t n, cudaStream_t st);
void launch_tl_start(const Grid& gf, const cufftComplex* rf, size_t csf, const Grid& gc, cufftComplex* rh,
                     cufftComplex* xh, cufftComplex* ph, cufftComplex* cp, size_t cs, SpectralOp op, RegParams rp,
                     float rscale, double* sc, const Reduction& red, cudaStream_t st);
void launch_tl_rank1(const float* gbar, float* p, size_t Nc, cudaStream_t st);
// second result: the breakdown flag (0; 1: pq <= 0; 2: pq is NaN)
void launch_tl_hp(const Grid& gc, const cufftComplex* T, const cufftComplex* ph, size_t cs, int kform, RegParams rp,
                  float scale, double* sc, const Reduction& red, cudaStream_t st);
void launch_tl_update(const Grid& gc, const cufftComplex* T, const cufftComplex* ph, cufftComplex* xh,
                      cufftComplex* rh, size_t cs, int kform, SpectralOp op, RegParams rp, float scale, double* sc,
                      const Reduction& red, cudaStream_t st);
void launch_dir_stored(const Grid& g, const cufftComplex* zh, cufftComplex* ph, cufftComplex* cp, size_t cs,
                       float beta, int first, cudaStream_t st);
void launch_tl_finish(const Grid& gf, const cufftComplex* rf, cufftComplex* zf, size_t csf, const Grid& gc,
                      const cufftComplex* xc, size_t csc, SpectralOp op, RegParams rp, float rscale, double* sc,
                      const Reduction& red, cudaStream_t st);
// Deterministic FP64 reductions (struct Reduction): totals at red.out
void launch_dot(const float* x, const float* y, size_t n, const Reduction& red, cudaStream_t st);
void launch_sqdiff(const void* a, const void* b, size_t n, Storage sto, const Reduction& red, cudaStream_t st);
void launch_maxnorm3(const float* v, size_t N, const Reduction& red, cudaStream_t st);
// Dice counts: |a >= t| and |b >= t| (both = 0) or |(a >= t) and (b >= t)| (both = 1)
void launch_count(const float* a, const float* b, size_t n, float t, int both, const Reduction& red, cudaStream_t st);

// y = a x + y
void launch_axpy(float a, const float* x, float* y, size_t n, cudaStream_t st);
// z = x + a y
void launch_xpay(const float* x, float a, const float* y, float* z, size_t n, cudaStream_t st);

}  // namespace claire
