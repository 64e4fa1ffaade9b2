// Kernel launchers of libclaire with inputs that its entry points do not take
// directly (test infrastructure; built and loaded by tests/test_gpu_direct.py).
// Each function returns 0 or a cudaError_t.
#include "detj.cuh"
#include "internal.h"

using namespace claire;

namespace {

Grid make_grid(int n1, int n2, int n3)
{
    const double two_pi = 6.283185307179586476925286766559;
    Grid g;
    g.n1 = n1; g.n2 = n2; g.n3 = n3;
    g.n23 = n2 * n3;
    g.N = static_cast<uint32_t>(n1) * n2 * n3;
    g.h1 = static_cast<float>(two_pi / n1); g.h2 = static_cast<float>(two_pi / n2); g.h3 = static_cast<float>(two_pi / n3);
    g.ih1 = static_cast<float>(n1 / two_pi); g.ih2 = static_cast<float>(n2 / two_pi); g.ih3 = static_cast<float>(n3 / two_pi);
    return g;
}

__global__ void k_det_bounds(const float* diff, const float* ih, int n, float* lo, double* det, float* hi)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    float e[3][3];
    for (int c = 0; c < 3; ++c)
        for (int a = 0; a < 3; ++a) e[c][a] = __fmul_rn(diff[(3 * c + a) * n + p], ih[a]);
    det_bounds(e, lo[p], hi[p]);
    det[p] = det_exact(e);
}

}  // namespace

// Bounds and FP64 value of det(I + e), e = diff ih: diff device [9][n], ih device [3].
extern "C" int direct_det_bounds(const float* diff, const float* ih, int n, float* lo, double* det, float* hi)
{
    k_det_bounds<<<(n + 255) / 256, 256>>>(diff, ih, n, lo, det, hi);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? cudaDeviceSynchronize() : e;
}

// Extrema of det(I + grad u), u device [3][N]; blocks CTAs; out: host, minimum and maximum.
extern "C" int direct_detj(int n1, int n2, int n3, const float* u, int blocks, double* out)
{
    double* dev = nullptr;  // partials, two results, the ticket
    cudaError_t e = cudaMalloc(&dev, (2 * blocks + 3) * sizeof(double));
    if (e != cudaSuccess) return e;
    e = cudaMemset(dev, 0, (2 * blocks + 3) * sizeof(double));
    if (e == cudaSuccess) {
        Reduction red{dev, blocks, 1.0, dev + 2 * blocks, nullptr, reinterpret_cast<unsigned*>(dev + 2 * blocks + 2)};
        launch_detj_minmax(make_grid(n1, n2, n3), u, red, nullptr);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpy(out, dev + 2 * blocks, 2 * sizeof(double), cudaMemcpyDeviceToHost);
    }
    cudaFree(dev);
    return e;
}

// out = mult ((accumulate ? out : 0) + acc / scale(maxabs)); all arrays on the device.
extern "C" int direct_fixed_to_float(unsigned long long* acc, const double* maxabs, int accumulate, float mult, float* out,
                                     long long n)
{
    launch_fixed_to_float(acc, maxabs, accumulate, mult, out, static_cast<size_t>(n), nullptr);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? cudaDeviceSynchronize() : e;
}
