// det(I + e) of a 3 x 3 matrix e of FP32 differences: in FP64, and in FP32 with
// bounds, for the filter of k_detj_minmax (sl_kernels.cu).
#pragma once

#include <cuda_runtime.h>

namespace claire {

__device__ __forceinline__ double det_exact(const float e[3][3])
{
    double F[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int a = 0; a < 3; ++a) F[c][a] = e[c][a];
#pragma unroll
    for (int c = 0; c < 3; ++c) F[c][c] += 1.0;
    return F[0][0] * (F[1][1] * F[2][2] - F[1][2] * F[2][1]) -
           F[0][1] * (F[1][0] * F[2][2] - F[1][2] * F[2][0]) +
           F[0][2] * (F[1][0] * F[2][1] - F[1][1] * F[2][0]);
}

// dlo <= det_exact(e) <= dhi, unless something overflows or is NaN (then not both
// are finite).  The half width is 4e-6 m^3 + 1e-36, m the largest |entry| of I + e:
// each of the six triple products (at most m^3) carries three entry roundings,
// two products and up to three sums of relative error 2^-24, together below
// 6 * 8 * 2^-24 m^3 = 2.9e-6 m^3; the constant covers products that underflow.
// An entry rounding is relative to the entry only if 1 + e is taken of the
// rounded e, as det_exact does: where e is a product, the caller rounds it
// (__fmul_rn), and the sum here is not left to the compiler to fuse with it: fused, it
// would be off by 2^-25 whatever the size of 1 + e, six times the bound at m = 0.01.
__device__ __forceinline__ void det_bounds(const float e[3][3], float& dlo, float& dhi)
{
    float f[3][3], m = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            f[c][a] = a == c ? __fadd_rn(1.0f, e[c][a]) : e[c][a];
            m = fmaxf(m, fabsf(f[c][a]));
        }
    const float det = f[0][0] * (f[1][1] * f[2][2] - f[1][2] * f[2][1]) -
                      f[0][1] * (f[1][0] * f[2][2] - f[1][2] * f[2][0]) +
                      f[0][2] * (f[1][0] * f[2][1] - f[1][1] * f[2][0]);
    const float E = fmaf(4e-6f * m * m, m, 1e-36f);
    dlo = det - E;
    dhi = det + E;
}

}  // namespace claire
