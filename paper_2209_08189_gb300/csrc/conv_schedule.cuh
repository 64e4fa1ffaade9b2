// Issue order of the stacked convolution's MMAs (net_kernels.cu), shared with the
// host test of it.
#pragma once

#include <cuda_runtime.h>

namespace claire {

// With the kd taps stacked along N, halo plane sd (0 .. bdc + 1) of a brick feeds
// the output planes z = sd - kd that lie in the brick: nz planes from z0 on, whose
// columns are adjacent, so one MMA covers them.  Block 0 of its B operand is
// that of z0, i.e. of tap kd = sd - z0.
struct StackedPlane {
    int z0, nz;
};

__host__ __device__ inline StackedPlane stacked_plane(int bdc, int sd)
{
    const int z0 = sd < 2 ? 0 : sd - 2;
    return {z0, (sd < bdc ? sd + 1 : bdc) - z0};
}

// The order of two MMAs is defined only where they have the same accumulator and
// the same shape, and planes one or two apart overlap in their columns with
// other bases and, at the brick's edges, other widths.  So the planes are issued in
// three groups, sd = g mod 3, whose members write disjoint columns; the issuing
// thread waits for a group before it issues the next.  Group 0 writes every
// column, so its first product of the first slice overwrites and all others add.
// (One output plane: every MMA has the same accumulator and shape, no waits.)
constexpr int kStackGroups = 3;

__host__ __device__ inline bool stacked_wait(int bdc, int group) { return group > 0 && bdc > 1; }

}  // namespace claire
