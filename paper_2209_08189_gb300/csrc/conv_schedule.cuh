// Issue order of the stacked convolution's MMAs (net_kernels.cu), shared with the
// host test of it.
#pragma once

#include <cuda_runtime.h>

namespace claire {

// With the kd taps stacked along N, halo plane sd (0 .. bdc + 1) of a brick feeds
// the output planes z = sd - kd that lie in the brick: nz planes from z0 on, whose
// columns are adjacent, so one MMA covers them.  Block 0 of its B operand is
// that of z0, i.e. of tap kd = sd - z0.
//
// The planes are issued in the order of sd, so that every output plane sums its depth
// taps kd = 0, 1, 2 as the unstacked kernel does (the same bits; an order that
// differs from plane to plane moves roundings, and with them the signs that the
// leaky ReLU's backward pass reads).
struct StackedPlane {
    int z0, nz;
};

__host__ __device__ inline StackedPlane stacked_plane(int bdc, int sd)
{
    const int z0 = sd < 2 ? 0 : sd - 2;
    return {z0, (sd < bdc ? sd + 1 : bdc) - z0};
}

// The order of two MMAs is defined only where they have the same accumulator and
// the same shape, and neighbouring planes overlap in their columns with another
// base or, at the brick's edges, another width: the issuing thread waits for
// plane sd - 1 before it issues such a plane sd.  The waits are hidden where the
// brick leaves room for four CTAs per SM and cost up to a sixth where it leaves
// three: 128^3 x 4, 16 -> 16 channels, eight planes 302 us (257 without them), four
// planes 373 either way; 64^3 x 4, 96 -> 32 channels 270 us (257).  Two interleaved
// chains of four planes, whose waits overlap, need two planes more and took 319;
// three groups of planes that do not overlap (two waits) took 266, but sum the depth taps
// in orders that differ from plane to plane.
__host__ __device__ inline bool stacked_wait(int bdc, int sd)
{
    if (sd == 0) return false;
    const StackedPlane a = stacked_plane(bdc, sd - 1), b = stacked_plane(bdc, sd);
    return a.z0 != b.z0 || a.nz != b.nz;
}

}  // namespace claire
