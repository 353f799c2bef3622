// Shared by the two kernels of the second-order form (wlr2.cu, wlr2_gram.cu).
#pragma once

#include <cuda_runtime.h>

namespace esim {

struct W2Params {
    int W, H, F, r, T, rgb, tiles_x;
    float h, log_eps, ridge;
    const float* radiance;   // [F][C][H][W]
    const float* features;   // [F][7][H][W]
    const float* bandwidth;  // [7]
    float4* packed;          // [F][2][H][W]: (y, normal xyz), (depth, albedo rgb)
    float* alpha;            // [F][H][W]
    // wlr2.cu
    int tw, gx, gy;          // pixel group tw x (16 / tw), groups across and down
    int part;                // neighbour pairs per partial sum
    int flush;               // some window has more pairs than that
    int seg;                 // neighbour pairs per table
};

// The packed frames -> alpha by the Gram in registers; cudaErrorInvalidValue: too many pixels.
cudaError_t launch_wlr2_gram(const W2Params& p, cudaStream_t s);

namespace {

constexpr float kExp2Scale = 0.84932180028801904272f;  // sqrt(log2(e) / 2)

// Quadratic unknown q (0..44) -> feature pair (a, b), a <= b, a-major order.
__host__ __device__ constexpr int pair_a(int q)
{
    int a = 0;
    while (q >= 9 - a) { q -= 9 - a; ++a; }
    return a;
}
__host__ __device__ constexpr int pair_b(int q)
{
    int a = 0;
    while (q >= 9 - a) { q -= 9 - a; ++a; }
    return a + q;
}

}  // namespace
}  // namespace esim
