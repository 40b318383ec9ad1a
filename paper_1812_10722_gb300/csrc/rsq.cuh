// Reciprocal square roots of the kernels (squared distances, far above the denormal range).
#pragma once

#include <cuda_runtime.h>

namespace lspr {

// FP32 1/sqrt(x): the hardware approximation with denormal inputs flushed (squared
// distances here are far above the denormal range), which spares the denormal fix-up
// instructions that rsqrtf carries without -ftz
static __device__ __forceinline__ float rsq(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// FP64 1/sqrt(x): the hardware's FP64 approximation (relative error e < 2^-19) as the seed and one
// third-order (Householder) step: 1/sqrt(x) = y (1 - h)^(-1/2) with h = 1 - x y^2, and the binomial series
// up to h^2 gives y <- y + y h (1/2 + 3/8 h), which leaves 5/16 h^3 = ~2.5 e^3 (below half a
// unit in the last place); five FP64 operations and no conversions through FP32 (one Newton step from
// an FP32 seed left ~2e-14).  FP64 products: 20480 panels by treecode 5528 -> 5317 us, 1280 panels
// direct 419 -> 399, their error against 64 bits 2.6e-15 -> 9e-16.
static __device__ __forceinline__ double rsq(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = fma(-x * y, y, 1.0);
    return fma(y * h, fma(0.375, h, 0.5), y);
}

}  // namespace lspr
