// rb_fp64.cuh -- reciprocal and reciprocal square root in FP64 from the
// hardware's coarse estimates.  On GB300 an FP64 instruction holds the SM's
// FP64 pipe 16 cycles per warp, and a division or an rsqrt() call issues two to
// three times as many of them.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace rb {

#ifdef __CUDACC__
// 1/x: with y the estimate and h = 1 - x y, 1/x = y / (1 - h) =
// y (1 + h + h^2 + ...), taken to h^2 (four FP64 operations).  x near the ends
// of the exponent range, where the estimate flushes to zero, takes the
// division.
__device__ __forceinline__ double rcp64(double x) {
    const int e = (int)((__double_as_longlong(x) >> 52) & 0x7ff);
    if (e < 64 || e > 1982) return __ddiv_rn(1.0, x);
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = fma(-x, y, 1.0);
    return fma(y, fma(h, h, h), y);
}

// 1/sqrt(x): with y the estimate and h = 1 - x y^2, 1/sqrt(x) =
// y (1 - h)^(-1/2) = y (1 + h/2 + 3 h^2/8 + ...), taken to h^2 (five FP64
// operations).  Zero, subnormal numbers (the estimate reads them as zero),
// negative numbers, infinity and NaN take the library's function.
__device__ __forceinline__ double rsqrt64(double x) {
    // biased exponent and sign in one test: 1 .. 2046 of a positive number
    if ((uint32_t)(__double2hiint(x) - 0x00100000) >= 0x7fe00000u) return rsqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = fma(-x * y, y, 1.0);
    return fma(y * h, fma(h, 0.375, 0.5), y);
}
#endif

}  // namespace rb
