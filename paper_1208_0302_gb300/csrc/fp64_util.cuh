// Replacements for operations that take the FP64 pipe, which issues a warp
// instruction every 16 clocks of an SM (sm_103a).
#pragma once

#include <cuda_runtime.h>

namespace genesis {

// Exact FP32 -> FP64 widening of normal numbers with integer operations (the
// conversion instruction takes the FP64 pipe).
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u) return (double)x;  // zero, subnormal, infinity, NaN
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// x >= 0 truncated to FP32 with integer operations; 0 below FP32's normal
// range, the largest finite value above it (and for NaN).
__device__ __forceinline__ float narrow(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if (hi < 0x38100000u) return 0.0f;
    if (hi >= 0x47f00000u) return 3.402823466e38f;
    return __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
}

// 1 / d for normal d: the hardware's approximate reciprocal r (relative error
// e below 2^-20) and one step of the third-order Newton iteration r (1 + e +
// e^2), whose remaining error e^3 is below 2^-60: three FP64 operations and
// within an ulp, where the division takes 5 to 6.
__device__ __forceinline__ double rcp_newton(double d)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

}  // namespace genesis
