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

// x >= 0, sign bit clear (a set one, -0 included, reads as a huge value),
// truncated to FP32 with integer operations; 0 below FP32's normal range, the
// largest finite value above it (and for NaN).
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
// within an ulp (1.4 of 10 000 random ones differ from the rounded reciprocal),
// where the division takes 5 to 6.
__device__ __forceinline__ double rcp_newton(double d)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// Correctly rounded a / b for a divisor whose correctly rounded reciprocal rb
// is at hand (Markstein 1990): two quotient corrections by exact remainders,
// five FP64 operations where the division takes 8 to 9.  rb = 0 marks a
// divisor outside 2^+-200; those, and dividends outside 2^+-700 other than 0,
// are divided outright (no remainder may underflow).
__device__ __forceinline__ double div_known(double a, double b, double rb)
{
    const unsigned ea = ((unsigned)__double2hiint(a) >> 20) & 0x7ffu;
    const bool zero = (((unsigned)__double2hiint(a) << 1) | (unsigned)__double2loint(a)) == 0u;
    if (rb == 0.0 || !(zero || ea - 323u < 1400u)) return __ddiv_rn(a, b);
    double q = __dmul_rn(a, rb);
    q = __fma_rn(__fma_rn(-b, q, a), rb, q);
    return __fma_rn(__fma_rn(-b, q, a), rb, q);
}
__device__ __forceinline__ double known_rcp(double b)
{
    const unsigned eb = ((unsigned)__double2hiint(b) >> 20) & 0x7ffu;
    return eb - 823u < 400u ? __ddiv_rn(1.0, b) : 0.0;
}

__device__ __forceinline__ float abs_of(float x) { return fabsf(x); }
__device__ __forceinline__ double abs_of(double x) { return fabs(x); }
__device__ __forceinline__ float max_of(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double max_of(double a, double b) { return fmax(a, b); }

// One warp: a pixel's squared weights into s_w2[4], the caller's or Section
// 5.4's inverse-max weights in FP64 (the extrema in the cube's own type).
template <class RO>
__device__ __forceinline__ void weights64(const RO *o, int nl, const double *w_user, int pix, double *s_w2)
{
    const int lane = threadIdx.x & 31;
    if (w_user) {
        if (lane < 4) {
            const double w = w_user[(size_t)pix * 4 + lane];
            s_w2[lane] = w * w;
        }
        return;
    }
    RO imax = -INFINITY, nmin = -INFINITY, m[3] = {0, 0, 0};  // nmin = -min I
    for (int j = lane; j < nl; j += 32) {
        imax = max_of(imax, o[j]);
        nmin = max_of(nmin, -o[j]);
#pragma unroll
        for (int s = 0; s < 3; ++s) m[s] = max_of(m[s], abs_of(o[(s + 1) * nl + j]));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        imax = max_of(imax, __shfl_xor_sync(0xffffffffu, imax, off));
        nmin = max_of(nmin, __shfl_xor_sync(0xffffffffu, nmin, off));
#pragma unroll
        for (int s = 0; s < 3; ++s) m[s] = max_of(m[s], __shfl_xor_sync(0xffffffffu, m[s], off));
    }
    if (lane < 4) {
        const double top = (double)imax;
        const double d = lane == 0 ? top + (double)nmin : (double)(lane == 1 ? m[0] : lane == 2 ? m[1] : m[2]);
        const double fl = 1e-6 * fabs(top);
        const double dd = d > fl ? d : fl;
        const double w = dd > 0.0 ? 1.0 / dd : 0.0;
        s_w2[lane] = w * w;
    }
}

// The warp sums of four FP64 values at once: the butterfly's additions (lane
// distances 16, 8, 4, 2, 1), but each lane keeps only the values it goes on
// with, so that 6 additions do what 20 would.  Sum s lands on the eight lanes
// with lane / 8 == s, the same bits that four butterflies give.
__device__ __forceinline__ double warp_sum4(double v0, double v1, double v2, double v3)
{
    const bool h16 = threadIdx.x & 16, h8 = threadIdx.x & 8;
    const double x0 = (h16 ? v2 : v0) + __shfl_xor_sync(0xffffffffu, h16 ? v0 : v2, 16);
    const double x1 = (h16 ? v3 : v1) + __shfl_xor_sync(0xffffffffu, h16 ? v1 : v3, 16);
    double v = (h8 ? x1 : x0) + __shfl_xor_sync(0xffffffffu, h8 ? x0 : x1, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

}  // namespace genesis
