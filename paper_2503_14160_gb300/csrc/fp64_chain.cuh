// Reciprocals and reciprocal square roots in FP64 for kernels whose time is a chain of dependent
// FP64 operations. On this part an FP64 instruction, a conversion between FP32 and FP64
// included, holds its scheduler's FP64 unit for 64 cycles and its result waits as long
// (measured with one warp), so the conversions are done on the bits by a few integer
// instructions, with the same rounding.
#pragma once

#include <cstdint>

namespace cp {

// a rounded to the nearest float (ties to even), for |a| in float's normal range: the exponent
// rebiased, the 52-bit fraction cut to 23 bits and rounded up on the cut part. Outside the
// range the result is unspecified.
static __device__ __forceinline__ float narrow_bits(double a)
{
    const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
    const uint32_t sign = hi & 0x80000000u;
    uint32_t f = (((hi & 0x7FFFFFFFu) - 0x38000000u) << 3) | (lo >> 29);
    f += (lo & 0x1FFFFFFFu) + (f & 1u) > 0x10000000u ? 1u : 0u;
    return __uint_as_float(f | sign);
}

// The double equal to the normal float y.
static __device__ __forceinline__ double widen_bits(float y)
{
    const uint32_t u = __float_as_uint(y);
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// a as a float, or 0 where a is not a positive number inside (1e-30, 1e30), the range of the
// short forms below.
static __device__ __forceinline__ float short_seed(double a)
{
    const uint32_t hi = (uint32_t)__double2hiint(a);
    const float f = narrow_bits(a);   // valid for exponents of float's normal range
    return hi - 0x38100000u < 0x47E00000u - 0x38100000u && f > 1e-30f && f < 1e30f ? f : 0.f;
}

// 1/a and 1/sqrt(a) for a > 0: a float seed refined by two Newton-Raphson steps in FP64
// (quadratic convergence: 23 -> 46 -> 92 bits). Arguments outside the range take the IEEE
// operations instead.
static __device__ __forceinline__ double recip_newton(double a)
{
    const float f = short_seed(a);
    if (f == 0.f) return 1.0 / a;
    double y = widen_bits(__frcp_rn(f));
    y = fma(y, fma(-a, y, 1.0), y);
    y = fma(y, fma(-a, y, 1.0), y);
    return y;
}

static __device__ __forceinline__ double rsqrt_newton(double a)
{
    const float f = short_seed(a);
    if (f == 0.f) return 1.0 / sqrt(a);
    double y = widen_bits(rsqrtf(f));
    // a / 2 by its exponent
    const double h = __hiloint2double(__double2hiint(a) - 0x00100000, __double2loint(a));
    y = y * fma(-h * y, y, 1.5);
    y = y * fma(-h * y, y, 1.5);
    return y;
}

}  // namespace cp
