// Double-precision reciprocals and reciprocal square roots with few FP64
// instructions, for kernels that the FP64 pipe bounds (one warp instruction
// in 17 cycles per SM on this GPU, conversions to and from double included).
//
// A single-precision estimate (relative error below 2^-21) is refined by one
// third-order Newton (Householder) step, from 1/d = r / (1 - e) with
// e = 1 - d r, and 1/sqrt(s) = y (1 - e)^(-1/2) with e = 1 - s y^2:
// the terms left out are below 2^-60, so the results are within about one
// unit in the last place.  Arguments whose exponent does not fit a normal
// float, zero, infinities and NaN take the ordinary division and square root.
#pragma once

#include <stdint.h>

namespace mhdpic {

// true when d is positive with an exponent well inside float's range
__device__ __forceinline__ bool plain_range(double d)
{
    return (uint32_t)__double2hiint(d) - 0x3a000000u < 0x0c000000u;   // 2^-95 .. 2^97
}

// d (plain_range) cut to single precision, and a normal positive float as
// double, by moving the exponent and the mantissa
__device__ __forceinline__ float cut_to_float(double d)
{
    return __int_as_float((int)(((uint32_t)__double2hiint(d) - 0x38000000u) << 3 |
                                ((uint32_t)__double2loint(d) >> 29)));
}

__device__ __forceinline__ double widen(float f)
{
    const uint32_t b = __float_as_uint(f);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

__device__ __forceinline__ double reciprocal(double d)
{
    if (!plain_range(d))
        return 1.0 / d;
    const double r = widen(__fdividef(1.f, cut_to_float(d)));
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

__device__ __forceinline__ double reciprocal_sqrt(double s)
{
    if (!plain_range(s))
        return 1.0 / sqrt(s);
    const double y = widen(rsqrtf(cut_to_float(s)));
    const double e = fma(-(s * y), y, 1.0);
    return fma(y, fma(e, 0.375, 0.5) * e, y);
}

// sqrt(s) from the same estimate, one operation less than s reciprocal_sqrt(s)
__device__ __forceinline__ double square_root(double s)
{
    if (!plain_range(s))
        return sqrt(s);
    const double y = widen(rsqrtf(cut_to_float(s)));
    const double r = s * y;
    const double e = fma(-r, y, 1.0);
    return fma(r, fma(e, 0.375, 0.5) * e, r);
}

// Whole part and rest of s, |s| < 2^31: s + 1.5 2^52 rounded down holds
// floor(s) in its low word.
__device__ __forceinline__ void floor_split(double s, int &whole, double &rest)
{
    constexpr double MAGIC_FLOOR = 6755399441055744.0;
    const double t = __dadd_rd(s, MAGIC_FLOOR);
    whole = __double2loint(t);
    rest = s - (t - MAGIC_FLOOR);
}

}  // namespace mhdpic
