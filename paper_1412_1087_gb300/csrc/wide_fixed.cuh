// 64-bit deposits in integer arithmetic.
//
// A contribution of a double-precision deposit is q w rounded to a whole
// number of fixed-point units, w the product of D one-dimensional TSC
// weights.  Formed in FP64 that is a product and a conversion to int64 for
// each of the 4 3^D values of a deposit, both on the FP64 pipe, where this
// GPU issues one warp instruction in 17 cycles per SM; a 64 x 64 -> upper 64
// bit product on the integer pipe takes 5.  So q is converted once per
// channel and everything after it is integer:
//
//   O   = o 2^63, the offset in the cell (the upper bits of o's mantissa);
//   W   = the three weights in units of 2^-63: (1-o)^2/2 and o^2/2 are the
//         upper halves of 64-bit squares and the centre weight is what is
//         missing to 1, so the weights add up to 1 exactly;
//   Q   = round(q 2^SH) as sign and magnitude;
//   v   = round((Q Wz) Wxy), each product rounded to nearest at its last
//         kept bit: SH extra bits of Q and 63 - (SH - 3) bits of Wxy put the
//         errors of the factors below a hundredth of the final rounding.
//
// Every value depends on the particle alone and is rounded once, so sums do
// not depend on the order or on the kernel that adds them.
#pragma once

#include "device_common.cuh"

namespace mhdpic {

// round(a b / 2^64) for b < 2^63 (schoolbook product of 32-bit halves, the
// rounding half added to the middle column)
__device__ __forceinline__ uint64_t mul_hi_round(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t p = (uint64_t)al * bl;
    const uint64_t m1 = (uint64_t)ah * bl + (p >> 32);
    const uint64_t m2 = (uint64_t)al * bh + ((uint64_t)(uint32_t)m1 + 0x80000000ull);
    return (uint64_t)ah * bh + (m1 >> 32) + (m2 >> 32);
}

// o 2^63 for o in [0, 1], truncated
__device__ __forceinline__ uint64_t frac63(double o)
{
    const uint64_t b = (uint64_t)__double_as_longlong(o);
    const int e = (int)((b >> 52) & 0x7ff);
    const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const int sh = e - 1012;   // o = m 2^(e - 1075)
    if (sh >= 0)
        return sh < 12 ? m << sh : 0ull;
    return sh > -53 ? m >> -sh : 0ull;
}

__device__ __forceinline__ uint64_t frac63(float o)
{
    const uint32_t b = __float_as_uint(o);
    const int e = (int)((b >> 23) & 0xff);
    const uint64_t m = (b & 0x7fffffu) | 0x800000u;
    const int sh = e - 87;     // o = m 2^(e - 150)
    if (sh >= 0)
        return sh < 41 ? m << sh : 0ull;
    return sh > -24 ? m >> -sh : 0ull;
}

// TSC weights of cells i-1, i, i+1 in units of 2^-63 (tsc_from_offset)
template <typename R>
__device__ __forceinline__ void wide_tsc(R o, uint64_t w[3])
{
    const uint64_t O = frac63(o), A = (1ull << 63) - O;
    w[0] = __umul64hi(A, A);
    w[2] = __umul64hi(O, O);
    w[1] = (1ull << 63) - w[0] - w[2];
}

// q 2^SH as a magnitude and a sign mask (0 or all ones); q already carries the
// fixed-point scale
template <int SH>
__device__ __forceinline__ void wide_q(double q, uint64_t &mag, uint64_t &sign)
{
    const long long i = __double2ll_rn(q * (double)(1 << SH));
    sign = (uint64_t)(i >> 63);
    mag = ((uint64_t)i ^ sign) - sign;
}

// Products of the x and y weights as the deposits take them (SH extra bits of
// the quantity cancel against the units of the three weights).
template <int SH>
__device__ __forceinline__ uint64_t wide_pair(uint64_t wa, uint64_t wb)
{
    return __umul64hi(wa, wb) >> (SH - 3);
}

// The signed contribution of |Q| wz (from mul_hi_round(Q, wz)) and a pair.
__device__ __forceinline__ unsigned long long wide_value(uint64_t qz, uint64_t pair, uint64_t sign)
{
    return (mul_hi_round(qz, pair) ^ sign) - sign;
}

}  // namespace mhdpic
