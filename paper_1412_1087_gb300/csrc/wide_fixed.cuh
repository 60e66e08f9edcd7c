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

// ---------------------------------------------------------------------------
// A warp deposits 32 particles straight into global accumulators.  Each lane
// prepares one particle; then 12 lanes of each half warp take one particle
// together, a lane per x node and channel, so that the 64-bit atomics of one
// instruction fall into few 32-byte sectors (what the L2 counts: 210e9 lane
// atomics/s with a sector each, 650e9 with 12 neighbours).
// ---------------------------------------------------------------------------
template <int D>
struct WideGroup {
    static constexpr int YZ = D == 3 ? 9 : 3;
    static constexpr int STRIDE = 33;   // one word beyond the lanes: no two rows on the same banks
    int64_t q[4][STRIDE];
    uint64_t wx[3][STRIDE];
    uint64_t yz[YZ][STRIDE];
    int32_t gx[3][STRIDE];
    int32_t row[YZ][STRIDE];
};

// live: this lane has a particle, with quantities q at their scales, offset o
// and stencil cells gx, gy, gz of a box whose first cell is cell0 and whose x
// and x y extents are n0 and n01.  Cell c, channel k is acc[c cell_stride + k
// chan_stride].  All lanes of the warp call it.
template <int D, int SH, typename R>
__device__ __forceinline__ void group_deposit(WideGroup<D> &s, bool live, const double q[4], const R o[3],
                                              const int gx[3], const int gy[3], const int gz[3], int64_t cell0, int n0,
                                              int n01, unsigned long long *__restrict__ acc, int64_t cell_stride,
                                              int64_t chan_stride)
{
    const int lane = threadIdx.x & 31;
    const unsigned mask = __ballot_sync(0xffffffffu, live);
    if (live) {
        uint64_t wx[3], wy[3], wz[3] = {0ull, 1ull << 63, 0ull};
        wide_tsc(o[0], wx);
        wide_tsc(o[1], wy);
        if (D == 3)
            wide_tsc(o[2], wz);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            s.q[k][lane] = __double2ll_rn(q[k] * (double)(1 << SH));
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            s.wx[a][lane] = wx[a];
            s.gx[a][lane] = gx[a];
        }
#pragma unroll
        for (int n = 0; n < WideGroup<D>::YZ; ++n) {
            s.yz[n][lane] = wide_pair<SH>(wy[n % 3], D == 3 ? wz[n / 3] : wz[1]);
            s.row[n][lane] = (int32_t)(cell0 + gy[n % 3] * n0 + (D == 3 ? gz[n / 3] * n01 : 0));
        }
    }
    __syncwarp();
    const int r = lane & 15, cx = r >> 2, ch = r & 3;
    for (int it = 0; it < 16; ++it) {
        const int p = 2 * it + (lane >> 4);
        if (r < 12 && ((mask >> p) & 1u)) {
            const int64_t i = s.q[ch][p];
            const uint64_t sign = (uint64_t)(i >> 63);
            const uint64_t qx = mul_hi_round(((uint64_t)i ^ sign) - sign, s.wx[cx][p]);
            unsigned long long *__restrict__ a = acc + s.gx[cx][p] * cell_stride + ch * chan_stride;
#pragma unroll
            for (int n = 0; n < WideGroup<D>::YZ; ++n)
                atomicAdd(a + s.row[n][p] * cell_stride, wide_value(qx, s.yz[n][p], sign));
        }
    }
    __syncwarp();
}

}  // namespace mhdpic
