// Reciprocals and quotients in a few multiply-adds, where the division's range
// checks and its length would set a kernel's pace.  The method is Markstein's
// ("Computation of elementary functions on the IBM RISC System/6000", 1990):
// Newton steps and a correction by the residual, which a fused multiply-add
// gives exactly.  His theorem makes a quotient correctly rounded if the
// reciprocal is; rcp_newton's and ratio's start from an approximation, so that
// they have the division's bits is observed, not proven.
#pragma once

#include <cuda_runtime.h>

namespace gsis {

// 1/d of an FP32 diagonal in [2^-100, 2^100]: one Newton step r + r (1 - d r)
// from an approximation within 1 ulp.  The bits of __frcp_rn for every float of
// the range.  Six instructions that overlap from cell to cell; __frcp_rn with
// its range checks took 136 cycles a cell, one after the other, and set the
// pace of the FP32 sweep (2179 cycles per 16-step chunk).
constexpr unsigned kRcpLo = (127u - 100u) << 23, kRcpHi = (127u + 100u) << 23;
__device__ __forceinline__ float rcp_newton(float d)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return __fmaf_rn(r, __fmaf_rn(-d, r, 1.0f), r);
}

// a / d for 0 <= a < d: reciprocal from the FP32 approximation of d's leading
// 24 bits (integer instructions), one third-order Newton step, and the quotient
// corrected by its exact residual.  The division's bits on all pairs tried
// (7e8: random mantissas, divisors next to a power of two, quotients next to 1).
// Six FP64 operations and no branch taken; the division is 140 cycles of the
// pipe and a call that keeps the other rows' work from overlapping
// (second-order residual 256^2 S12: 554 -> 482 us).  Exponents for which an
// intermediate could leave the normal range take the division.
__device__ __forceinline__ double ratio(double a, double d)
{
    const unsigned dh = (unsigned)__double2hiint(d), ah = (unsigned)__double2hiint(a);
    const unsigned ed = dh >> 20, ea = ah >> 20;
    if (ed - 600u > 800u || (ea - 400u > 1000u && __double_as_longlong(a) != 0)) return a / d;
    const float m = __uint_as_float(0x3f800000u | (__funnelshift_l((unsigned)__double2loint(d), dh, 3) & 0x7fffffu));
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
    const unsigned rb = __float_as_uint(r);
    const double y0 = __hiloint2double((int)((rb >> 3) + ((1023u - 127u + 1023u - ed) << 20)), (int)(rb << 29));
    const double e = fma(-d, y0, 1.0);
    const double y = fma(y0, fma(e, e, e), y0);
    const double q = a * y;
    return fma(fma(-q, d, a), y, q);
}

// x / h, h > 0, with y = 1/h correctly rounded: x y corrected by its exact
// residual is the correctly rounded quotient, in three FP64 operations; the sign
// of x is put back for x = -0.  The residual is exact, and the bits are the
// division's, for |x| in [2^-960, 2^960] and |x / h| in [2^-1000, 2^1000], h in
// [2^-500, 2^500] (the gradient's weights need h^2 in range anyway).  Beyond
// that the last place may differ.  Those exponents have no branch to the
// division: a check per quotient costs more than it mends (256^2 S12 residual
// with a branch to the division, which beams in thick cells then take: 482 -> 550 us,
// and 830 with the range of ratio; one branch for both quotients: 500).
__device__ __forceinline__ double div_by(double x, double h, double y)
{
    const double q = x * y;
    double r = fma(fma(-q, h, x), y, q);
    if ((__double2hiint(r) & 0x7ff80000) == 0x7ff80000) r = q;   // x y overflowed, or x is not a number
    return __hiloint2double((__double2hiint(r) & 0x7fffffff) | (__double2hiint(x) & (int)0x80000000), __double2loint(r));
}
__device__ __forceinline__ float div_by(float x, float h, float) { return x / h; }

}  // namespace gsis
