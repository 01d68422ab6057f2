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

// x / h with y = 1/h correctly rounded: the quotient x y corrected by its exact
// residual is the correctly rounded one (Markstein 1990, "Computation of
// elementary functions on the IBM RISC System/6000"), so the bits of x / h, in
// three FP64 operations.
__device__ __forceinline__ double div_by(double x, double h, double y)
{
    const double q = x * y;
    return fma(fma(-q, h, x), y, q);
}
__device__ __forceinline__ float div_by(float x, float h, float) { return x / h; }

}  // namespace gsis
