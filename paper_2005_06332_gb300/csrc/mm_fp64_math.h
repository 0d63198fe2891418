// mm_fp64_math.h -- device helpers of the FP64 kernels.
//
// FP64 instructions are scarce on this chip: a warp's takes its scheduler's
// unit for 64 clocks (measured: one warp 64 clocks each, dependent or not; an
// SM one every 16).  These helpers keep the division short and do powers of
// two in integer instructions.
#pragma once
#include <stdint.h>

namespace mmk {

// 1/x from the approximate reciprocal (about 20 bits) by one step of third
// order, r (1 + e + e^2) with e = 1 - x r: FP64 rounding in three instructions.
// For normal x below 2^1022 (the approximation is zero or infinite beyond, and
// e NaN for an infinite x or reciprocal).
__device__ __forceinline__ double rcp_approx(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}

__device__ __forceinline__ double rcp_nr(double x)
{
    const double r = rcp_approx(x), e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// a / x given r = rcp_nr(x): one residual correction.  NaN where a or the
// quotient is infinite, and short of bits where a is below 2^-960.
__device__ __forceinline__ double div_nr(double a, double x, double r)
{
    const double q = a * r;
    return fma(r, fma(-x, q, a), q);
}

// x 2^(d >> 20); d a difference of exponent fields
__device__ __forceinline__ double scale2(double x, int d)
{
    const int h = __double2hiint(x), e = h & 0x7FF00000, ne = e + d;
    if (e != 0 && e != 0x7FF00000 && ne > 0 && ne < 0x7FF00000) return __hiloint2double(h + d, __double2loint(x));
    return (x == 0.0 || e == 0x7FF00000) ? x : scalbn(x, d >> 20);
}

// the exponent field of x less that of 1 (0 for zero, subnormals, infinities
// and NaN, which then stay as they are): scale2(x, -that) lies in [1, 2)
__device__ __forceinline__ int exponent2(double x)
{
    const uint32_t e = (uint32_t)__double2hiint(x) & 0x7FF00000u;
    return e - 0x00100000u < 0x7FE00000u ? (int)e - 0x3FF00000 : 0;
}

// x 2^-(exponent2(x) >> 20)
__device__ __forceinline__ double mantissa(double x)
{
    return __hiloint2double(__double2hiint(x) - exponent2(x), __double2loint(x));
}

}  // namespace mmk
