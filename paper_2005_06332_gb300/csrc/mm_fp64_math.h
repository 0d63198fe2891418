// mm_fp64_math.h -- device helpers of the FP64 kernels.
//
// FP64 instructions are scarce on this chip: a warp's takes its scheduler's
// unit for 64 clocks (measured: one warp 64 clocks each, dependent or not; an
// SM one every 16).  These helpers keep the division short and do powers of
// two in integer instructions.
#pragma once
#include <stdint.h>

namespace mmk {

// 1/x by Newton's iteration from the approximate reciprocal (about 20 bits):
// two steps reach FP64 rounding, half the instructions of the compiled
// division.
__device__ __forceinline__ double rcp_nr(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// a / x given r = rcp_nr(x): one residual correction
__device__ __forceinline__ double div_nr(double a, double x, double r)
{
    const double q = a * r;
    return fma(r, fma(-x, q, a), q);
}

}  // namespace mmk
