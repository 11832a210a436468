// Double-precision reciprocal, quotient and reciprocal square root for kernels that are
// bound by the FP64 pipe: the hardware's approximation (PTX rcp.approx.ftz.f64 and
// rsqrt.approx.ftz.f64, which work on the operand's upper 32 bits) and one iteration of
// third order, in 4 to 6 FP64 instructions and without a branch.  rcp_refined holds for
// 2^-1020 <= |d| <= 2^1020, the others for operands with refinable(); callers take the plain
// operations elsewhere (zero, subnormal, the ends of the range, infinities, NaN).
//
// With e the approximation's relative error and u = 2^-53:
//  * rcp_refined: the hyperpower iteration of order three (M. Altman, Pacific J. Math. 10
//    (1960) 1107), r (1 + e + e^2).  It leaves e^3 and the last rounding u; |e| <= 2^-18
//    gives below 1.5 u, so at most 1 ulp from the rounded value.
//  * div_refined: n r corrected by its remainder (P. Markstein, IBM J. Res. Dev. 34 (1990)
//    111), which an FMA forms exactly: the last rounding, at most 1 ulp from the rounded
//    value.
//  * rsqrt_refined: Householder's iteration of order three (The Numerical Treatment of a
//    Single Nonlinear Equation, 1970), y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2.
//    It leaves 5/16 e^3, half the rounding of x y and the last one: below 1.6 u, at most 2
//    ulp from the rounded value.
// evp_selftest compares the three with CUDA's rounded division and square root over these
// ranges, and e with 2^-18.
#pragma once

namespace evp {

__device__ __forceinline__ double rcp_seed(double d) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    return r;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}

// 2^-500 <= |x| < 2^500 (integer compare); the reciprocals, squares and products of two
// such values are normal
__device__ __forceinline__ bool refinable(double x) {
    return (unsigned)(__double2hiint(x) & 0x7fffffff) - (523u << 20) < (1000u << 20);
}

__device__ __forceinline__ double rcp_refined(double d) {
    const double r = rcp_seed(d);
    double e = fma(-d, r, 1.0);
    e = fma(e, e, e);
    return fma(r, e, r);
}
__device__ __forceinline__ double div_refined(double n, double d) {
    const double r = rcp_refined(d), q = n * r;
    return fma(fma(-d, q, n), r, q);
}
__device__ __forceinline__ double rsqrt_refined(double x) {
    const double y = rsqrt_seed(x), e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

}  // namespace evp
