// FP64 reciprocal and square root by one third-order correction of the hardware's
// approximations (PTX rcp.approx.ftz.f64 / rsqrt.approx.ftz.f64: 20 mantissa bits, measured
// relative errors below 2^-19.9 and 2^-20).  The FP64 unit is the scarce resource of the
// propagation kernel: one step of third order triples the correct bits, three FP64
// instructions for the reciprocal, five for the square root, and the approximations run on
// the special-function unit straight from the double's high word (made from
// single-precision estimates, a seed took ten integer instructions more).  Results are
// within a few ulp of the IEEE operations (checked by pch_selftest_math).  Inputs outside
// [2^-1000, 2^1000) (where a seed could leave the normal range) use the IEEE operations instead.
#pragma once
#include <cuda_runtime.h>

namespace pch {

__device__ __forceinline__ float rsqrt_approx_f32(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ double rcp_approx(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}

__device__ __forceinline__ double rsqrt_approx(double x) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}

// 2^-1000 <= |x| < 2^1000, from the biased exponent field.
__device__ __forceinline__ bool nr_range(double x) {
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    return e - (1023u - 1000u) < 2000u;
}
// 2^-1000 <= x < 2^1000 (the sign bit lands above the exponent field and fails the test).
__device__ __forceinline__ bool nr_range_pos(double x) {
    const unsigned e = (unsigned)__double2hiint(x) >> 20;
    return e - (1023u - 1000u) < 2000u;
}

// 1 / x from the seed r (|1 - x r| <= about 2^-19.9): with e = 1 - x r, 1 / x = r / (1 - e)
// = r (1 + e + e^2 + ...); one step of third order (the Newton-Raphson iteration carried to
// the quadratic term of that series) leaves a truncation of about e^3 <= 2^-59.
__device__ __forceinline__ double rcp_nr(double x) {
    if (!nr_range(x)) return 1.0 / x;
    const double r = rcp_approx(x);
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// sqrt(x) from Goldschmidt's coupled start for the square root as given by P. Markstein,
// "Software Division and Square Root Using Goldschmidt's Algorithms" (Proc. 6th Conference
// on Real Numbers and Computers, 2004), and in his "IA-64 and Elementary Functions"
// (Prentice Hall, 2000): from the seed y ~ 1/sqrt(x), g = x y ~ sqrt(x) and h = y / 2 ~
// 1 / (2 sqrt(x)); with r = 1/2 - g h, (2 g h) = 1 - 2 r and sqrt(x) = g (1 - 2 r)^(-1/2)
// = g (1 + r + 3/2 r^2 + ...).  Carried to the quadratic term (one step of third order;
// Goldschmidt's own step stops at the linear term) the truncation is about 5/2 r^3 <=
// 2^-58, and the rounding of g cancels to first order in the correction.
__device__ __forceinline__ double sqrt_nr(double x) {
    if (!nr_range_pos(x)) return sqrt(x);
    const double y = rsqrt_approx(x);
    const double g = x * y;
    const double h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));   // y / 2, exactly
    const double r = fma(-g, h, 0.5);
    return fma(g, r * fma(1.5, r, 1.0), g);
}

}  // namespace pch
