// Two-float images of doubles for the propagation kernel's order tests.
//
// GB300's FP64 unit is 64 times slower than its FP32 units, and most of a window's
// arithmetic only decides something (does a ray pass a vertex, is a window dominated).
// Such a test is evaluated in FP32, on images of the doubles scaled by a power of two
// (the mesh's mean edge length lands in [1, 2)), with a bound of its error: it acts only
// where the sign is certain.  A value becomes the unevaluated sum h + l of two floats by
// integer operations (h its leading 24 bits, l the next 23: truncation below 2^-46
// relative); F2F conversions would run on the FP64 unit.  Sums use the exact two-sum of
// D. Knuth (The Art of Computer Programming, vol. 2, section 4.2.2, theorem B), products the exact
// FMA residual.  Zero stays 0, magnitudes below the normal floats become some value below
// 2^-126, magnitudes above the floats (and infinities) infinity or NaN; every test is
// written so that a NaN decides nothing.  An image takes five integer instructions, a
// two-float eight operations; they are half of what the propagation kernel issues (with
// seven and fourteen, eight fields on 327,680 faces took 37.9 ms, with these 37.5; a field on
// the 1M-face torus 21.6 and 21.3).
#pragma once
#include <cuda_runtime.h>

#include "fastmath.cuh"

namespace pch {

struct F2 {
    float h, l;
};

// |x| as a float bit pattern, truncated; `bias` = (1023 - 127 + E) << 20 for a scale 2^-E.
__device__ __forceinline__ unsigned f_mag_bits(double x, unsigned bias) {
    const int m = (int)((unsigned)__double2hiint(x) & 0x7fffffffu) - (int)bias;
    return __funnelshift_l((unsigned)__double2loint(x), (unsigned)min(max(m, 0), 0x0ff00000), 3);
}
// x scaled, rounded towards zero.
__device__ __forceinline__ float f_of(double x, unsigned bias) {
    return __uint_as_float(f_mag_bits(x, bias) | ((unsigned)__double2hiint(x) & 0x80000000u));
}
// The double whose image these float bits are (exact; for images of nonnegative values).
__device__ __forceinline__ double of_f_bits(unsigned f, unsigned bias) {
    return f == 0u ? 0.0 : __hiloint2double((int)((f >> 3) + bias), (int)(f << 29));
}
// |x| scaled, as a two-float.
__device__ __forceinline__ F2 f2_mag(double x, unsigned bias) {
    const unsigned f = f_mag_bits(x, bias);
    // bits 28..6 of the low word follow the leading 24 bits of the mantissa: made the mantissa
    // of a float with f's exponent
    const unsigned e = f & 0x7f800000u;
    const float m = __uint_as_float((((unsigned)__double2loint(x) >> 6) & 0x7fffffu) | e) - __uint_as_float(e);
    return {__uint_as_float(f), m * 0x1p-23f};
}

__device__ __forceinline__ F2 two_sum(float a, float b) {
    const float s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}

// d - g for nonnegative two-floats (an exact leading sum, the rest rounded).
__device__ __forceinline__ F2 f2_sub(F2 d, F2 g) {
    F2 r = two_sum(d.h, -g.h);
    r.l += d.l - g.l;
    return r;
}
// x + y rounded to one float.
__device__ __forceinline__ float f2_add_f(F2 x, F2 y) {
    const F2 s = two_sum(x.h, y.h);
    return s.h + (s.l + (x.l + y.l));
}
// x^2 as a two-float (the square of the low part, below 2^-46, is dropped).
__device__ __forceinline__ F2 f2_sq(F2 x) {
    const float p = x.h * x.h;
    return {p, fmaf(x.h + x.h, x.l, fmaf(x.h, x.h, -p))};
}
// sqrt(x^2 + yy) as a two-float, relative error below 2^-44.
__device__ __forceinline__ F2 f2_hyp(F2 x, F2 yy) {
    const F2 xx = f2_sq(x);
    const F2 s = two_sum(xx.h, yy.h);
    const float e = s.l + (xx.l + yy.l);
    const float r = rsqrt_approx_f32(s.h);
    const float q = s.h * r;
    return {q, 0.5f * r * (fmaf(-q, q, s.h) + e)};
}

}  // namespace pch
