// FP64 quotient, reciprocal and square root as the operators round them, in few instructions,
// for a warp that works through a chain of them.  On GB300 a warp gets one FP64 instruction through
// every 64 cycles, dependent or not; a division takes 564 cycles and a square root 686.  The
// forms below take a 22-bit start from the FP32 unit, two Newton terms at once, and one
// residual correction by fused multiply-adds, which rounds correctly when the value it
// corrects is within one unit in the last place and the reciprocal that it uses is correctly
// rounded (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", IBM J. Res. Dev. 34, 1990): 7 instructions for a quotient, 5 for the
// reciprocal, 9 for a root, 2 for the reciprocal of a root just taken.  The reciprocals here
// are within 2^-66 of the true value before their rounding, not proven rounded; the results
// have the operators' bits on the random, special and near-midpoint operands of
// tests/test_gpu_fp64_fast.py.  One class is left out: the reciprocal of a value with every
// mantissa bit set may miss the last bit.  Operands outside a wide middle range of exponents
// (where a start or a residual could over- or underflow) take the plain operators, as do
// zeros, infinities and NaN.
#pragma once

#include <stdint.h>

namespace fp64_fast {

__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// 2^e of the value with x's mantissa in [1, 2), as FP32 (top 23 bits).
__device__ __forceinline__ float mantissa32(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    return __uint_as_float(0x3F800000u | (uint32_t)((b >> 29) & 0x7FFFFFu));
}
// f (positive, normal) times 2^e as a double.
__device__ __forceinline__ double widen(float f, int e) {
    const uint64_t b = (uint64_t)__float_as_uint(f);
    return __longlong_as_double((long long)((b << 29) + ((uint64_t)(1023 - 127 + e) << 52)));
}
// x / 2 and 2 x of a value in the middle range (exponent arithmetic, no FP64 instruction)
__device__ __forceinline__ double halve(double x) { return __longlong_as_double(__double_as_longlong(x) - (1ll << 52)); }
__device__ __forceinline__ double twice(double x) { return __longlong_as_double(__double_as_longlong(x) + (1ll << 52)); }
// Whether every step below stays far from the ends of the exponent range.
__device__ __forceinline__ bool middle(double x) {
    const int e = exponent(x);
    return e > 1023 - 400 && e < 1023 + 400;
}

// 1 / |d| to about 22 bits.
__device__ __forceinline__ double rcp_start(double d) { return widen(__frcp_rn(mantissa32(d)), 1023 - exponent(d)); }

// n / d
__device__ __forceinline__ double divide(double n, double d) {
    if (!middle(d) || !middle(n)) return n / d;
    const double r0 = copysign(rcp_start(d), d);
    const double e = fma(-d, r0, 1.0), t = fma(e, e, e);  // 1 / (1 - e) = 1 + e + e^2 + O(2^-66)
    const double r = fma(r0, t, r0);
    const double q0 = n * r0, q1 = fma(q0, t, q0);
    return fma(fma(-d, q1, n), r, q1);
}

// sign / d, sign = 1 or -1
__device__ __forceinline__ double reciprocal(double sign, double d) {
    if (!middle(d)) return sign / d;
    const double r0 = copysign(rcp_start(d), d);
    const double e = fma(-d, r0, 1.0), r1 = fma(r0, fma(e, e, e), r0);
    const double r = fma(fma(-d, r1, 1.0), r1, r1);
    return __double2hiint(sign) < 0 ? -r : r;
}

// sqrt(x), x > 0; y: 1 / sqrt(x) to about one unit in the last place
__device__ __forceinline__ double root(double x, double &y) {
    if (!middle(x)) {
        const double s = sqrt(x);
        y = 1.0 / s;
        return s;
    }
    const int ex = exponent(x) - 1023, odd = ex & 1;
    const float m = odd ? 2.0f * mantissa32(x) : mantissa32(x);  // x = m 2^(ex - odd), m in [1, 4)
    const double y0 = widen(rsqrtf(m), -((ex - odd) >> 1));
    const double h0 = x * y0;
    const double e = fma(-h0, y0, 1.0);       // 1 / sqrt(1 - e) = 1 + e (1/2 + 3/8 e) + O(2^-64)
    const double p = fma(e, 0.375, 0.5);
    const double s1 = fma(h0 * e, p, h0);
    y = fma(y0 * e, p, y0);
    return fma(fma(-s1, s1, x), halve(y), s1);
}

// 1 / s, where y is 1 / s to about one unit in the last place.
__device__ __forceinline__ double reciprocal_near(double s, double y) {
    if (!middle(s)) return 1.0 / s;
    return fma(fma(-s, y, 1.0), y, y);
}

}  // namespace fp64_fast
