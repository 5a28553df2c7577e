// FP64 building blocks for short dependent chains (the swap transforms of the
// window tasks): reciprocals, square roots and rotations that start from the
// special function unit's approximations, conversions to and from FP32 on the
// integer pipe, and tests that stay off the FP64 pipe.
#pragma once

#include "swap_math.cuh"

#include <float.h>

namespace gbr {

// Seeds with about 20 correct bits (PTX rcp/rsqrt.approx.ftz.f64).
__device__ __forceinline__ double rcp_seed(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
// x times 2^-1 for a normal x above the smallest binade, and for no other: the
// exponent field of 0, of a subnormal or of an infinity gives a wrong number.
// (In sqrt64 x is the seed of a normal number: within [2^-512, 2^511].)
__device__ __forceinline__ double half_of(double x) {
    return __longlong_as_double(__double_as_longlong(x) - (1LL << 52));
}
// x >= 0 and x == 0 (either zero) on the integer pipe.
__device__ __forceinline__ bool nonneg(double x) {
    return __double_as_longlong(x) >= 0 || __double_as_longlong(x) == (long long)(1ULL << 63);
}
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
// max(10 eps m, DBL_MIN), the threshold of the stability tests, as a bit
// pattern (m >= 0).
__device__ __forceinline__ unsigned long long thresh_bits(unsigned long long m) {
    const unsigned long long t = abs_bits(10.0 * DBL_EPSILON * bits_double(m));
    return t > 0x0010000000000000ULL ? t : 0x0010000000000000ULL;
}
// 1/x for normal x: one third-order step, y (1 + e + e^2) with e = 1 - x y
// (the geometric series of 1 / (1 - e)).
__device__ __forceinline__ double rcp64(double x) {
    const double y = rcp_seed(x), e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// sqrt(x) for normal x: one step of Goldschmidt's iteration on (sqrt, 1/(2
// sqrt)) and a final residual correction (Markstein 2004).
__device__ __forceinline__ double sqrt64(double x) {
    const double y = rsqrt_seed(x);
    double g = x * y, h = half_of(y);
    const double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    return fma(fma(-g, g, x), h, g);
}
// x 2^(127 - eoff) as a float by truncation, and a float as a double, both on
// the integer pipe (0 below the normal range, infinity above it).
__device__ __forceinline__ float to_f32(double x, int eoff) {
    const unsigned hi = __double2hiint(x), lo = __double2loint(x);
    const int fld = (int)((hi >> 20) & 0x7ff), e = fld - eoff;
    const unsigned b = e <= 0 || fld == 0 ? 0u
                     : e >= 255 ? 0x7f800000u
                                : ((unsigned)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    return __uint_as_float((hi & 0x80000000u) | b);
}
__device__ __forceinline__ double from_f32(float x) {
    const unsigned b = __float_as_uint(x), e = (b >> 23) & 255u;
    if (e == 0) return 0.0;
    return __hiloint2double((int)((b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3)),
                            (int)(b << 29));
}

// Givens rotation (c, s) from (t, d): (t, d) / |(t, d)|.  Values whose squares
// leave the normal range are scaled by a power of two first.  A component that
// is more than 2^27 times the other one is +-1, its correctly rounded value:
// the product t rh rounds to the number below 1 in about half of such cases
// (mean of c^2 + s^2 - 1 at d = 1e-9 t: -0.26 2^-53) and never to the one above,
// and a matrix that many of these rotations are accumulated into would shrink.
__device__ __forceinline__ void givens64(double t, double d, double* c, double* s) {
    double nn = fma(t, t, d * d);
    const unsigned e = (unsigned)__double2hiint(nn) >> 20;
    if (e < 100u || e > 1900u) {
        const unsigned long long bt = abs_bits(t), bd = abs_bits(d);
        const int em = (int)((bt > bd ? bt : bd) >> 52);
        const double sc = __hiloint2double((em < 1 ? 2045 : (em > 2045 ? 1 : 2046 - em)) << 20, 0);
        t *= sc;
        d *= sc;
        nn = fma(t, t, d * d);
    }
    // 1 / sqrt(nn): one third-order step, y (1 + e/2 + 3 e^2 / 8) with
    // e = 1 - nn y^2 (the binomial series of (1 - e)^(-1/2))
    const double y = rsqrt_seed(nn);
    const double r = fma(-(nn * y), y, 1.0);
    const double rh = fma(y * r, fma(0.375, r, 0.5), y);
    const int et = (__double2hiint(t) >> 20) & 0x7ff, ed = (__double2hiint(d) >> 20) & 0x7ff;
    *c = et - ed >= 28 ? copysign(1.0, t) : t * rh;
    *s = ed - et >= 28 ? copysign(1.0, d) : d * rh;
}

}  // namespace gbr
