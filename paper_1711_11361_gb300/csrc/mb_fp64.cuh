// mb_fp64.cuh -- reciprocal, square root, sign tests and ordering of doubles
// with few instructions on the FP64 pipe.
//
// GB300 does 2 FP64 lane operations per clock and SM (64 times fewer than
// FP32 or integer ones), and every FP64 instruction counts, comparisons and
// min/max included.  So the seeds below come from the FP32 reciprocal and
// reciprocal square root of the significand, the exponents are moved with
// integer instructions, and the tests compare bit patterns.
#pragma once
#include <cuda_runtime.h>

namespace mbfp {

// the top 23 significand bits of x (hi, lo: its words) as a float with
// exponent field e
__device__ __forceinline__ float significand(int hi, int lo, unsigned e) {
    return __uint_as_float((__funnelshift_l((unsigned)lo, (unsigned)hi, 3) & 0x7fffffu) | (e << 23));
}
// the float r (normal, positive) as a double, its exponent field raised by
// shift >> 20
__device__ __forceinline__ double widen_scaled(float r, int shift) {
    const unsigned b = __float_as_uint(r);
    return __hiloint2double((int)(b >> 3) + 0x38000000 + shift, (int)(b << 29));
}

// 1 / d for 2^-1021 <= |d| <= 2^1021: seed y0 = 1 / m from the FP32
// reciprocal of the significand (relative error at most 2^-22 from the
// truncated significand and 2^-23 from rcp.approx), then one step of the
// third-order hyperpower iteration y = y0 (1 + e + e^2), e = 1 - d y0.  The
// remaining error e^3 < 2^-63 is below the last rounding: 3 FP64
// instructions.  A zero gives infinity and a NaN NaN.
__device__ __forceinline__ double rcp64(double d) {
    const int hi = __double2hiint(d), lo = __double2loint(d);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(significand(hi, lo, 127u)));
    double y = widen_scaled(r, 0x3ff00000 - (hi & 0x7ff00000));
    y = __hiloint2double(__double2hiint(y) | (hi & (int)0x80000000), __double2loint(y));
    const double e = __fma_rn(-d, y, 1.0);
    return __fma_rn(y, __fma_rn(e, e, e), y);
}

// sqrt(x) for 2^-1021 <= x <= 2^1021 (0 for 0, NaN for a negative x): seed
// y0 = 1 / sqrt(x) from the FP32 reciprocal square root of the significand
// with an even exponent (relative error below 2^-21), then with s = x y0,
// e = 1 - s y0 the series sqrt(x) = s (1 + e/2 + 3 e^2 / 8 + ...) to third
// order: 5 FP64 instructions
__device__ __forceinline__ double sqrt64(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int k = ((hi >> 20) - 1023) >> 1;                       // x = m 4^k, 1 <= m < 4
    const unsigned odd = ((unsigned)(hi >> 20) + 1u) & 1u;
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(significand(hi, lo, 127u + odd)));
    double y = widen_scaled(r, -(k << 20));
    if (hi < 0) y = __hiloint2double(0x7ff80000, 0);
    const double s = x * y;
    const double e = __fma_rn(-s, y, 1.0);
    return __fma_rn(s, e * __fma_rn(0.375, e, 0.5), s);
}

// x > 0 (false for NaN), x >= 0 with -0 counting as 0, by the bits
__device__ __forceinline__ bool pos64(double x) {
    return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool nonneg64(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return b <= 0x7ff0000000000000ull || b == 0x8000000000000000ull;
}
// order-preserving integer key, and min / max by it (numbers; a NaN orders
// by its bits)
__device__ __forceinline__ long long key64(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double min64(double a, double b) { return key64(a) < key64(b) ? a : b; }
__device__ __forceinline__ double max64(double a, double b) { return key64(a) < key64(b) ? b : a; }
__device__ __forceinline__ double abs64(double x) {
    return __hiloint2double(__double2hiint(x) & 0x7fffffff, __double2loint(x));
}
__device__ __forceinline__ double neg64(double x) {
    return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}
// x / 2 and 2 x of normal numbers by the exponent field (0 stays 0)
__device__ __forceinline__ double twice64(double x) {
    const int hi = __double2hiint(x);
    return (hi & 0x7ff00000) ? __hiloint2double(hi + 0x100000, __double2loint(x)) : x + x;
}

}  // namespace mbfp
