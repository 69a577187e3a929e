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
// instructions.  A zero gives infinity, a NaN NaN, and an infinity (not 0 as
// in 1 / d) no finite number either: a flow that overflows does not come back
// as one that looks sound.
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
// 2 x and x / 2 by the exponent field, for 0 and 2^-1020 <= |x| <= 2^1022
// (infinities and NaN stay; no multiplication as a second case, which the
// compiler would issue for every x and select from)
__device__ __forceinline__ double twice64(double x) {
    const int hi = __double2hiint(x);
    const bool normal = (unsigned)(hi & 0x7ff00000) - 0x100000u < 0x7fe00000u;
    return __hiloint2double(normal ? hi + 0x100000 : hi, __double2loint(x));
}
__device__ __forceinline__ double half64(double x) {
    const int hi = __double2hiint(x);
    const bool normal = (unsigned)(hi & 0x7ff00000) - 0x100000u < 0x7fe00000u;
    return __hiloint2double(normal ? hi - 0x100000 : hi, __double2loint(x));
}

// x rounded to float (to nearest, ties to even) by integer instructions where
// the result is a normal float or zero, else by the conversion
__device__ __forceinline__ float narrow32(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned m = hi & 0x7fffffffu;
    if (m - 0x38100000u < 0x0fd00000u) {   // exponent field 897 .. 1149
        const unsigned long long r = ((unsigned long long)(m - 0x38000000u) << 32 | lo) + 0x0fffffffull +
                                     ((lo >> 29) & 1u);
        return __uint_as_float((unsigned)(r >> 29) | (hi & 0x80000000u));
    }
    if ((m | lo) == 0u) return __uint_as_float(hi);
    return (float)x;
}
// a float that is x to 2^-22 where *ok stays true (tiny values become 0)
__device__ __forceinline__ float near32(double x, bool &ok) {
    const unsigned hi = (unsigned)__double2hiint(x), m = hi & 0x7fffffffu;
    ok = ok && m < 0x47e00000u;
    const unsigned f = __funnelshift_l((unsigned)__double2loint(x), m - 0x38000000u, 3);
    return m < 0x38100000u ? 0.0f : __uint_as_float(f | (hi & 0x80000000u));
}

// Wave speeds in FP32 as a screen for the FP64 ones: 1/rho and the speed of
// sound of a state x to 2^-22 (near32); true where every |m_a| / rho + c is
// trusted to 3e-6.  The pressure is h1 e2, h1 = (gamma - 1) / 2, e2 = 2 E -
// m^2 / rho: cutting the inputs, the square, the reciprocal and the difference
// round e2 by at most 1.6e-6 E, so where e2 > E / 2 the root's relative error
// is below 2e-6, whatever gamma is (in air that is p > E / 10).  Two cells'
// errors stay below the 1e-5 by which a caller lets one lead.  rho E, which
// bounds m^2, and the squared speed of sound lie far inside FP32's range: in
// units that put them near its ends m^2 is lost (at rho about 1e-21 a cell at
// rest counted as slower than one whose kinetic energy had underflowed).
template <int NC>
__device__ __forceinline__ bool speeds32(float gf, float h1f, const float *x, float &ir, float &cs) {
    constexpr int E = NC - 1;
    float m2 = x[E - 1] * x[E - 1];
#pragma unroll
    for (int k = E - 2; k >= 1; --k) m2 = fmaf(x[k], x[k], m2);
    ir = __fdividef(1.0f, x[0]);
    const float e2 = fmaf(-m2, ir, 2.0f * x[E]), c2 = gf * (h1f * e2) * ir;
    const float rE = x[0] * x[E];
    cs = sqrtf(c2);
    return x[0] > 1e-30f && x[0] < 1e30f && rE > 1e-30f && rE < 1e30f && c2 > 1e-30f && c2 < 1e30f && e2 > 0.5f * x[E];
}

// ---------------------------------------------------------------------------
// FP64 Euler arithmetic, conserved variables q[NC] = rho, momenta, E; D: the
// momentum normal to the faces
// ---------------------------------------------------------------------------
// a face's side: state, 1/rho and pressure
template <int NC>
struct Side { double q[NC], ir, p; };
template <int NC>
__device__ __forceinline__ double msq64(const double *q) {   // |m|^2
    double s = q[NC - 2] * q[NC - 2];
#pragma unroll
    for (int k = NC - 3; k >= 1; --k) s = __fma_rn(q[k], q[k], s);
    return s;
}
// pressure, h1 = (gamma - 1) / 2
template <int NC>
__device__ __forceinline__ double press64(double h1, const double *q, double ir) {
    return h1 * __fma_rn(-msq64<NC>(q), ir, twice64(q[NC - 1]));
}
// rho > 0 and 2 rho E > |m|^2, in FP32 where that decides with a margin of
// 1e-5 (its error is below 2e-6 where no product underflows, which the bounds
// on 2 rho E leave out), else in FP64
template <int NC>
__device__ __forceinline__ bool physical64(const double *q) {
    bool ok = true;
    const float r = near32(q[0], ok), E = near32(q[NC - 1], ok);
    float m2 = 0.0f;
#pragma unroll
    for (int k = 1; k < NC - 1; ++k) {
        const float m = near32(q[k], ok);
        m2 = fmaf(m, m, m2);
    }
    const float t = 2.0f * r * E;
    if (ok && r > 0.0f && E > 0.0f && t > 1e-30f && t < 1e38f && t - m2 > 1e-5f * t) return true;
    return pos64(q[0]) && 2.0 * q[0] * q[NC - 1] > msq64<NC>(q) && q[NC - 1] - q[NC - 1] == 0.0;
}
// MUSCL-Hancock evolved states of one cell: van Leer slopes in conserved
// variables (none where !lim), half-step evolution (hl = dt / 2h, h1 =
// (gamma - 1) / 2), first order
// where an evolved state is not physical.  One reciprocal of the product of
// two densities serves both sides; the positivity tests use the pressures
// that the Riemann solver takes.
template <int NC, int D>
__device__ __forceinline__ void evolve64(double h1, double hl, const double *qm, const double *q0, const double *qp,
                                         bool lim, Side<NC> &L, Side<NC> &R) {
    constexpr int in = 1 + D, E = NC - 1;
    double l[NC], r[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        // half the slope: dm dp / (dm + dp)
        const double dm = q0[k] - qm[k], dp = qp[k] - q0[k];
        double pr = dm * dp, y = 0.0;
        if (lim && pos64(pr)) y = rcp64(dm + dp);
        else pr = 0.0;
        l[k] = __fma_rn(-pr, y, q0[k]);
        r[k] = __fma_rn(pr, y, q0[k]);
    }
    double rr = rcp64(l[0] * r[0]);
    const double il = r[0] * rr, ig = l[0] * rr;
    const double pl = press64<NC>(h1, l, il), pg = press64<NC>(h1, r, ig);
    const double ul = l[in] * il, ug = r[in] * ig;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        double df;   // flux of the low side less that of the high side
        if (k == 0) df = l[in] - r[in];
        else if (k == in) df = __fma_rn(l[in], ul, pl) - __fma_rn(r[in], ug, pg);
        else if (k == E) df = __fma_rn(ul, l[E] + pl, -(ug * (r[E] + pg)));
        else df = __fma_rn(l[k], ul, -(r[k] * ug));
        L.q[k] = __fma_rn(hl, df, l[k]);
        R.q[k] = __fma_rn(hl, df, r[k]);
    }
    rr = rcp64(L.q[0] * R.q[0]);
    L.ir = R.q[0] * rr;
    R.ir = L.q[0] * rr;
    L.p = press64<NC>(h1, L.q, L.ir);
    R.p = press64<NC>(h1, R.q, R.ir);
    if (!(pos64(L.q[0]) && pos64(R.q[0]) && pos64(L.p) && pos64(R.p))) {
#pragma unroll
        for (int k = 0; k < NC; ++k) L.q[k] = R.q[k] = q0[k];
        L.ir = R.ir = rcp64(q0[0]);
        L.p = R.p = press64<NC>(h1, q0, L.ir);
    }
}
// HLLC flux with Davis wave speeds (Toro, ch. 10), the star flux in the form
// [S* (S Q - F) + S p* (0, n, S*)] / (S - S*) with p* = p + rho (S - u)(S* - u)
// of the side that holds the face
template <int NC, int D>
__device__ __forceinline__ void hllc64(double g, const Side<NC> &L, const Side<NC> &R, double *F) {
    constexpr int in = 1 + D, E = NC - 1;
    const double uL = L.q[in] * L.ir, uR = R.q[in] * R.ir;
    const double cL = sqrt64(g * (L.p * L.ir)), cR = sqrt64(g * (R.p * R.ir));
    const double SL = min64(uL - cL, uR - cR), SR = max64(uL + cL, uR + cR);
    const bool supL = nonneg64(SL), supR = !pos64(SR);
    if (supL || supR) {
        const double u = supL ? uL : uR, p = supL ? L.p : R.p;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const double q = supL ? L.q[k] : R.q[k], m = supL ? L.q[in] : R.q[in];
            F[k] = k == 0 ? m : k == in ? __fma_rn(q, u, p) : k == E ? u * (q + p) : q * u;
        }
        return;
    }
    const double vL = SL - uL, vR = SR - uR;
    const double aL = L.q[0] * vL, aR = R.q[0] * vR;
    const double num = __fma_rn(uL, aL, __fma_rn(-uR, aR, R.p - L.p));
    const double Ss = num * rcp64(aL - aR);
    const bool left = nonneg64(Ss);
    const double S = left ? SL : SR, u = left ? uL : uR, v = left ? vL : vR, a = left ? aL : aR;
    const double p = left ? L.p : R.p;
    const double k1 = rcp64(S - Ss), kS = k1 * Ss;
    const double Sp = S * __fma_rn(a, Ss - u, p);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const double q = left ? L.q[k] : R.q[k];
        if (k == 0) F[k] = a * kS;
        else if (k == in) F[k] = __fma_rn(kS, __fma_rn(q, v, -p), k1 * Sp);
        else if (k == E) F[k] = kS * (__fma_rn(q, v, -(u * p)) + Sp);
        else F[k] = q * v * kS;
    }
}

}  // namespace mbfp
