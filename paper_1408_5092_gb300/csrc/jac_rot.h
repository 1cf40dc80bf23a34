// Rotations of the Jacobi eigensolvers without the float64 divide and square
// root: on this GPU one dependent double division or square root takes about
// 650 clocks and a float64 FMA 64, so a rotation computed with them (two
// divisions, two to three square roots) was a chain of 3300 clocks and more
// than half of a round's time at n below 100.
#pragma once
#include <cuda_runtime.h>

namespace mpspt {

// float64 -> float32 of v * 2^-sh, round to nearest even, by integer
// operations; magnitudes below the float32 normal range become signed zero,
// above it infinity.
__device__ __forceinline__ float d2f_scaled(double v, int sh) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const int e = (int)((b >> 52) & 0x7FF);
    const unsigned long long m = b & 0xFFFFFFFFFFFFFULL;
    if (e == 0x7FF) return __uint_as_float(sign | 0x7F800000u | (m ? 0x400000u : 0u));
    const int fe = e - 1023 + 127 - sh;
    if (e == 0 || fe <= 0) return __uint_as_float(sign);
    if (fe >= 255) return __uint_as_float(sign | 0x7F800000u);
    const unsigned rem = (unsigned)(m & 0x1FFFFFFFULL);
    unsigned f = sign | ((unsigned)fe << 23) | (unsigned)(m >> 29);
    if (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) f += 1u;   // a carry may reach the exponent
    return __uint_as_float(f);
}
__device__ __forceinline__ int dexp(double v) { return (int)(((unsigned long long)__double_as_longlong(v) >> 52) & 0x7FF); }

// Cheap conversions for the float64 rotations (40 clocks by integer
// operations; the conversion instructions take about 100): float64 -> float32
// truncated, below the float32 normal range to signed zero (|v| < 2^127 is
// the caller's), and float32 (normal or zero) -> float64.
__device__ __forceinline__ float d2f_trunc(double v) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int e = (hi >> 20) & 0x7FF;
    const unsigned f = ((unsigned)(e - 896) << 23) | (((unsigned)hi & 0xFFFFFu) << 3) | ((unsigned)lo >> 29);
    return __uint_as_float(((unsigned)hi & 0x80000000u) | (e > 896 ? f : 0u));
}
__device__ __forceinline__ double f2d_exact(float v) {
    const unsigned b = __float_as_uint(v);
    const unsigned mag = b & 0x7FFFFFFFu;
    const unsigned hi = (b & 0x80000000u) | (mag ? (mag >> 3) + (896u << 20) : 0u);
    return __hiloint2double((int)hi, (int)(b << 29));
}
// |x| < y for y >= 0, and x == 0, by the bits (a float64 comparison takes 110 clocks)
__device__ __forceinline__ bool abs_below(double x, double y) {
    return (unsigned long long)(__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL) < (unsigned long long)__double_as_longlong(y);
}
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL) == 0; }

// tan of the rotation that annihilates e between diagonal entries a and
// a + d: the root of e t^2 + d t - e = 0 of smaller magnitude (positive for
// d = 0, e > 0), in float32, t = 2 e / (d + sgn(d) sqrt(d^2 + 4 e^2)).
// |d|, |e| < 2^60; e must not be zero.
__device__ __forceinline__ float jac_tan(float d, float e) {
    const float up = fmaxf(fabsf(d), fabsf(e)) < 0x1p-40f ? 0x1p64f : 1.f;   // keeps the squares normal
    d *= up;
    e *= 2.f * up;
    const float h = fmaf(d, d, e * e);
    const float r = fabsf(d) + h * rsqrtf(h);
    return __fdividef(d < 0.f ? -e : e, r);
}

// What one Newton step of e t^2 + d t - e takes from the float32 tangent t (the
// residual in float64, the slope in float32): t - dt is right to 1e-13 of itself.
__device__ __forceinline__ float jac_newton(double d, double e, float fd, float fe, float t) {
    const double td = f2d_exact(t);
    const float r = d2f_trunc(fma(fma(e, td, d), td, -e));
    return __fdividef(r, fmaf(2.f * fe, t, fd));
}

// Rotations are applied by their sine s and the tangent h of half their angle,
//   x' = c x - s y = x - s (y + h x),   y' = s x + c y = y + s (x - h y)
// with c = 1 - s h (Rutishauser, Numer. Math. 9, 1966).  As many operations on a
// pair as with (c, s), but what rounding takes from c^2 + s^2 = 1 is s h eps
// instead of eps for every rotation, however small, and nothing of the angle's
// error as long as s = 2 h / (1 + h^2).  With a rounded (c, s) the columns of V
// lose their common length while the diagonal keeps its own: vectors 8 to 13%
// further from the exact ones than with divisions and square roots (n = 8 to 90,
// four decades); with (s, h) they are 3 to 20% nearer, orthonormality and
// eigenvalues 2.5 to 20 times better, at the same number of float64 operations
// on a pair (noalloc, twelve 13 x 13: 235 us with (c, s), 230 with (s, h)).
//
// h for the tangent t - dt, |t| <= 1 or so: the float32 value and one Newton step
// of t h^2 + 2 h - t, to 1e-12 of itself.  (2 h - t and h^2 are exact.)
__device__ __forceinline__ double jac_half64(float t, float dt) {
    const float x = fmaf(t, t, 1.f), hf = __fdividef(t, fmaf(x, rsqrtf(x), 1.f));
    const double h = f2d_exact(hf);
    const float r = d2f_trunc(fma(f2d_exact(t), h * h, f2d_exact(fmaf(2.f, hf, -t))));
    const float slope = 2.f * fmaf(t, hf, 1.f);
    return h - f2d_exact(__fdividef(r, slope) + dt * __fdividef(fmaf(hf, hf, 1.f), 2.f * x));
}
// s = 2 h / (1 + h^2), |h| <= 1/2 or so: the float32 reciprocal and one
// third-order Newton step (1 - r is exact in float32).
__device__ __forceinline__ double jac_sine64(double h) {
    const float hf = d2f_trunc(h), rf = fminf(__fdividef(1.f, fmaf(hf, hf, 1.f)), 1.f);
    const double e = fma(-(h * h), f2d_exact(rf), f2d_exact(1.f - rf)), r = f2d_exact(2.f * rf);
    return h * fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double rot_first(double s, double h, double x, double y) { return fma(-s, fma(h, x, y), x); }
__device__ __forceinline__ double rot_second(double s, double h, double x, double y) { return fma(s, fma(-h, y, x), y); }
// A symmetric 2 x 2 block [[a, e], [e, b]] under that rotation:
//   a' = a - u,  b' = b + u,  u = 2 s c e - s^2 (b - a),
//   e' = (1 - 2 s^2) e - s c (b - a), what a rounded angle leaves of e.
// (|e| >= 2^-960, so that twice of it is one exponent up.)
__device__ __forceinline__ void jac_block64(double s, double h, double& a, double& e, double& b) {
    const double e2 = __hiloint2double(__double2hiint(e) + (1 << 20), __double2loint(e));
    const double q = s * fma(-s, h, 1.0), p = s * s, d = b - a;
    const double u = fma(q, e2, -(p * d));
    e = fma(-q, d, fma(-p, e2, e));
    a -= u;
    b += u;
}
// |e| <= 2^-60 sqrt|a b| (1e-18), by the exponents
__device__ __forceinline__ bool jac_negligible(double e, double a, double b) {
    return 2 * dexp(e) < dexp(a) + dexp(b) - 120;
}

}  // namespace mpspt
