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

// One Newton step of e t^2 + d t - e on the float32 tangent, the residual in
// float64 and the slope in float32: t to about 1e-14 of itself.
__device__ __forceinline__ double jac_tan64(double d, double e, float fd, float fe) {
    const float t = jac_tan(fd, fe);
    const double td = f2d_exact(t);
    const float r = d2f_trunc(fma(fma(e, td, d), td, -e));
    return td - f2d_exact(__fdividef(r, fmaf(2.f * fe, t, fd)));
}

// c = 1 / sqrt(1 + t^2) and s = t c in float64 for |t| <= 1 or so: the float32
// value of 1 / sqrt(x), x = 1 + t^2, and one third-order step (the binomial
// series of (1 - h)^(-1/2) to h^2, h = 1 - x y^2); its error is 5/16 h^3 with
// |h| < 2^-20, far below rounding.  Orthonormal to rounding for any t.
__device__ __forceinline__ void jac_cs64(double td, double& c, double& s) {
    const float t = d2f_trunc(td);
    const double y = f2d_exact(rsqrtf(fmaf(t, t, 1.f)));
    const double x = fma(td, td, 1.0), yy = y * y;
    const double h = fma(-x, yy, 1.0);
    c = fma(y * h, fma(0.375, h, 0.5), y);
    s = td * c;
}
// A symmetric 2 x 2 block [[a, e], [e, b]] under that rotation:
//   a' = a - t (e - x),  e' = -x,  b' = b + t (e - x),
// x = c^2 (e t^2 + (b - a) t - e), the part of e that a rounded tangent leaves.
__device__ __forceinline__ void jac_block64(double td, double c, double& a, double& e, double& b) {
    const double x = c * c * fma(fma(e, td, b - a), td, -e), u = td * (e - x);
    a -= u;
    b += u;
    e = -x;
}
// |e| <= 2^-60 sqrt|a b| (1e-18), by the exponents
__device__ __forceinline__ bool jac_negligible(double e, double a, double b) {
    return 2 * dexp(e) < dexp(a) + dexp(b) - 120;
}

}  // namespace mpspt
