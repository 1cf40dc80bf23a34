// Host check of the float64 rotations of the Jacobi solvers (jac_rot.h), with
// the device intrinsics written out for the host and the float32 reciprocal
// and square root wrong by up to two units in the last place.
//  * R^T R = I: with c = 1 - s h, c^2 + s^2 - 1 = s (s (1 + h^2) - 2 h), of which
//    s, within 1.5 eps' (eps' = 2^-53) of 2 h / (1 + h^2), leaves |2 s h| 1.5
//    eps'; with the rounding inside 1 + h^2: 8 eps' |s h|.
//  * the angle: the half tangent's two corrections are below 2^-20 of it each
//    (float32 values up to a few units off), so the neglected second order is
//    below (2^-19)^2 = 2^-38 of it, and the tangent's below 2^-37.
//  * jac_block64 gives the block under the rotation as applied: its entries to
//    16 eps' of the block, its off-diagonal to 16 eps' of the former one.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#include <cuda_runtime.h>

static long long __double_as_longlong(double v) { long long b; std::memcpy(&b, &v, 8); return b; }
static float __uint_as_float(unsigned b) { float v; std::memcpy(&v, &b, 4); return v; }
static unsigned __float_as_uint(float v) { unsigned b; std::memcpy(&b, &v, 4); return b; }
static int __double2hiint(double v) { return (int)(__double_as_longlong(v) >> 32); }
static int __double2loint(double v) { return (int)__double_as_longlong(v); }
static double __hiloint2double(int hi, int lo) {
    const unsigned long long b = ((unsigned long long)(unsigned)hi << 32) | (unsigned)lo;
    double v;
    std::memcpy(&v, &b, 8);
    return v;
}
static int off_ulps = 0;
static float off(float v) { return __uint_as_float(__float_as_uint(v) + off_ulps); }
static float rsqrtf(float x) { return off((float)(1.0 / std::sqrt((double)x))); }
static float __fdividef(float x, float y) { return off(x / y); }
using std::fma;

#include "jac_rot.h"

using namespace mpspt;
typedef long double LD;

int main() {
    std::mt19937_64 g(7);
    std::uniform_real_distribution<double> u(-1.0, 1.0), ex(-30.0, 0.0);
    const LD eps = 0x1p-53L;
    int cases = 0;
    for (int i = 0; i < 400000; ++i) {
        off_ulps = i % 5 - 2;
        const double td = i < 8 ? (i & 1 ? -1.0 : 1.0) : u(g) * std::exp2(i & 1 ? ex(g) : 0.0);
        if (std::fabs(td) < 1e-9) continue;
        const float t = (float)td, dt = i % 3 ? 0.f : t * (float)(u(g) * 0x1p-21);
        double h = jac_half64(t, dt), s = jac_sine64(h);
        const LD nu = (LD)s * ((LD)s * (1.0L + (LD)h * h) - 2.0L * h);
        if (fabsl(nu) > 8.0L * eps * fabsl((LD)s * h)) { printf("t=%.9g: norm off by %.2Le\n", t, nu); return 1; }
        const LD c = 1.0L - (LD)s * h, tx = (LD)t - dt;
        if (fabsl((LD)s / c - tx) > 0x1p-37L * fabsl(tx)) { printf("t=%.9g: angle off by %.2Le\n", t, (LD)s / c / tx - 1.0L); return 1; }
        ++cases;
        // a block under the rotation of its own tangent
        double a = u(g), b = u(g), e = u(g) * std::exp2(ex(g));
        const float fd = d2f_trunc(b - a), fe = d2f_trunc(e), tb = jac_tan(fd, fe);
        h = jac_half64(tb, jac_newton(b - a, e, fd, fe, tb));
        s = jac_sine64(h);
        const LD cc = 1.0L - (LD)s * h;
        const LD e1 = cc * s * ((LD)a - b) + (cc * cc - (LD)s * s) * e;
        const LD a1 = cc * cc * a - 2.0L * cc * s * e + (LD)s * s * b;
        const LD m = fabsl((LD)a) + fabsl((LD)b) + fabsl((LD)e);
        double a2 = a, e2 = e, b2 = b;
        jac_block64(s, h, a2, e2, b2);
        if (fabsl(e2 - e1) > 16.0L * eps * (fabsl((LD)e) + eps * m) || fabsl(a2 - a1) > 16.0L * eps * m) {
            printf("block a=%g b=%g e=%g: %.2Le %.2Le\n", a, b, e, fabsl(e2 - e1) / fabsl((LD)e), fabsl(a2 - a1));
            return 1;
        }
    }
    printf("ok %d\n", cases);
    return 0;
}
