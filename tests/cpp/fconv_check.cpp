// Host check of the integer float32 -> float64 conversion (fconv.h) against the
// language's: every exponent with random and extreme fractions, subnormals,
// zeros, infinities, and NaN to NaN.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#include <cuda_runtime.h>

static double __hiloint2double(int hi, int lo) {
    const unsigned long long b = ((unsigned long long)(unsigned)hi << 32) | (unsigned)lo;
    double v;
    std::memcpy(&v, &b, 8);
    return v;
}
static int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }

#include "fconv.h"

int main() {
    std::mt19937 g(5);
    int cases = 0;
    for (unsigned sign = 0; sign < 2; ++sign)
        for (unsigned e = 0; e < 256; ++e)
            for (int q = 0; q < 3000; ++q) {
                const unsigned f = q == 0 ? 0u : q == 1 ? 0x7FFFFFu : q == 2 ? 1u : (g() & 0x7FFFFFu) >> (q % 23);
                const unsigned b = sign << 31 | e << 23 | f;
                float v;
                std::memcpy(&v, &b, 4);
                const double want = (double)v, got = mpspt::f2d_int(b);
                if (std::isnan(want) ? !std::isnan(got) : std::memcmp(&want, &got, 8) != 0) {
                    printf("%08x: %.17g, not %.17g\n", b, got, want);
                    return 1;
                }
                ++cases;
            }
    printf("ok %d\n", cases);
    return 0;
}
