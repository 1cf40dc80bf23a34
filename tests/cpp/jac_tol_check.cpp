// Host check of the polish's stopping rule (jac_tol.h): over rounds of every
// start and every rate of shrinking, a matrix is done only at off^2 <= 1e-30
// |A|_F^2, or stalled at off^2 <= 1e-8 |A|_F^2 by a sweep that took less than 19%,
// in a round whose start float32 resolves to 1e-16 |A|_F; never without a sweep
// unless nothing is off the diagonal; and every sequence ends.
#include <cmath>
#include <cstdio>
#include <initializer_list>

#include "jac_tol.h"

using namespace mpspt;

int main() {
    int cases = 0;
    for (double sa : {1.0, 0.3, 1e4})
        for (double l0 = -34.0; l0 <= 0.0; l0 += 0.25)
            for (double rate = 0.1; rate <= 16.0; rate += 0.3)
                for (double floor = -40.0; floor <= -10.0; floor += 2.5) {
                    const double off0 = std::pow(10.0, l0) * sa;
                    double so = off0, prev = 1e300;
                    int s = 0;
                    for (;; ++s) {
                        const JacStop q = polish_stop(s, so, sa, off0, prev);
                        const bool stalled = so <= 1e-8 * sa && so > 0.81 * prev;
                        if (q.done && !(q.stop && off0 <= 1e-18 * sa && s > 0 && (so <= 1e-30 * sa || stalled))) {
                            printf("done at so=%g sa=%g off0=%g s=%d\n", so, sa, off0, s);
                            return 1;
                        }
                        if (q.stop) break;
                        if (s > 1000) { printf("no end from off0=%g\n", off0); return 1; }
                        prev = so;
                        so = std::fmax(so * std::pow(10.0, -rate), std::pow(10.0, floor) * sa);
                    }
                    ++cases;
                }
    if (!polish_stop(0, 0.0, 1.0, 0.0, 1e300).done || !polish_stop(0, 0.0, 0.0, 0.0, 1e300).done) return 1;
    const double nan = std::nan("");
    if (polish_stop(0, nan, 1.0, nan, 1e300).stop || polish_stop(1, nan, nan, nan, 1.0).done) return 1;
    printf("ok %d\n", cases);
    return 0;
}
