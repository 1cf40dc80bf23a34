// Host check of the mixed eigensolver's scratch sizes (jac_lists.h).  Sweeps of
// a launch are the matrix's own: lists of at most kListBytes (one sweep at
// least), all twelve up to n = 590 whatever else is in the batch.
#include <cstdio>

#include "jac_lists.h"

using namespace mpspt;

int main() {
    int cases = 0;
    for (int n = 1; n <= 2048; ++n) {
        size_t slots = 0;   // the schedule, counted
        const int m = n + (n & 1);
        for (int r = 0; r < m - 1; ++r) slots += m / 2;
        if (jac_rot_entries(n) != slots) { printf("n=%d: entries\n", n); return 1; }
        const int c = jac_sweep_cap(n);
        if (c < 1 || c > 12 || (n <= 590 && c != 12)) { printf("n=%d: %d sweeps\n", n, c); return 1; }
        if (c > 1 && slots * 16 * c > kListBytes) { printf("n=%d: lists\n", n); return 1; }
        if (n > 236 && jac_e_bytes(n) < (size_t)4 * m * (m - 1)) return 1;
        ++cases;
    }
    printf("ok %d\n", cases);
    return 0;
}
