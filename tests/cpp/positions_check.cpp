// Host check of the position-addressed form of the Jacobi schedule
// (jacobi_schedule.h): entries that are read at their slots' positions and
// written to the next round's must always belong to the pairs that rr_pair
// names, every entry must be written once per round, the blocks must be every
// pair of slots once, and a sweep must bring every entry back.
#include <cstdio>
#include <vector>

#include "jacobi_schedule.h"

using namespace mpspt;

int main() {
    int cases = 0;
    for (int m = 2; m <= 64; m += 2) {
        const int half = m / 2, np = m * (m - 1) / 2;
        std::vector<int> cur(np, -1), nxt;
        auto label = [m](int x, int y) { return x < y ? x * m + y : y * m + x; };
        for (int a = 0; a < m; ++a)
            for (int b = a + 1; b < m; ++b) cur[tri(m, a, b)] = label(a, b);
        const std::vector<int> start = cur;
        for (int r = 0; r < m - 1; ++r) {
            nxt.assign(np, -1);
            std::vector<int> wrote(np, 0), seen(half * half, 0);
            auto move = [&](int a, int b, int want) {
                const int from = tri(m, a, b), to = tri_next(m, a, b);
                if (cur[from] != want) { printf("m=%d r=%d (%d,%d) holds %d, not %d\n", m, r, a, b, cur[from], want); return false; }
                nxt[to] = cur[from];
                return ++wrote[to] == 1;
            };
            for (int k = 0; k < half; ++k) {
                int x, y;
                rr_pair(k, r, m, x, y);
                if (!move(k, m - 1 - k, label(x, y))) return 1;
            }
            for (int e = 0; e < half * (half - 1) / 2; ++e) {
                int k, l, x, y, u, v;
                block_slots(half, e, k, l);
                if (!(0 <= k && k < l && l < half) || seen[k * half + l]++) { printf("block m=%d e=%d\n", m, e); return 1; }
                rr_pair(k, r, m, x, y);
                rr_pair(l, r, m, u, v);
                const int kb = m - 1 - k, lb = m - 1 - l;
                if (!move(k, l, label(x, u)) || !move(k, lb, label(x, v)) || !move(l, kb, label(y, u)) ||
                    !move(lb, kb, label(y, v)))
                    return 1;
            }
            cur = nxt;
        }
        if (cur != start) { printf("m=%d does not come back\n", m); return 1; }
        ++cases;
    }
    printf("ok %d\n", cases);
    return 0;
}
