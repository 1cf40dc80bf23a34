// Host check of the float64 eigensolver's dispatch rule (eig_route.h).  A
// cluster is 8 CTAs: no call of equal matrices that one CTA each can hold may
// put more than six of them on an SM (152 SMs) on average, a batch that leaves
// SMs idle takes clusters, small matrices in the batch do not count as large
// ones, and a list sorted by size changes its kernel at most twice.
#include <cstdio>
#include <vector>

#include "eig_route.h"

using namespace mpspt;

int main() {
    int cases = 0;
    for (int n = 1; n <= 2048; n = n < 300 ? n + 1 : n + 97)
        for (int batch = 1; batch <= 1024; batch = batch < 140 ? batch + 1 : batch + 37) {
            const int nt = eig_threads(n, eig_mid_threads_of(batch, [n](int) { return n; }));
            if (nt != 0 && nt != 128 && nt != 256 && nt != 512) return 1;
            if (nt == 0 && n <= kEigOneMaxN && 8 * batch > 6 * 152) { printf("n=%d batch=%d: clusters\n", n, batch); return 1; }
            if (nt == 0 && n <= 64 && 8 * batch > 2 * 152 + 8) { printf("n=%d batch=%d: clusters\n", n, batch); return 1; }
            if (nt != 0 && n >= kEigOneMinN && 8 * batch <= 2 * 152) { printf("n=%d batch=%d: one CTA\n", n, batch); return 1; }
            if (nt != 0 && n > kEigOneMaxN) return 1;
            ++cases;
        }
    for (int small = 0; small <= 900; small += 100) {   // two large matrices among small ones
        std::vector<int> v{600, 200, 190};
        v.insert(v.end(), small, 30);
        v.insert(v.end(), 50, 9);
        const int mid = eig_mid_threads_of((int)v.size(), [&](int i) { return v[i]; });
        if (mid != 0) { printf("%d small matrices\n", small); return 1; }
        int changes = 0;
        for (size_t i = 1; i < v.size(); ++i) changes += eig_threads(v[i], mid) != eig_threads(v[i - 1], mid);
        if (changes > 2) return 1;
        ++cases;
    }
    printf("ok %d\n", cases);
    return 0;
}
