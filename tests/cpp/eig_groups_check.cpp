// Host check of how the mixed eigensolver divides a batch (jac_lists.h): every
// matrix in one group, in order; a group's scratch within the budget unless it
// is a single matrix; one group while it fits; and against an allocator with
// less to give, the largest groups that it can hold, or none.  Where one
// launch per sweep had its 4 n^2 doubles a matrix, a batch still fits if its
// largest matrix does.
#include <cstdio>
#include <initializer_list>
#include <random>

#include "jac_lists.h"

using namespace mpspt;

int main() {
    int cases = 0;
    std::mt19937 g(3);
    for (int c = 0; c < 400; ++c) {
        const int count = 1 + (int)(g() % 1024), top = 1 + (int)(g() % (c % 4 ? 300 : 2048));
        std::vector<int> v(count);
        size_t all = 0, largest = 0, before = 0;
        for (int& n : v) {
            n = 1 + (int)(g() % top);
            const size_t b = eig_scratch_bytes(n);
            all += b;
            largest = b > largest ? b : largest;
            before += (size_t)32 * n * n;
        }
        auto n = [&](int i) { return v[i]; };
        for (size_t budget : {(size_t)0, largest, all / 3, all, all + 1}) {
            const std::vector<int> f = eig_groups(count, n, budget);
            if (f.empty() || f[0] != 0) return 1;
            for (size_t q = 0; q < f.size(); ++q) {
                const int end = q + 1 < f.size() ? f[q + 1] : count;
                if (end <= f[q]) { printf("empty group\n"); return 1; }
                size_t sum = 0;
                for (int i = f[q]; i < end; ++i) sum += eig_scratch_bytes(v[i]);
                if (sum > budget && end - f[q] > 1) { printf("group over its budget\n"); return 1; }
            }
            if (budget >= all && f.size() != 1) { printf("more groups than needed\n"); return 1; }
        }
        for (size_t have : {all, all / 2, largest + largest / 2, largest, largest - 1}) {
            size_t asked = 0;
            const std::vector<int> f = eig_fit_groups(count, n, [&](size_t b) { asked = b; return b <= have; });
            if (f.empty() != (have < largest)) { printf("have %zu of %zu\n", have, largest); return 1; }
            if (!f.empty() && asked > have) return 1;
            if (have >= all && all <= kEigScratch && f.size() != 1) return 1;
        }
        if (count >= 16 && before >= largest &&
            eig_fit_groups(count, n, [&](size_t b) { return b <= before; }).empty()) { printf("%d matrices no longer fit\n", count); return 1; }
        ++cases;
    }
    printf("ok %d\n", cases);
    return 0;
}
