// Host check that an operator's element lists are made where they are asked for:
// none by building it, one site and direction at a time, the same list from
// many threads at once, and still right after the operator has been moved.
#include <cstdio>
#include <random>
#include <thread>
#include <vector>

#include "../../paper_1408_5092_gb300/csrc/plans.h"

using namespace mpspt;

int main() {
    const int k = 7, ka = 4;
    std::mt19937 g(2);
    std::uniform_real_distribution<double> u(-1, 1);
    std::vector<double> h(k * k), eri((size_t)k * k * k * k);
    for (auto& v : h) v = u(g);
    for (auto& v : eri) v = u(g);
    std::vector<Term> t;
    add_one_body(t, h, k, 0, k, 0, k);
    add_two_body(t, eri, k, 0, k, 0, k, -1);
    MPO W0 = build_mpo(t, k, ka);
    MPO W = std::move(W0);
    for (int p = 0; p < k; ++p)
        if (W.in_el.l->has(p) || W.out_el.l->has(p)) { printf("lists of site %d made by the builder\n", p); return 1; }
    std::vector<const std::vector<MPO::El>*> seen(8);
    std::vector<std::thread> th;
    for (int i = 0; i < 8; ++i) th.emplace_back([&, i] { seen[i] = &W.in_el[3]; });
    for (auto& x : th) x.join();
    for (int i = 0; i < 8; ++i)
        if (seen[i] != seen[0] || seen[i]->empty()) { printf("thread %d\n", i); return 1; }
    for (int p = 0; p < k; ++p)
        if (W.in_el.l->has(p) != (p == 3) || W.out_el.l->has(p)) { printf("site %d\n", p); return 1; }
    size_t n = 0;
    for (const auto& e : W.W[3])
        for (double v : W.ops[e.op]) n += v != 0.0;
    if (W.in_el[3].size() != n || W.out_el[3].size() != n || W.in_at[3].back() != (int)n) { printf("elements\n"); return 1; }
    printf("ok %zu\n", n);
    return 0;
}
