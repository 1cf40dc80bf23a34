// Host check of the planners' tables of one MPO: the two-site operator Omega
// of every bond against the plain sum of products in an ordered map (bit for
// bit: both add in the entries' order), and the element lists of every site
// against the entries.  Prints "ok <Omega entries> <elements>".
#include <cstdio>
#include <cstring>
#include <map>
#include <random>
#include <tuple>
#include <vector>

#include "../../paper_1408_5092_gb300/csrc/plans.h"

using namespace mpspt;

int main() {
    size_t no = 0, ne = 0;
    for (int which = 0; which < 3; ++which) {
        const int k = 7, ka = 4;
        std::mt19937 g(which + 1);
        std::uniform_real_distribution<double> u(-1, 1);
        std::vector<double> h(k * k), eri((size_t)k * k * k * k), eps(k);
        for (auto& v : h) v = u(g);
        for (auto& v : eri) v = u(g);
        for (auto& v : eps) v = u(g);
        std::vector<Term> t;
        if (which == 0) {
            add_one_body(t, h, k, 0, ka, 0, ka);
            add_number(t, eps, ka, k);
            t.push_back(Term{-0.5, 0, {}});
        } else if (which == 1) {
            add_one_body(t, h, k, ka, k, 0, ka);
            add_two_body(t, eri, k, 0, k, 0, ka, ka);
        } else {
            add_one_body(t, h, k, 0, k, 0, k);
            add_two_body(t, eri, k, 0, k, 0, k, -1);
        }
        const MPO W = build_mpo(t, k, ka);
        for (int i = 0; i + 1 < k; ++i) {
            std::map<std::tuple<int, int, int, int>, double> acc;   // (a, out, c, in)
            for (const auto& e1 : W.W[i])
                for (const auto& e2 : W.W[i + 1]) {
                    if (e2.a != e1.b) continue;
                    const double cc = e1.coef * e2.coef;
                    for (int s1 = 0; s1 < 4; ++s1)
                        for (int t1 = 0; t1 < 4; ++t1)
                            for (int s2 = 0; s2 < 4; ++s2)
                                for (int t2 = 0; t2 < 4; ++t2) {
                                    const double v1 = W.ops[e1.op][s1 * 4 + t1], v2 = W.ops[e2.op][s2 * 4 + t2];
                                    if (v1 != 0.0 && v2 != 0.0) acc[{e1.a, s1 * 4 + s2, e2.b, t1 * 4 + t2}] += cc * v1 * v2;
                                }
                }
            Omega om;
            om.build(W, i);
            size_t q = 0;
            for (const auto& kv : acc) {
                if (kv.second == 0.0) continue;
                if (q >= om.e.size()) { printf("missing entry, bond %d\n", i); return 1; }
                const Omega::E& e = om.e[q];
                if (std::make_tuple(e.a, e.out, e.c, e.in) != kv.first || std::memcmp(&e.v, &kv.second, 8)) {
                    printf("entry %zu of bond %d differs\n", q, i);
                    return 1;
                }
                if ((int)q < om.begin(e.a, e.out) || (int)q >= om.end(e.a, e.out)) { printf("row index\n"); return 1; }
                ++q;
            }
            if (q != om.e.size() || om.Da != W.dim[i]) { printf("extra entries\n"); return 1; }
            no += q;
        }
        for (int p = 0; p < k; ++p) {
            std::vector<std::vector<MPO::El>> in((size_t)W.dim[p + 1] * 4), out((size_t)W.dim[p] * 4);
            for (const auto& e : W.W[p])   // entries are sorted by (a, b)
                for (int s = 0; s < 4; ++s)
                    for (int x = 0; x < 4; ++x) {
                        const double v = W.ops[e.op][s * 4 + x];
                        if (v == 0.0) continue;
                        in[(size_t)e.b * 4 + s].push_back({e.a, x, e.coef * v});
                        out[(size_t)e.a * 4 + s].push_back({e.b, x, e.coef * v});
                    }
            auto same = [&](const std::vector<std::vector<MPO::El>>& ref, const std::vector<MPO::El>& el, const std::vector<int>& at) {
                if (at.size() != ref.size() + 1) return false;
                for (size_t r = 0; r < ref.size(); ++r) {
                    if (at[r + 1] - at[r] != (int)ref[r].size()) return false;
                    for (size_t q = 0; q < ref[r].size(); ++q) {
                        const MPO::El &x = el[at[r] + q], &y = ref[r][q];
                        if (x.x != y.x || x.t != y.t || x.v != y.v) return false;
                        ++ne;
                    }
                }
                return true;
            };
            if (!same(in, W.in_el[p], W.in_at[p]) || !same(out, W.out_el[p], W.out_at[p])) { printf("elements of site %d\n", p); return 1; }
        }
    }
    printf("ok %zu %zu\n", no, ne);
    return 0;
}
