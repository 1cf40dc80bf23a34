// Sizes of the mixed eigensolver's device scratch, per matrix.
#pragma once
#include <cstddef>
#include <vector>

namespace mpspt {

// rotation-list entries of one sweep: m - 1 rounds of m / 2 slots
constexpr size_t jac_rot_entries(int n) { return (size_t)(n + (n & 1) - 1) * ((n + (n & 1)) / 2); }
// global float32 triangles of the mixed sweeps (0: in shared memory)
constexpr size_t jac_e_bytes(int n) { return n <= 236 ? 0 : (size_t)4 * (n + (n & 1)) * (n + (n & 1) - 1); }

constexpr int kStartSweeps = 12;                 // float32 start (a cap is not an error: the polish follows)
constexpr int kPolishSweeps = 8;                 // sweeps of one polish round
constexpr size_t kListBytes = (size_t)32 << 20;  // rotation lists of one launch, per matrix
// Sweeps of one launch: what the matrix's own lists allow (all twelve up to n =
// 590), whatever it is batched with.
constexpr int jac_sweep_cap(int n) {
    const size_t s = kListBytes / (jac_rot_entries(n) * 16);
    return s < 1 ? 1 : s > (size_t)kStartSweeps ? kStartSweeps : (int)s;
}

constexpr size_t jac_a16(size_t b) { return (b + 15) & ~(size_t)15; }
constexpr size_t jac_rot_bytes(int n) { return jac_a16(jac_rot_entries(n) * jac_sweep_cap(n) * 8); }
constexpr size_t jac_rot64_bytes(int n) {
    return jac_a16(jac_rot_entries(n) * (jac_sweep_cap(n) < kPolishSweeps ? jac_sweep_cap(n) : kPolishSweeps) * 16);
}
// One matrix's share: two n x n float64 work matrices, both lists, triangles.
constexpr size_t eig_scratch_bytes(int n) {
    return 16 * (size_t)n * n + jac_rot_bytes(n) + jac_rot64_bytes(n) + jac_a16(jac_e_bytes(n));
}

// A batch is solved in groups that use the same scratch in turn (nothing of it
// outlives a launch but V and the flags).  First members of the groups of sizes
// n(0 .. count): each takes as many matrices as fit into `budget` bytes, one at
// least.
constexpr size_t kEigScratch = (size_t)1 << 30;   // 500 of 128 x 128 or 140 of 236 x 236
template <class N>
std::vector<int> eig_groups(int count, const N& n, size_t budget) {
    std::vector<int> first;
    size_t sum = 0;
    for (int i = 0; i < count; ++i) {
        const size_t b = eig_scratch_bytes(n(i));
        if (first.empty() || sum + b > budget) {
            first.push_back(i);
            sum = 0;
        }
        sum += b;
    }
    return first;
}
// The groups of the largest budget, from kEigScratch down by halves, whose
// scratch try_alloc(bytes) can provide; empty if one matrix at a time is too much.
template <class N, class Try>
std::vector<int> eig_fit_groups(int count, const N& n, const Try& try_alloc) {
    for (size_t budget = kEigScratch;; budget /= 2) {
        const std::vector<int> first = eig_groups(count, n, budget);
        size_t need = 0;
        for (size_t g = 0; g < first.size(); ++g) {
            size_t sum = 0;
            for (int i = first[g]; i < (g + 1 < first.size() ? first[g + 1] : count); ++i) sum += eig_scratch_bytes(n(i));
            need = sum > need ? sum : need;
        }
        if (try_alloc(need)) return first;
        if ((int)first.size() == count) return {};
    }
}

}  // namespace mpspt
