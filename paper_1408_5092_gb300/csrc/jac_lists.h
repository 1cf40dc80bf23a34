// Sizes of the mixed eigensolver's device scratch, per matrix.
#pragma once
#include <cstddef>

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

}  // namespace mpspt
