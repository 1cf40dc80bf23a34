// Pair schedules of the batched Jacobi eigensolver (kernels_eig.cu).  Host
// and device code: the host tests check the schedules' coverage.
#pragma once

#if defined(__CUDACC__)
#define JAC_HD __host__ __device__ __forceinline__
#else
#define JAC_HD inline
#endif

namespace mpspt {

// Round-robin ordering: in round r (0 <= r < m - 1) slot k pairs (pa, pb);
// over the m - 1 rounds every pair of 0 .. m-1 meets exactly once.
JAC_HD void rr_pair(int k, int r, int m, int& pa, int& pb) {
    pa = (k == 0) ? 0 : ((k - 1 + r) % (m - 1)) + 1;
    pb = ((m - 1 - k - 1 + r) % (m - 1)) + 1;
}

// Pair schedule of one sweep: the round-robin ordering, m - 1 rounds of
// m/2 slots (m = n rounded up to even).  A slot is a pair (p < q) or a
// single index (q = -1) that is not rotated in that round; every index is
// in exactly one slot per round, so the 2x2 block update over all slot
// pairs touches every matrix entry once, and every pair meets once per
// sweep.  (The kernels work out the same pairs in place; the host check of
// the ordering goes by this.)
struct Sched {
    int n, m, half;
    JAC_HD void init(int n_) {
        n = n_; m = n + (n & 1); half = m / 2;
    }
    JAC_HD int rounds() const { return m - 1; }
    JAC_HD int slots(int) const { return half; }
    JAC_HD void slot(int r, int k, int& p, int& q) const {
        int x, y;
        rr_pair(k, r, m, x, y);
        p = x < y ? x : y;
        q = x < y ? y : x;
        if (q >= n) q = -1;
    }
};

// The same ordering with the entries addressed by slot position: slot k holds
// positions k and m-1-k.  Position 0 keeps its player, the others move down by
// one after every round (1 to m-1), so the player at position j >= 1 of round
// r is ((j - 1 + r) mod (m - 1)) + 1 and after m - 1 rounds everybody is back.
JAC_HD int next_pos(int m, int j) { return j == 0 ? 0 : j == 1 ? m - 1 : j - 1; }
// Place of the entry of positions a < b among m (m - 1) / 2: where a + b < m
// row a, consecutive in b; where a + b >= m row b, consecutive in a.  The four
// entries of a block of slots (k, l), k < l, are then each consecutive in l
// for a fixed k (a packed upper triangle puts two of them in its columns, and
// a warp's accesses to those fell on the same banks three or four at a time).
JAC_HD int tri(int m, int a, int b) {
    const int half = m / 2;
    if (a + b < m) return a * (m - a) + (b - a - 1);
    return half * half + (b - half) * (b - half - 1) + (a - (m - b));
}
// place of the same two players' entry in the next round
JAC_HD int tri_next(int m, int a, int b) {
    const int x = next_pos(m, a), y = next_pos(m, b);
    return x < y ? tri(m, x, y) : tri(m, y, x);
}
// Block number e in [0, half (half - 1) / 2) -> slots k < l: the rows of the
// strict triangle folded in pairs of one length, so that consecutive numbers
// stay in one row for as long as possible.
JAC_HD void block_slots(int half, int e, int& k, int& l) {
    const int W = (half & 1) ? half : half - 1;
    const int i = e / W, j = e - i * W;
    const int len = half - 1 - i;   // blocks of row i
    if (j < len) {
        k = i;
        l = i + 1 + j;
    } else {
        k = (half & 1) ? half - 2 - i : half - 1 - i;
        l = k + 1 + (j - len);
    }
}

}  // namespace mpspt
