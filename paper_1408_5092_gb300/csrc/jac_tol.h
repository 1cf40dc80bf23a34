// Stopping rules of the Jacobi eigensolvers (so = off(A)^2 without null pairs,
// sa = |A|_F^2).
//
// stop: so <= stop sa; a solve that reached so <= stall sa also ends when a sweep
// shrinks so by less than 19%.
// Null pairs: a pair (p, q) whose 2x2 block has every entry below
// null * |A|_F is neither rotated nor counted in the off-diagonal norm.  Its
// eigenvalues are below 2 null |A|_F, so inside such a cluster the vectors
// are set by rounding anyway; every coupling of a null index to a larger
// entry is still rotated away.  For the density matrices of the truncation
// (positive semidefinite) these are the exactly rank-deficient directions,
// far below the keep threshold; skipping them saves the sweeps the polish
// spent circulating rounding noise inside the null cluster.  The float32
// start sweeps every pair.
#pragma once

#ifdef __CUDACC__
#define MPSPT_HD __host__ __device__ inline
#else
#define MPSPT_HD inline
#endif

namespace mpspt {

struct Tol {
    static constexpr double stop = 1e-30, stall = 1e-8, null = 1e-14;
    // start of the mixed solver: off^2 <= 1e-9 |A|_F^2.  Against 1e-11 it
    // saves one or two float32 sweeps of eight to ten and costs the polish
    // none (graded, rank-deficient and degenerate spectra)
    static constexpr double start = 1e-9;
    // A polish round may be the last one if it started from so <= last sa:
    // float32 resolves 1e-7 of the start's off-norm, so what its rounding leaves
    // is below 1e-16 |A|_F.  Any other round ends at so <= gain of its start.
    static constexpr double gain = 1e-11, last = 1e-18;
};

struct JacStop {
    bool stop, done;   // end of the launch's sweeps; the matrix has converged
};

MPSPT_HD bool jac_stalled(double so, double sa, double prev) { return so <= Tol::stall * sa && so > 0.81 * prev; }

MPSPT_HD JacStop start_stop(double so, double sa, double prev) {
    return {so <= Tol::start * sa || jac_stalled(so, sa, prev), false};
}

// Before sweep s of a polish round; off0: so before its first sweep.  A last
// round meets the stop test after a sweep of its own, which takes out what B
// shows below it and above rounding (n = 3: vectors a third nearer).
MPSPT_HD JacStop polish_stop(int s, double so, double sa, double off0, double prev) {
    const bool last = off0 <= Tol::last * sa;
    const bool met = so <= Tol::stop * sa && (s > 0 || so == 0.0);
    const bool stalled = jac_stalled(so, sa, prev);
    return {met || stalled || (!last && so <= Tol::gain * off0), last && (met || stalled)};
}

}  // namespace mpspt
