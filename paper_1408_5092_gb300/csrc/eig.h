// Batched symmetric eigen-decomposition of the truncation step's density
// matrices (one dense block per composite QN sector).
#pragma once
#include <vector>

#include "core.h"
#include "kernels.h"
#include "plans.h"

namespace mpspt {

struct EigSolver {
    // per task of the last run: 0 another round is needed, 1 converged, 2
    // stopped by the sweep cap (device ints, valid once the stream has
    // reached them; see again)
    DBuf flags;
    int nflags = 0;
    bool stats = false;   // count sweeps per matrix (sum, matrices, max)
    long long sweeps32[3] = {0, 0, 0}, sweeps_polish[3] = {0, 0, 0};

    // For every task: A (n x n, symmetric, left unchanged) -> V (eigenvectors
    // as columns) and w (unsorted eigenvalues).  All pointers must lie in
    // library allocations.  fp64_only: float64 Jacobi from the identity.
    // Otherwise (the float64 pipe is the scarce one on this GPU):
    //  1. cyclic Jacobi in float32 from the identity, giving V orthonormal to
    //     float32 rounding;
    //  2. two Newton-Schulz steps V <- V (3/2 I - 1/2 V^T V) in float64, each
    //     squaring the departure from orthonormality;
    //  3. rounds of: B = V^T A V in float64; Jacobi sweeps on B with its
    //     diagonal in float64 and its off-diagonal part (3e-5 |A| in the first
    //     round, about 1e-11 in the second) in float32; V <- V R with the
    //     rotations in float64.  Float32 resolves an off-diagonal part to 1e-7
    //     of itself, so a round that starts below 1e-9 |A| ends at float64
    //     rounding and is the last.  Two rounds are enqueued.
    // Scratch: up to kEigScratch bytes, less where the device has less to give.
    void run(const std::vector<EigTask>& et, bool fp64_only, cudaStream_t st);
    // With the flags of the last run on the host: false if all are set, else
    // enqueues two more rounds for the matrices that need them (w and flags
    // have to be read again) and returns true.  A matrix that needs more than
    // the cap of rounds is an error.
    bool again(const int* flags_host, cudaStream_t st);

  private:
    // matrices that are solved side by side (jac_lists.h): sizes, and the device
    // lists in blob
    struct Group {
        int first = 0, ntask = 0, nsmall = 0, nmax_small = 0, nmax = 0, nrows = 0, nunit = 0, tile = 16;
        const JacTask *start = nullptr, *polish = nullptr;   // (polish: input B); small matrices first
        const JacRows* rows = nullptr;
        const GemmBlk* blk = nullptr;                        // ntask blocks per product
        const unsigned* unit = nullptr;
        const GemmOp* ops = nullptr;
    };
    void fp64(const std::vector<EigTask>& et, cudaStream_t st);
    void rounds(const Group& g, int n, cudaStream_t st);
    void product(const Group& g, int j, cudaStream_t st);
    void count(long long (&acc)[3], int which, cudaStream_t st);
    DBuf scratch, blob;
    GemmPlan ge;                // shape of the batched square products
    std::vector<Group> groups;
    int nround = 0;
};

}  // namespace mpspt
