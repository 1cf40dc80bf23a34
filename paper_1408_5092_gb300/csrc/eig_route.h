// Which kernel of the float64 eigensolver (kernels_eig.cu) takes a matrix:
// one CTA below n = 28, a cluster of 8 CTAs above n = 215 (whose triangle does
// not fit into one CTA's shared memory), and between them one of the two for
// all matrices of a call.
//
// A cluster divides a matrix's float64 operations by eight, but each of its
// CTAs computes all rotations and its barriers are dearer, so it pays while SMs
// would otherwise be idle: up to two CTAs per SM (38 matrices) for n up to 64,
// four (76) up to 112 and six (114) above, where more of the time is the
// divided part.  Matrices are counted by n^2 against the largest, since a few
// large ones end last whatever the small ones do.  Beyond that a CTA per
// matrix, with the more threads the larger n.
// Measured (ms; cluster / one CTA; equal sizes): n = 32, 24 matrices 1.1 / 1.0,
// 152: 4.6 / 1.0; n = 48, 24: 1.7 / 2.3, 40: 3.2 / 2.3, 1000: 42.6 / 9.9; n = 90,
// 64: 10.3 / 11.6, 100: 15.4 / 11.6; n = 128, 64: 23.0 / 28.6, 152: 55.5 / 28.6;
// n = 200, 100: 111 / 118, 152: 180 / 118.  Threads of the one CTA, 512 matrices
// (128 / 256 / 512): n = 32 1.9 / 2.3 / 3.6; n = 64 12.5 / 13.3 / 16; n = 90 41.8 /
// 38.4 / 43; n = 128 170 / 117 / 114; up to 304 matrices (two CTAs per SM) 256.
#pragma once

namespace mpspt {

constexpr int kEigOneMinN = 28, kEigOneMaxN = 215;

// The matrices of size kEigOneMinN to kEigOneMaxN: threads of their CTA, 0: a
// cluster each.  nmax: the largest; count: the sum of n^2 / nmax^2.
constexpr int eig_mid_threads(int nmax, double count) {
    if (count < (nmax > 112 ? 114.0 : nmax > 64 ? 77.0 : 39.0)) return 0;
    return nmax > 112 ? 512 : nmax <= 64 && count > 304.0 ? 128 : 256;
}
constexpr int eig_threads(int n, int mid) { return n < kEigOneMinN ? 128 : n > kEigOneMaxN ? 0 : mid; }

// sizes n(i), i < batch
template <class N>
int eig_mid_threads_of(int batch, const N& n) {
    int nmax = 0;
    double sum = 0.0;
    for (int i = 0; i < batch; ++i)
        if (n(i) >= kEigOneMinN && n(i) <= kEigOneMaxN) {
            nmax = n(i) > nmax ? n(i) : nmax;
            sum += (double)n(i) * n(i);
        }
    return nmax ? eig_mid_threads(nmax, sum / ((double)nmax * nmax)) : 0;
}

}  // namespace mpspt
