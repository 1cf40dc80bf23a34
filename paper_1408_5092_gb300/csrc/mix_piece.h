// The values [e, e + MIX_PIECE) of an operator-weighted block sum, by one warp.
#pragma once
#include "kernels.h"

namespace mpspt {

// COH: the sources may have been written by this launch (no read-only loads)
template <bool COH>
__device__ __forceinline__ void mix_piece(const MixTask& t, int e, const MixSrc* __restrict__ srcs, int lane) {
    const int n = t.rows * t.cols;
    const int e0 = e + lane, e1 = e0 + 32;
    const bool in1 = e1 < n;
    if (e0 >= n) return;
    const int i0 = e0 / t.cols, j0 = e0 - i0 * t.cols;
    const int i1 = in1 ? e1 / t.cols : i0, j1 = in1 ? e1 - i1 * t.cols : j0;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
    for (int q = t.s0; q < t.s1; ++q) {
        const MixSrc m = srcs[q];
        const double *p0 = m.src + (size_t)i0 * m.lds + j0, *p1 = m.src + (size_t)i1 * m.lds + j1;
        s0 = fma(m.coef, COH ? __ldcg(p0) : __ldg(p0), s0);
        s1 = fma(m.coef, COH ? __ldcg(p1) : __ldg(p1), s1);
    }
    t.dst[(size_t)i0 * t.ldd + j0] = s0;
    if (in1) t.dst[(size_t)i1 * t.ldd + j1] = s1;
}

}  // namespace mpspt
