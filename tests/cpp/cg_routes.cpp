// Sweeps of one problem with the small local solves on a cluster, and with every
// cluster launch refused.  Arguments: problem file (k_act, k_virt, n_elec, n_chol
// as int64, then h, L, ci as float64), bond dimensions.  Prints per run: M,
// graphs, refused, local solves on a cluster, launches, CG iterations, float64
// applications, their counted flops, E2 per sweep.
#include <cstdio>
#include <cstdlib>
#include <fstream>

#include "../../paper_1408_5092_gb300/csrc/engine.h"

using namespace mpspt;

static bool refuse(const CgArgs&, cudaStream_t) { return false; }

int main(int argc, char** argv) {
    std::ifstream f(argv[1], std::ios::binary);
    long long d[4];
    f.read(reinterpret_cast<char*>(d), sizeof(d));
    const size_t k = (size_t)(d[0] + d[1]);
    std::vector<double> h(k * k), L((size_t)d[3] * k * k), ci((size_t)1 << (2 * d[0]));
    for (auto* v : {&h, &L, &ci}) f.read(reinterpret_cast<char*>(v->data()), (std::streamsize)(v->size() * 8));
    if (!f) return 2;
    cudaStream_t own;
    MPSPT_CUDA(cudaStreamCreate(&own));
    for (int a = 2; a < argc; ++a)
        for (int mode = 0; mode < 4; ++mode) {
            mpspt_options o;
            mpspt_default_options(&o);
            o.max_sweeps = 2;
            o.e_tol = 1e-14;
            o.cuda_graphs = mode & 1;
            o.stream = (mode & 1) ? own : nullptr;
            Ctx c(o);
            set_integrals(c, (int)d[0], (int)d[1], (int)d[2], h.data(), L.data(), (int)d[3]);
            set_reference(c, ci.data(), (long long)ci.size());
            if (mode & 2) c.cg_cluster = &refuse;
            SweepResult r;
            minimize(c, MPSPT_H0_DYALL, std::atoi(argv[a]), r);
            printf("%s %d %d %lld %lld %lld %lld %.17g", argv[a], mode & 1, mode >> 1, r.cluster_solves, r.launches,
                   r.cg_iters, r.sigma64_calls, r.sigma64_flops);
            for (double e : r.e2_sweep) printf(" %.17g", e);
            printf("\n");
        }
    return 0;
}
