#include "eig.h"
#include "jac_lists.h"

#include <algorithm>
#include <array>
#include <cstring>
#include <numeric>

namespace mpspt {

namespace {
constexpr int kMaxSweepsF64 = 60;    // float64 Jacobi from the identity
constexpr int kMaxRounds = 60;       // polish rounds
size_t a16(size_t b) { return (b + 15) & ~(size_t)15; }

// Host image of several device arrays, sent with one copy.
struct Blob {
    std::vector<unsigned char> h;
    template <class T>
    size_t add(const std::vector<T>& v) {
        const size_t o = a16(h.size());
        h.resize(o + v.size() * sizeof(T));
        if (!v.empty()) std::memcpy(h.data() + o, v.data(), v.size() * sizeof(T));
        return o;
    }
};
}  // namespace

// Counters of the tasks behind the flags: sweeps of the last launch, of the
// start, of the polish (which = 1, 2).
void EigSolver::count(long long (&acc)[3], int which, cudaStream_t st) {
    if (!stats || groups.empty()) return;   // diagnostics; synchronises
    std::vector<int> k((size_t)nflags * 3);
    MPSPT_CUDA(cudaMemcpyAsync(k.data(), flags.as<int>() + nflags, k.size() * sizeof(int), cudaMemcpyDeviceToHost, st));
    MPSPT_CUDA(cudaStreamSynchronize(st));
    for (int i = 0; i < nflags; ++i) {
        acc[0] += k[(size_t)3 * i + which];
        acc[1] += 1;
        acc[2] = std::max<long long>(acc[2], k[(size_t)3 * i + which]);
    }
}

// Plain float64 sweeps from the identity (a work copy where the solver needs
// one: matrices whose triangle does not fit into a cluster's shared memory).
void EigSolver::fp64(const std::vector<EigTask>& et, cudaStream_t st) {
    std::vector<EigTask> t = et;
    order_eig_tasks(t.data(), (int)t.size());
    size_t tot = 0;
    for (const auto& x : t)
        if (eig_in_place(x.n)) tot += (size_t)x.n * x.n;
    scratch.ensure((tot + 1) * sizeof(double), st);
    double* p = scratch.as<double>();
    for (auto& x : t)
        if (eig_in_place(x.n)) {
            MPSPT_CUDA(cudaMemcpyAsync(p, x.A, (size_t)x.n * x.n * sizeof(double), cudaMemcpyDeviceToDevice, st));
            x.A = p;
            p += (size_t)x.n * x.n;
        }
    upload(blob, t, st);
    launch_eig(blob.as<EigTask>(), t.data(), (int)t.size(), true, kMaxSweepsF64, flags.as<int>(), st);
}

void EigSolver::run(const std::vector<EigTask>& et_in, bool fp64_only, cudaStream_t st) {
    groups.clear();
    nflags = nround = 0;
    if (et_in.empty()) return;
    for (const auto& t : et_in) {
        require(t.n >= 1 && t.n <= 2048, "eigenproblem size must be in [1, 2048]");
        check_range(t.A, (size_t)t.n * t.n * sizeof(double), "eig A");
        check_range(t.V, (size_t)t.n * t.n * sizeof(double), "eig V");
        check_range(t.w, (size_t)t.n * sizeof(double), "eig w");
    }
    nflags = (int)et_in.size();
    flags.ensure((size_t)nflags * 4 * sizeof(int) + 16, st);
    if (fp64_only) {
        fp64(et_in, st);
        return;
    }
    // matrices whose float32 triangles fit into shared memory first
    std::vector<EigTask> et;
    for (int big = 0; big < 2; ++big)
        for (const auto& t : et_in)
            if ((jac_e_bytes(t.n) > 0) == (big != 0)) et.push_back(t);
    const std::vector<int> first = eig_fit_groups(nflags, [&](int i) { return et[i].n; }, [&](size_t bytes) {
        try {
            scratch.ensure(bytes, st);
            return true;
        } catch (const Error& e) {
            if (e.status != MPSPT_ERR_OOM) throw;
            cudaGetLastError();
            return false;
        }
    });
    require(!first.empty(), "eigensolver scratch", MPSPT_ERR_OOM);

    // batched products C_i = op(A_i) B_i; all have the same block list but for
    // the pointers (and the Newton-Schulz form 3/2 I - 1/2 X of the output)
    enum Src { TA, TV, TVT, TG };
    struct Prod { Src a; int trans; Src b, c; bool ns; };
    static const Prod prods[] = {
        {TV, 1, TV, TG, true},      // G = 3/2 I - 1/2 V^T V
        {TV, 0, TG, TVT, false},    // Vt = V G
        {TVT, 1, TVT, TG, true},    // G = 3/2 I - 1/2 Vt^T Vt
        {TVT, 0, TG, TV, false},    // V = Vt G
        {TA, 0, TV, TVT, false},    // Vt = A V
        {TV, 1, TVT, TG, false},    // B = V^T Vt
    };
    Blob blb;
    size_t pe_max = 0, tk_max = 0;
    std::vector<std::array<size_t, 6>> at;   // places of each group's lists in the blob
    for (size_t q = 0; q < first.size(); ++q) {
        Group gr;
        gr.first = first[q];
        gr.ntask = (q + 1 < first.size() ? first[q + 1] : nflags) - gr.first;
        const EigTask* t0 = et.data() + gr.first;
        unsigned char* p = static_cast<unsigned char*>(scratch.get());
        const unsigned char* end = p + scratch.bytes();
        std::vector<double*> vt(gr.ntask), g(gr.ntask);
        std::vector<JacTask> start, polish;
        std::vector<JacRows> rows;
        ge.clear();
        for (int i = 0; i < gr.ntask; ++i) {
            const int n = t0[i].n;
            gr.nmax = std::max(gr.nmax, n);
            if (jac_e_bytes(n) == 0) {
                ++gr.nsmall;
                gr.nmax_small = std::max(gr.nmax_small, n);
            }
            vt[i] = reinterpret_cast<double*>(p);
            g[i] = vt[i] + (size_t)n * n;
            unsigned char* R = p + 16 * (size_t)n * n;
            unsigned char* R64 = R + jac_rot_bytes(n);
            unsigned char* P = R64 + jac_rot64_bytes(n);
            p += eig_scratch_bytes(n);
            require(p <= end, "eigensolver scratch");
            int* cnt = flags.as<int>() + nflags + 3 * (gr.first + i);
            JacTask t{t0[i].A, t0[i].V, nullptr, P, reinterpret_cast<float2*>(R), reinterpret_cast<double2*>(R64),
                      flags.as<int>() + gr.first + i, cnt, cnt + 1, n, jac_sweep_cap(n)};
            start.push_back(t);
            t.A = g[i];
            t.w = t0[i].w;
            t.total += 1;
            polish.push_back(t);
            for (int r0 = 0; r0 < n; r0 += JAC_APPLY_ROWS) rows.push_back({i, r0, std::min(JAC_APPLY_ROWS, n - r0), 0});
            const int m0 = ge.mark();
            ge.op(t0[i].V, n, t0[i].V, n, n, 0, 1.0);
            ge.block(g[i], n, n, n, 0, m0);
        }
        gr.nrows = (int)rows.size();
        std::vector<GemmBlk> gb, blks;
        std::vector<unsigned> ub;
        size_t pe = 0, tk = 0;
        gr.tile = ge.tile_rule();
        ge.units(gr.tile, gb, ub, nullptr, &pe, &tk);
        gr.nunit = (int)ub.size();
        pe_max = std::max(pe_max, pe);
        tk_max = std::max(tk_max, tk);
        auto ptr = [&](Src s, int i) -> double* {
            switch (s) {
                case TA: return const_cast<double*>(t0[i].A);
                case TV: return t0[i].V;
                case TVT: return vt[i];
                default: return g[i];
            }
        };
        std::vector<GemmOp> ops;
        for (const Prod& pr : prods) {
            const int o0 = (int)ops.size();
            for (int i = 0; i < gr.ntask; ++i) {
                const int n = t0[i].n;
                ops.push_back({ptr(pr.a, i), ptr(pr.b, i), n, n, n, pr.trans, 1.0});
            }
            for (const GemmBlk& b0 : gb) {   // b0.op0: the block's task
                GemmBlk b = b0;
                b.C = ptr(pr.c, b0.op0);
                b.op0 = o0 + b0.op0;
                b.op1 = b.op0 + 1;
                if (pr.ns) {
                    b.scale = -0.5f;
                    b.diag = 1.5f;
                }
                blks.push_back(b);
            }
        }
        at.push_back({blb.add(start), blb.add(polish), blb.add(rows), blb.add(blks), blb.add(ub), blb.add(ops)});
        groups.push_back(gr);
    }
    ge.workspace(pe_max, tk_max, st);
    upload(blob, blb.h, st);
    const unsigned char* d = static_cast<const unsigned char*>(blob.get());
    for (size_t q = 0; q < groups.size(); ++q) {
        Group& gr = groups[q];
        gr.start = reinterpret_cast<const JacTask*>(d + at[q][0]);
        gr.polish = reinterpret_cast<const JacTask*>(d + at[q][1]);
        gr.rows = reinterpret_cast<const JacRows*>(d + at[q][2]);
        gr.blk = reinterpret_cast<const GemmBlk*>(d + at[q][3]);
        gr.unit = reinterpret_cast<const unsigned*>(d + at[q][4]);
        gr.ops = reinterpret_cast<const GemmOp*>(d + at[q][5]);
        launch_jac_mixed(gr.start, gr.nsmall, gr.nmax_small, false, st);
        launch_jac_mixed(gr.start + gr.nsmall, gr.ntask - gr.nsmall, gr.nmax, false, st);
        launch_jac_apply(gr.start, gr.rows, gr.nrows, gr.nmax, true, true, st);
        for (int j = 0; j < 4; ++j) product(gr, j, st);
        rounds(gr, 2, st);
    }
    nround = 2;
    count(sweeps32, 1, st);
}

void EigSolver::product(const Group& g, int j, cudaStream_t st) {
    launch_dgemm(g.tile, g.blk + (size_t)j * g.ntask, g.unit, g.nunit, g.ops, ge.dpart.as<double>(),
                 ge.dtick.as<unsigned>(), st);
}

void EigSolver::rounds(const Group& g, int n, cudaStream_t st) {
    for (int r = 0; r < n; ++r) {
        product(g, 4, st);
        product(g, 5, st);
        launch_jac_mixed(g.polish, g.nsmall, g.nmax_small, true, st);
        launch_jac_mixed(g.polish + g.nsmall, g.ntask - g.nsmall, g.nmax, true, st);
        launch_jac_rot64(g.polish, g.ntask, st);
        launch_jac_apply(g.polish, g.rows, g.nrows, g.nmax, false, false, st);
    }
}

bool EigSolver::again(const int* flags_host, cudaStream_t st) {
    bool more = false;
    for (const Group& g : groups) {
        bool all = true;
        for (int i = 0; i < g.ntask; ++i) all = all && flags_host[g.first + i] != 0;
        if (all) continue;
        require(nround < kMaxRounds, "eigensolver: round cap reached before the convergence test", MPSPT_ERR_NOT_CONVERGED);
        rounds(g, 2, st);
        more = true;
    }
    nround += 2;
    if (!more) {
        count(sweeps_polish, 2, st);
        groups.clear();
    }
    return more;
}

}  // namespace mpspt
