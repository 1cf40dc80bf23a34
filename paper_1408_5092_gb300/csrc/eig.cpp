#include "eig.h"
#include "jac_lists.h"

#include <algorithm>
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

void EigSolver::count(long long (&acc)[3], const std::vector<JacTask>& jt, cudaStream_t st) {
    if (!stats) return;   // diagnostics; synchronises
    for (const auto& t : jt) {
        int k = 0;
        MPSPT_CUDA(cudaMemcpyAsync(&k, t.total, sizeof(int), cudaMemcpyDeviceToHost, st));
        MPSPT_CUDA(cudaStreamSynchronize(st));
        acc[0] += k;
        acc[1] += 1;
        acc[2] = std::max<long long>(acc[2], k);
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
    ntask = 0;
    nflags = 0;
    if (et_in.empty()) return;
    for (const auto& t : et_in) {
        require(t.n >= 1 && t.n <= 2048, "eigenproblem size must be in [1, 2048]");
        check_range(t.A, (size_t)t.n * t.n * sizeof(double), "eig A");
        check_range(t.V, (size_t)t.n * t.n * sizeof(double), "eig V");
        check_range(t.w, (size_t)t.n * sizeof(double), "eig w");
    }
    nflags = (int)et_in.size();
    flags.ensure((size_t)nflags * sizeof(int) + 16, st);
    if (fp64_only) {
        fp64(et_in, st);
        return;
    }
    // matrices whose float32 triangles fit into shared memory first
    std::vector<EigTask> et;
    for (int big = 0; big < 2; ++big)
        for (const auto& t : et_in)
            if ((jac_e_bytes(t.n) > 0) == (big != 0)) et.push_back(t);
    ntask = (int)et.size();
    nsmall = nmax_small = nmax = nround = 0;
    size_t tot = 0, elems = 0;
    std::vector<size_t> off(ntask), eoff(ntask);
    for (int i = 0; i < ntask; ++i) {
        const int n = et[i].n;
        nmax = std::max(nmax, n);
        if (jac_e_bytes(n) == 0) {
            ++nsmall;
            nmax_small = std::max(nmax_small, n);
        }
        eoff[i] = elems;
        elems += (size_t)n * n;
    }
    auto rot_b = [](int n) { return a16(jac_rot_entries(n) * jac_sweep_cap(n) * sizeof(float2)); };
    auto rot64_b = [](int n) { return a16(jac_rot_entries(n) * std::min(jac_sweep_cap(n), kPolishSweeps) * sizeof(double2)); };
    for (int i = 0; i < ntask; ++i) {
        off[i] = tot;
        tot += rot_b(et[i].n) + rot64_b(et[i].n) + a16(jac_e_bytes(et[i].n)) + 16;
    }
    scratch.ensure(tot + 16, st);
    vt.ensure((elems + 1) * sizeof(double), st);
    g.ensure((elems + 1) * sizeof(double), st);
    unsigned char* base = static_cast<unsigned char*>(scratch.get());
    double *vtp = vt.as<double>(), *gp = g.as<double>();
    std::vector<JacTask> start;
    std::vector<JacRows> rows;
    polish.clear();
    for (int i = 0; i < ntask; ++i) {
        const int n = et[i].n;
        unsigned char* R = base + off[i];
        unsigned char* R64 = R + rot_b(n);
        unsigned char* P = R64 + rot64_b(n);
        unsigned char* S = P + a16(jac_e_bytes(n));
        check_range(R, (size_t)(S + 16 - R), "jacobi scratch");
        JacTask t{et[i].A, et[i].V, nullptr, P, reinterpret_cast<float2*>(R), reinterpret_cast<double2*>(R64),
                  flags.as<int>() + i, reinterpret_cast<int*>(S), reinterpret_cast<int*>(S + 4), n, jac_sweep_cap(n)};
        start.push_back(t);
        t.A = gp + eoff[i];
        t.w = et[i].w;
        t.total += 1;
        polish.push_back(t);
        for (int r0 = 0; r0 < n; r0 += JAC_APPLY_ROWS) rows.push_back({i, r0, std::min(JAC_APPLY_ROWS, n - r0), 0});
    }
    nrows = (int)rows.size();
    // batched products C_i = op(A_i) B_i; all have the same block list but for
    // the pointers (and the Newton-Schulz form 3/2 I - 1/2 X of the output)
    ge.clear();
    for (int i = 0; i < ntask; ++i) {
        const int n = et[i].n, m0 = ge.mark();
        ge.op(et[i].V, n, et[i].V, n, n, 0, 1.0);
        ge.block(gp + eoff[i], n, n, n, 0, m0);
    }
    std::vector<GemmBlk> gb, blks;
    std::vector<unsigned> ub;
    size_t pe = 0, tk = 0;
    const int tile = ge.tile_rule();
    ge.tile64 = tile;
    ge.units(tile, gb, ub, nullptr, &pe, &tk);
    nunit = (int)ub.size();
    ge.workspace(pe, tk, st);
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
    auto ptr = [&](Src s, int i) -> double* {
        switch (s) {
            case TA: return const_cast<double*>(et[i].A);
            case TV: return et[i].V;
            case TVT: return vtp + eoff[i];
            default: return gp + eoff[i];
        }
    };
    std::vector<GemmOp> ops;
    for (const Prod& p : prods) {
        const int o0 = (int)ops.size();
        for (int i = 0; i < ntask; ++i) {
            const int n = et[i].n;
            ops.push_back({ptr(p.a, i), ptr(p.b, i), n, n, n, p.trans, 1.0});
        }
        for (const GemmBlk& b0 : gb) {   // b0.op0: the block's task
            GemmBlk b = b0;
            b.C = ptr(p.c, b0.op0);
            b.op0 = o0 + b0.op0;
            b.op1 = b.op0 + 1;
            if (p.ns) {
                b.scale = -0.5f;
                b.diag = 1.5f;
            }
            blks.push_back(b);
        }
    }
    Blob b;
    const size_t os = b.add(start), op = b.add(polish), orow = b.add(rows), ob = b.add(blks), ou = b.add(ub),
                 oo = b.add(ops);
    upload(blob, b.h, st);
    const unsigned char* d = static_cast<const unsigned char*>(blob.get());
    dtask = reinterpret_cast<const JacTask*>(d + op);
    drows = reinterpret_cast<const JacRows*>(d + orow);
    dblk = reinterpret_cast<const GemmBlk*>(d + ob);
    dunit = reinterpret_cast<const unsigned*>(d + ou);
    dops = reinterpret_cast<const GemmOp*>(d + oo);
    const JacTask* ds = reinterpret_cast<const JacTask*>(d + os);
    launch_jac_mixed(ds, nsmall, nmax_small, false, st);
    launch_jac_mixed(ds + nsmall, ntask - nsmall, nmax, false, st);
    launch_jac_apply(ds, drows, nrows, nmax, true, true, st);
    count(sweeps32, start, st);
    for (int j = 0; j < 4; ++j) product(j, st);
    rounds(2, st);
}

void EigSolver::product(int j, cudaStream_t st) {
    launch_dgemm(ge.tile64, dblk + (size_t)j * ntask, dunit, nunit, dops, ge.dpart.as<double>(), ge.dtick.as<unsigned>(), st);
}

void EigSolver::rounds(int n, cudaStream_t st) {
    for (int r = 0; r < n; ++r, ++nround) {
        product(4, st);
        product(5, st);
        launch_jac_mixed(dtask, nsmall, nmax_small, true, st);
        launch_jac_mixed(dtask + nsmall, ntask - nsmall, nmax, true, st);
        launch_jac_rot64(dtask, ntask, st);
        launch_jac_apply(dtask, drows, nrows, nmax, false, false, st);
    }
}

bool EigSolver::again(const int* flags_host, cudaStream_t st) {
    bool all = true;
    for (int i = 0; i < nflags; ++i) all = all && flags_host[i] != 0;
    if (all || ntask == 0) {
        count(sweeps_polish, polish, st);
        polish.clear();
        return false;
    }
    require(nround < kMaxRounds, "eigensolver: round cap reached before the convergence test", MPSPT_ERR_NOT_CONVERGED);
    rounds(2, st);
    return true;
}

}  // namespace mpspt
