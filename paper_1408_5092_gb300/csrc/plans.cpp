// Task-list planner for the block-sparse contractions of the sweep.
#include "plans.h"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <map>
#include <tuple>

namespace mpspt {

void GemmPlan::block(double* C, int ldc, int m, int n, int accumulate, int op0, long long cmap_off,
                     int cmap_rows) {
    if (m <= 0 || n <= 0) return;
    const int op1 = (int)ops.size();
    for (int o = op0; o < op1; ++o) flops += 2.0 * m * n * ops[o].k;
    blocks.push_back({C, cmap_off, ldc, m, n, accumulate, op0, op1, cmap_rows});
}

int GemmPlan::kchunks(long long m, long long n, long long K) {
    if (K < 1024 || m * n > 128LL * 512) return 1;
    return (int)std::min<long long>(8, K / 512);
}

void GemmPlan::split(int tm_, int tn_, std::vector<GemmTask>& out, std::vector<long long>* cm,
                     std::vector<SplitRed>* rd, std::vector<long long>* rcm, size_t* part_elems) const {
    out.clear();
    if (cm) cm->clear();
    if (rd) rd->clear();
    if (rcm) rcm->clear();
    size_t pe = 0;
    // tensor-core plans: the stages of 64 K are cut so that 304 CTAs (two a
    // SM) of equal length would cover the plan, but into no chunk of fewer
    // than two stages nor a block into more than 32.  A stage is bound by its
    // operand staging (1.3 us), so the longest chunk sets the launch's time:
    // with chunks of 512 K and more, and none below K = 1024, most launches
    // ran 8 to 16 stages on a few dozen CTAs (36.3 -> 31.3 us a launch in the
    // M = 256 sweep, integer float32 -> float64 stores included).
    auto stages = [](long long K) { return (K + 63) / 64; };
    double target = 0.0;
    if (rd && is_tc(kind)) {
        for (const Blk& b : blocks) {
            long long K = 0;
            for (int o = b.op0; o < b.op1; ++o) K += ops[o].k;
            target += (double)((b.m + tm_ - 1) / tm_) * ((b.n + tn_ - 1) / tn_) * stages(K);
        }
        target = std::max(2.0, target / 304.0);
    }
    for (const Blk& b : blocks) {
        long long K = 0;
        for (int o = b.op0; o < b.op1; ++o) K += ops[o].k;
        int S = 1;
        if (rd && is_tc(kind)) S = (int)std::max(1.0, std::min(32.0, std::ceil(stages(K) / target)));
        else if (rd) S = kchunks(b.m, b.n, K);
        const int step = (int)((K + S - 1) / S + 63) / 64 * 64;   // whole K-stages of either kernel
        for (int r0 = 0; r0 < b.m; r0 += tm_)
            for (int c0 = 0; c0 < b.n; c0 += tn_) {
                if (S == 1) {
                    out.push_back({b.C, nullptr, b.ldc, b.m, b.n, r0, c0, b.op0, b.op1, b.accumulate, b.cmap_rows,
                                   nullptr, 0, 1 << 30});
                    if (cm) cm->push_back(b.cmap_off);
                    continue;
                }
                int np = 0;
                for (long long k0 = 0; k0 < K; k0 += step, ++np) {
                    // the partial pointer holds an element offset until upload
                    out.push_back({b.C, nullptr, b.ldc, b.m, b.n, r0, c0, b.op0, b.op1, 0, b.cmap_rows,
                                   reinterpret_cast<double*>((pe + (size_t)np * tm_ * tn_) * sizeof(double) + 8),
                                   (int)k0, (int)std::min<long long>(K, k0 + step)});
                    if (cm) cm->push_back(-1);
                }
                rd->push_back({reinterpret_cast<const double*>(pe * sizeof(double) + 8), b.C, nullptr, np, tm_, tn_,
                               b.ldc, b.m, b.n, r0, c0, b.accumulate, b.cmap_rows});
                if (rcm) rcm->push_back(b.cmap_off);
                pe += (size_t)np * tm_ * tn_;
            }
    }
    if (part_elems) *part_elems = pe;
}

// Float64 units.  A block's K-list counts steps of four K per entry, rounded
// up; a 16 x 16 tile of a full block costs 4 DMMAs a step.  The work is cut so
// that 1216 units (eight a SM) of equal cost would cover it, but into no
// piece of fewer than eight steps (two per warp: 2.4 us on its
// sub-partition, about what a unit costs to start) nor a tile into more than
// 64 pieces.  The cut depends on the block list only, not on the tile, and so
// do the results.
void GemmPlan::units(int tile, std::vector<GemmBlk>& gb, std::vector<unsigned>& ub,
                     std::vector<long long>* cm, size_t* part_elems, size_t* ticks) const {
    const int nb = (int)blocks.size();
    std::vector<int> q(nb), cost(nb), ord(nb);
    double total = 0.0;
    for (int i = 0; i < nb; ++i) {
        const Blk& b = blocks[i];
        long long s = 0;
        for (int o = b.op0; o < b.op1; ++o) s += (ops[o].k + 3) / 4;
        require(s < (1LL << 30), "gemm K-list too long");
        q[i] = (int)s;
        total += (double)((b.m + 7) / 8) * ((b.n + 7) / 8) * s;
        ord[i] = i;
    }
    const double target = std::max(32.0, total / 1216.0);
    std::vector<int> qs(nb);
    for (int i = 0; i < nb; ++i) {
        const Blk& b = blocks[i];
        const double tc = (double)std::min(2, (b.m + 7) / 8) * std::min(2, (b.n + 7) / 8) * q[i];
        int S = (int)std::min(64.0, std::ceil(tc / target));
        S = std::max(1, std::min(S, q[i] / 8));
        qs[i] = std::max(1, (q[i] + S - 1) / S);
        cost[i] = (int)std::min(1e9, std::min(tile / 8, (b.m + 7) / 8) * (double)std::min(tile / 8, (b.n + 7) / 8) * qs[i]);
    }
    // costliest units first: the persistent CTAs take units in strides of the grid
    std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    gb.clear();
    ub.clear();
    if (cm) cm->clear();
    size_t pe = 0, tk = 0;
    for (int k = 0; k < nb; ++k) {
        const int i = ord[k];
        const Blk& b = blocks[i];
        const int mt = (b.m + tile - 1) / tile, nt = (b.n + tile - 1) / tile;
        const int S = std::max(1, (q[i] + qs[i] - 1) / qs[i]);
        gb.push_back({b.C, nullptr, pe, (int)tk, b.ldc, b.m, b.n, b.op0, b.op1, b.accumulate, b.cmap_rows, q[i], qs[i], S,
                      nt, (int)ub.size()});
        if (cm) cm->push_back(b.cmap_off);
        const size_t tiles = (size_t)mt * nt;
        if (S > 1) {
            pe += tiles * S * tile * tile;
            tk += tiles;
        }
        require(ub.size() + tiles * S < (1ULL << 31) && tk < (1ULL << 31), "gemm unit list too long");
        ub.insert(ub.end(), tiles * S, (unsigned)k);
    }
    *part_elems = pe;
    *ticks = tk;
}

// 32 x 32 units when there are enough of them to keep every SM busy for two
// rounds of its eight (fewer unit starts, half the operand traffic), the
// narrow 16 x 16 ones below that.  Both give the same bits and nearly the same
// time near the line (the float64 pipe bounds both); in the M = 256 sweep the
// tuner takes 32 x 32 for a third of the launches.
int GemmPlan::tile_rule() const {
    size_t n = 0;
    for (const auto& b : blocks) n += (size_t)((b.m + 31) / 32) * ((b.n + 31) / 32);
    return n >= 2432 ? 32 : 16;
}

void GemmPlan::workspace(size_t part_elems, size_t ticks, cudaStream_t st) {
    if (part_elems) dpart.ensure(part_elems * sizeof(double) + 16, st);
    if (ticks) {
        const size_t had = dtick.bytes();
        dtick.ensure(ticks * sizeof(unsigned), st);
        if (dtick.bytes() != had) MPSPT_CUDA(cudaMemsetAsync(dtick.get(), 0, dtick.bytes(), st));
    }
}

namespace {
// longest K-list first: the persistent kernels hand out tasks in strides of
// the grid, so this order balances the CTAs (each output tile has exactly
// one task, so the order does not change any result)
void order_tasks(std::vector<GemmTask>& tasks, std::vector<long long>* cm, const std::vector<GemmOp>& ops) {
    std::vector<long long> cost(tasks.size());
    for (size_t i = 0; i < tasks.size(); ++i) {
        long long k = 0;
        for (int o = tasks[i].op0; o < tasks[i].op1; ++o) k += ops[o].k;
        cost[i] = k;
    }
    std::vector<size_t> ord(tasks.size());
    for (size_t i = 0; i < ord.size(); ++i) ord[i] = i;
    std::stable_sort(ord.begin(), ord.end(), [&](size_t a, size_t b) { return cost[a] > cost[b]; });
    std::vector<GemmTask> t2(tasks.size());
    std::vector<long long> c2(cm ? tasks.size() : 0);
    for (size_t i = 0; i < ord.size(); ++i) {
        t2[i] = tasks[ord[i]];
        if (cm) c2[i] = (*cm)[ord[i]];
    }
    tasks.swap(t2);
    if (cm) cm->swap(c2);
}

int bucket(long long x) {
    int b = 0;
    while (x > 1) { x >>= 1; ++b; }
    return b;
}
}  // namespace

void GemmPlan::upload(cudaStream_t st) {
    mpspt::upload(dops, ops, st);
    steps = 0.0;
    if (kind == GEMM_F64)
        for (const Blk& b : blocks) {
            long long q = 0;
            for (int o = b.op0; o < b.op1; ++o) q += (ops[o].k + 3) / 4;
            steps += (double)((b.m + 7) / 8) * ((b.n + 7) / 8) * q;
        }
    // (float64 plans of few steps take the narrow units: the two differ by the
    // launch alone there, and their timing would stand for larger plans)
    const bool few = kind == GEMM_F64 && steps <= kClusterSteps;
    const bool tune = tuner && !is_tc(kind) && !blocks.empty() && !few;
    if (tune) {
        const std::pair<int, int> t = tuner->choose(*this, st);
        tm = t.first;
        tn = t.second;
    }
    if (!cmaps.empty()) mpspt::upload(dcmaps, cmaps, st);
    const int* cbase = dcmaps.as<int>();
    size_t pe = 0;
    if (kind == GEMM_F64) {
        size_t tk = 0;
        std::vector<long long> cm;
        tile64 = few ? 16 : tune ? (tm == 32 ? 32 : 16) : tile_rule();
        units(tile64, gblk, unit_blk, &cm, &pe, &tk);
        for (size_t i = 0; i < gblk.size(); ++i) gblk[i].cmap = cm[i] >= 0 ? cbase + cm[i] : nullptr;
        workspace(pe, tk, st);
        mpspt::upload(dgblk, gblk, st);
        mpspt::upload(dunit, unit_blk, st);
    } else {
        split(tm, tn, tasks, &task_cmap, &reds, &red_cmap, &pe);
        if (pe) dpart.ensure(pe * sizeof(double) + 16, st);
        double* pbase = dpart.as<double>();
        for (auto& t : tasks)   // partial offsets (stored as byte offsets + 8) become pointers
            if (t.part) t.part = pbase + ((reinterpret_cast<uintptr_t>(t.part) - 8) / sizeof(double));
        for (auto& r : reds) r.part = pbase + ((reinterpret_cast<uintptr_t>(r.part) - 8) / sizeof(double));
        order_tasks(tasks, &task_cmap, ops);
        for (size_t i = 0; i < tasks.size(); ++i)
            tasks[i].cmap = task_cmap[i] >= 0 ? cbase + task_cmap[i] : nullptr;
        for (size_t i = 0; i < reds.size(); ++i) reds[i].cmap = red_cmap[i] >= 0 ? cbase + red_cmap[i] : nullptr;
        if (!reds.empty()) mpspt::upload(dreds, reds, st);
        mpspt::upload(dtasks, tasks, st);
    }
    if (checks_enabled()) {
        RangeCheck check_range;
        // per planned block (all tiles of a block share its output and its
        // K-list): the output range, or the span of its mapped addresses,
        // and every operand range of its K-list
        for (const Blk& b : blocks) {
            if (b.cmap_off < 0) {
                check_range(b.C, ((size_t)(b.m - 1) * b.ldc + b.n) * sizeof(double), "gemm C");
                if (b.ldc < b.n) throw Error(MPSPT_ERR_INVALID, "gemm ldc");
            } else {
                const long long o = b.cmap_off;
                const int nmap = b.cmap_rows ? b.m : b.n, other = b.cmap_rows ? b.n : b.m;
                require((size_t)(o + 2 * (long long)nmap) <= cmaps.size(), "gemm cmap range");
                long long lo = 0, hi = 0;
                for (int q = 0; q < nmap; ++q) {
                    const long long base = cmaps[o + 2 * q], ld = cmaps[o + 2 * q + 1];
                    require(base >= 0 && ld >= 0, "gemm cmap entry");
                    const long long last = base + (long long)(other - 1) * ld;
                    lo = q ? std::min(lo, base) : base;
                    hi = q ? std::max(hi, last) : last;
                }
                check_range(b.C + lo, (size_t)(hi - lo + 1) * sizeof(double), "gemm cmap dst");
            }
            for (int q = b.op0; q < b.op1; ++q) {
                const GemmOp& op = ops[q];
                const size_t ea = (op.trans & 1) ? (size_t)(op.k - 1) * op.lda + b.m : (size_t)(b.m - 1) * op.lda + op.k;
                const size_t eb = (op.trans & 2) ? (size_t)(b.n - 1) * op.ldb + op.k : (size_t)(op.k - 1) * op.ldb + b.n;
                check_range(op.A, ea * sizeof(double), "gemm A");
                check_range(op.B, eb * sizeof(double), "gemm B");
                if ((op.trans & 1) ? op.lda < b.m : op.lda < op.k) throw Error(MPSPT_ERR_INVALID, "gemm lda");
                if ((op.trans & 2) ? op.ldb < op.k : op.ldb < b.n) throw Error(MPSPT_ERR_INVALID, "gemm ldb");
            }
        }
    }
}

void Autotuner::RawBuf::ensure(size_t bytes) {
    if (bytes <= n) return;
    const size_t want = std::max(bytes, 2 * n);
    if (p) old.push_back(p);
    p = nullptr;
    n = 0;
    MPSPT_CUDA(cudaMalloc(&p, want));
    Registry::get().add(p, want);
    n = want;
}

Autotuner::RawBuf::~RawBuf() {
    old.push_back(p);
    for (void* q : old)
        if (q) {
            Registry::get().remove(q);
            cudaFree(q);
        }
}

Autotuner::~Autotuner() {
    for (auto& e : ev)
        if (e) cudaEventDestroy(e);
}

std::pair<int, int> Autotuner::choose(const GemmPlan& g, cudaStream_t st) {
    std::vector<long long> ms, ns, ks;
    size_t cmax = 1;
    for (const auto& b : g.blocks) {
        long long k = 0;
        for (int o = b.op0; o < b.op1; ++o) k += g.ops[o].k;
        ms.push_back(b.m);
        ns.push_back(b.n);
        ks.push_back(k);
        cmax = std::max(cmax, (size_t)b.m * b.n);
    }
    auto med = [](std::vector<long long>& v) {
        std::nth_element(v.begin(), v.begin() + v.size() / 2, v.end());
        return v[v.size() / 2];
    };
    const Key key{g.kind, g.skinny ? 1 : 0, bucket(med(ms)), bucket(med(ns)), bucket(med(ks)),
                  bucket((long long)g.blocks.size())};
    std::lock_guard<std::mutex> lk(mu);
    auto it = best.find(key);
    // (a float64 entry of another tile than its two, from an older file, is timed again)
    const std::pair<int, int> wide{32, 32}, narrow{16, 128};
    if (it != best.end() && (g.kind != GEMM_F64 || it->second == wide || it->second == narrow)) {
        ++reused;
        return it->second;
    }
    static const int cand_wide[][2] = {{64, 64}, {32, 64}, {64, 32}, {32, 32}};
    static const int cand_skinny[][2] = {{16, 128}, {32, 64}, {32, 32}};
    static const int cand_f64[][2] = {{32, 32}, {16, 128}};
    const bool f64 = g.kind == GEMM_F64;
    const int (*cand)[2] = f64 ? cand_f64 : g.skinny ? cand_skinny : cand_wide;
    const int nc = f64 ? 2 : g.skinny ? 3 : 4;
    if (!ev[0]) {
        MPSPT_CUDA(cudaEventCreate(&ev[0]));
        MPSPT_CUDA(cudaEventCreate(&ev[1]));
    }
    scratch.ensure(cmax * sizeof(double) + 16);
    std::pair<int, int> win{cand[0][0], cand[0][1]};
    float tbest = 1e30f;
    std::vector<GemmTask> tt;
    std::vector<GemmBlk> gb;
    std::vector<unsigned> ub;
    for (int c = 0; c < nc; ++c) {
        // outputs go to scratch: dense m x n, no map; operands are the plan's
        size_t pe = 0, tk = 0;
        if (f64) {
            g.units(cand[c][0] == 32 ? 32 : 16, gb, ub, nullptr, &pe, &tk);
            for (auto& b : gb) {
                b.C = static_cast<double*>(scratch.p);
                b.ldc = b.n;
                b.accumulate = b.cmap_rows = 0;
            }
            dpart.ensure(pe * sizeof(double) + 16);
            dtick.ensure(tk * sizeof(unsigned) + 16);
            MPSPT_CUDA(cudaMemsetAsync(dtick.p, 0, tk * sizeof(unsigned) + 16, st));
            dtasks.ensure(gb.size() * sizeof(GemmBlk) + 16);
            dunits.ensure(ub.size() * sizeof(unsigned) + 16);
            if (!ub.empty()) {
                copy_h2d(dtasks.p, gb.data(), gb.size() * sizeof(GemmBlk), st);
                copy_h2d(dunits.p, ub.data(), ub.size() * sizeof(unsigned), st);
            }
        } else {
            g.split(cand[c][0], cand[c][1], tt, nullptr);
            order_tasks(tt, nullptr, g.ops);
            for (auto& t : tt) {
                t.C = static_cast<double*>(scratch.p);
                t.ldc = t.n;
                t.cmap = nullptr;
                t.cmap_rows = 0;
            }
            dtasks.ensure(tt.size() * sizeof(GemmTask) + 16);
            if (!tt.empty()) copy_h2d(dtasks.p, tt.data(), tt.size() * sizeof(GemmTask), st);
        }
        auto run = [&] {
            if (f64)
                launch_dgemm(cand[c][0] == 32 ? 32 : 16, static_cast<const GemmBlk*>(dtasks.p),
                             static_cast<const unsigned*>(dunits.p), (int)ub.size(), g.dops.as<GemmOp>(),
                             static_cast<double*>(dpart.p), static_cast<unsigned*>(dtick.p), st);
            else
                launch_gemm_tile(cand[c][0], cand[c][1], static_cast<const GemmTask*>(dtasks.p), (int)tt.size(),
                                 g.dops.as<GemmOp>(), st);
        };
        run();
        MPSPT_CUDA(cudaEventRecord(ev[0], st));
        for (int r = 0; r < 3; ++r) run();
        MPSPT_CUDA(cudaEventRecord(ev[1], st));
        MPSPT_CUDA(cudaEventSynchronize(ev[1]));
        float ms_ = 0.f;
        MPSPT_CUDA(cudaEventElapsedTime(&ms_, ev[0], ev[1]));
        if (ms_ < tbest) { tbest = ms_; win = {cand[c][0], cand[c][1]}; }
    }
    ++timed;
    best[key] = win;
    return win;
}

void Autotuner::load(const std::string& path) {
    FILE* f = std::fopen(path.c_str(), "r");
    if (!f) return;
    int a[8];
    std::lock_guard<std::mutex> lk(mu);
    while (std::fscanf(f, "%d %d %d %d %d %d %d %d", &a[0], &a[1], &a[2], &a[3], &a[4], &a[5], &a[6], &a[7]) == 8)
        if (gemm_tile_supported(a[6], a[7])) best[Key{a[0], a[1], a[2], a[3], a[4], a[5]}] = {a[6], a[7]};
    std::fclose(f);
}

void Autotuner::save(const std::string& path) {
    FILE* f = std::fopen(path.c_str(), "w");
    if (!f) return;
    std::lock_guard<std::mutex> lk(mu);
    for (const auto& kv : best) {
        const Key& k = kv.first;
        std::fprintf(f, "%d %d %d %d %d %d %d %d\n", std::get<0>(k), std::get<1>(k), std::get<2>(k), std::get<3>(k),
                     std::get<4>(k), std::get<5>(k), kv.second.first, kv.second.second);
    }
    std::fclose(f);
}

void GemmPlan::run(cudaStream_t st) const {
    if (kind == GEMM_F64) {
        launch_dgemm(tile64, dgblk.as<GemmBlk>(), dunit.as<unsigned>(), (int)unit_blk.size(), dops.as<GemmOp>(),
                     dpart.as<double>(), dtick.as<unsigned>(), st, skip);
        return;
    }
    const int nt = (int)tasks.size();
    if (nt == 0) return;
    const GemmTask* t = dtasks.as<GemmTask>();
    const GemmOp* o = dops.as<GemmOp>();
    if (is_tc(kind)) launch_gemm_tc(t, nt, o, err, st, skip, kind == GEMM_TC16);
    else launch_gemm_tile(tm, tn, t, nt, o, st, skip);
    if (!reds.empty()) launch_splitk_reduce(dreds.as<SplitRed>(), (int)reds.size(), st, skip);
}

// Omega_ac of bond (i, i+1): the products of the two sites' elements, added in
// the order of the entries.  One dense accumulator per source state a over
// (out, c, in) with a bitmap of the touched places: no ordered container.
void Omega::build(const MPO& W, int i) {
    Da = W.dim[i];
    const int Dc = W.dim[i + 2];
    struct N2 { int s, t; double v; };
    std::vector<N2> nz;                    // non-zero elements of the second site's entries
    std::vector<int> nzp;
    for (const auto& e2 : W.W[i + 1]) {
        nzp.push_back((int)nz.size());
        const Mat4& o = W.ops[e2.op];
        for (int s = 0; s < 4; ++s)
            for (int t = 0; t < 4; ++t)
                if (o[s * 4 + t] != 0.0) nz.push_back({s, t, o[s * 4 + t]});
    }
    nzp.push_back((int)nz.size());
    const size_t places = (size_t)16 * Dc * 16;   // (out * Dc + c) * 16 + in
    std::vector<double> acc(places, 0.0);
    std::vector<uint64_t> bits((places + 63) / 64, 0);
    e.clear();
    first.assign((size_t)Da * 16 + 1, 0);
    const auto& p1 = W.out_ptr[i];
    const auto& p2 = W.out_ptr[i + 1];
    for (int a = 0; a < Da; ++a) {
        for (int q1 = p1[a]; q1 < p1[a + 1]; ++q1) {
            const MpoEntry& e1 = W.W[i][q1];
            const Mat4& o1 = W.ops[e1.op];
            for (int q2 = p2[e1.b]; q2 < p2[e1.b + 1]; ++q2) {
                const MpoEntry& e2 = W.W[i + 1][q2];
                const double cc = e1.coef * e2.coef;
                for (int s1 = 0; s1 < 4; ++s1)
                    for (int t1 = 0; t1 < 4; ++t1) {
                        const double v1 = o1[s1 * 4 + t1];
                        if (v1 == 0.0) continue;
                        for (int k = nzp[q2]; k < nzp[q2 + 1]; ++k) {
                            const size_t at = ((size_t)(s1 * 4 + nz[k].s) * Dc + e2.b) * 16 + t1 * 4 + nz[k].t;
                            acc[at] += cc * v1 * nz[k].v;
                            bits[at >> 6] |= 1ULL << (at & 63);
                        }
                    }
            }
        }
        int out = 0;
        for (size_t w = 0; w < bits.size(); ++w) {
            for (uint64_t m = bits[w]; m; m &= m - 1) {
                const size_t at = w * 64 + (size_t)__builtin_ctzll(m);
                const int o16 = (int)(at / ((size_t)Dc * 16));
                for (; out <= o16; ++out) first[(size_t)a * 16 + out] = (int)e.size();
                if (acc[at] != 0.0) e.push_back({a, (int)(at / 16 % Dc), o16, (int)(at % 16), acc[at]});
                acc[at] = 0.0;
            }
            bits[w] = 0;
        }
        for (; out < 16; ++out) first[(size_t)a * 16 + out] = (int)e.size();
    }
    first[(size_t)Da * 16] = (int)e.size();
}

void mix_pieces(std::vector<MixTask>& tasks, std::vector<unsigned>& piece_task) {
    int np = 0;
    for (MixTask& t : tasks) {
        t.p0 = np;
        np += (t.rows * t.cols + MIX_PIECE - 1) / MIX_PIECE;
    }
    piece_task.resize(np);
    for (size_t i = 0; i < tasks.size(); ++i)
        std::fill(piece_task.begin() + tasks[i].p0,
                  i + 1 < tasks.size() ? piece_task.begin() + tasks[i + 1].p0 : piece_task.end(), (unsigned)i);
}

void TwoSitePlan::build(const Omega& om, const TwoT& bra, const TwoT& ket, const Bond& braL,
                        const Bond& ketL, const Bond& braR, const Bond& ketR, const EnvT& L,
                        const EnvT& R, const double* x, double* out, cudaStream_t st) {
    g1.clear(); g2.clear(); g2s.clear();
    mtasks.clear(); msrc.clear();
    const int np = (int)ket.panels.size();
    const int nc = R.na;
    const int na = om.Da;
    // ---- Rpack per ket right sector: blocks R_c(sb_c, sk) stacked by c
    std::vector<long long> rp_off(ketR.nsec(), -1);
    std::vector<int> rp_rows(ketR.nsec(), 0);
    std::vector<int> rcol((size_t)nc * ketR.nsec(), -1);   // row offset of c inside Rpack(sk), sk by sk
    std::vector<int> rsb((size_t)nc * ketR.nsec(), -1);    // its bra sector
    size_t rps = 0;
    std::vector<CopyTask> pk_tasks;
    for (const auto& P : ket.panels) {
        const int sk = P.sr;
        int rows = 0;
        for (int c = 0; c < nc; ++c) {
            int rb = R.find(c, sk);
            if (rb < 0) continue;
            rcol[(size_t)sk * nc + c] = rows;
            rsb[(size_t)sk * nc + c] = R.blk[rb].sb;
            rows += braR.sec[R.blk[rb].sb].dim;
        }
        rp_rows[sk] = rows;
        rp_off[sk] = (long long)rps;
        rps += (size_t)rows * ketR.sec[sk].dim;
    }
    // ---- Lpack per bra left sector: blocks L_a(sl, sk_a) side by side
    std::vector<int> lp_cols(braL.nsec(), 0);
    std::vector<long long> lp_off(braL.nsec(), -1);
    std::vector<int> lcol((size_t)na * braL.nsec(), -1);
    std::vector<int> l_blk((size_t)na * braL.nsec(), -1);
    for (int b = 0; b < (int)L.blk.size(); ++b) l_blk[(size_t)L.blk[b].a * braL.nsec() + L.blk[b].sb] = b;
    size_t lps = 0;
    for (int sl = 0; sl < braL.nsec(); ++sl) {
        int cols = 0;
        for (int a = 0; a < na; ++a) {
            int lb = l_blk[(size_t)a * braL.nsec() + sl];
            if (lb < 0) continue;
            lcol[(size_t)a * braL.nsec() + sl] = cols;
            cols += ketL.sec[L.blk[lb].sk].dim;
        }
        lp_cols[sl] = cols;
        lp_off[sl] = (long long)lps;
        lps += (size_t)braL.sec[sl].dim * cols;
    }
    Rp.ensure((rps + 1) * sizeof(double), st);
    Lp.ensure((lps + 1) * sizeof(double), st);
    double* Rpp = Rp.as<double>();
    double* Lpp = Lp.as<double>();
    for (const auto& P : ket.panels) {
        const int sk = P.sr, dk = ketR.sec[sk].dim;
        for (int c = 0; c < nc; ++c) {
            int rb = R.find(c, sk);
            if (rb < 0) continue;
            const int db = braR.sec[R.blk[rb].sb].dim;
            pk_tasks.push_back({R.ptr(R.blk[rb]), Rpp + rp_off[sk] + (size_t)rcol[(size_t)sk * nc + c] * dk,
                                nullptr, db, dk, dk, dk, 0, 0});
        }
    }
    for (int sl = 0; sl < braL.nsec(); ++sl)
        for (int a = 0; a < na; ++a) {
            int lb = l_blk[(size_t)a * braL.nsec() + sl];
            if (lb < 0) continue;
            const int dl = braL.sec[sl].dim, dk = ketL.sec[L.blk[lb].sk].dim;
            pk_tasks.push_back({L.ptr(L.blk[lb]), Lpp + lp_off[sl] + lcol[(size_t)a * braL.nsec() + sl],
                                nullptr, dl, dk, dk, lp_cols[sl], 0, 0});
        }
    if (checks_enabled()) {
        RangeCheck check;
        for (const auto& t : pk_tasks) {
            check(t.src, ((size_t)(t.rows - 1) * t.lds + t.cols_n) * sizeof(double), "pack src");
            check(t.dst, ((size_t)(t.rows - 1) * t.ldd + t.cols_n) * sizeof(double), "pack dst");
        }
    }
    mpspt::upload(pk, pk_tasks, st);
    launch_copy(pk.as<CopyTask>(), (int)pk_tasks.size(), st);
    // ---- T panels
    std::vector<long long> toff(np, -1);
    std::vector<int> panel_of(ket.blk.size());
    tsize = 0;
    for (int p = 0; p < np; ++p) {
        const auto& P = ket.panels[p];
        for (int b = P.b0; b < P.b1; ++b) panel_of[b] = p;
        if (rp_rows[P.sr] == 0) continue;
        toff[p] = (long long)tsize;
        tsize += (size_t)P.rows * rp_rows[P.sr];
    }
    T.ensure((tsize + 1) * sizeof(double), st);
    double* Tp = T.as<double>();
    for (int p = 0; p < np; ++p) {
        if (toff[p] < 0) continue;
        const auto& P = ket.panels[p];
        const int dk = ketR.sec[P.sr].dim, nr = rp_rows[P.sr];
        int m0 = g1.mark();
        g1.op(x + P.off, dk, Rpp + rp_off[P.sr], dk, dk, 2, 1.0);
        g1.block(Tp + toff[p], nr, P.rows, nr, 0, m0);
    }
    // ---- bra left panels, V stacks and mix tasks
    std::vector<std::vector<int>> left_blocks(braL.nsec());
    for (int b = 0; b < (int)bra.blk.size(); ++b) left_blocks[bra.blk[b].sl].push_back(b);
    std::vector<long long> voff(braL.nsec(), -1);
    std::vector<int> wd(braL.nsec(), 0);
    size_t vs = 0;
    for (int sl = 0; sl < braL.nsec(); ++sl) {
        int w = 0;
        for (int b : left_blocks[sl]) w += bra.blk[b].cols;
        wd[sl] = w;
        if (w == 0 || lp_cols[sl] == 0) continue;
        voff[sl] = (long long)vs;
        vs += (size_t)lp_cols[sl] * w;
    }
    V.ensure((vs + 1) * sizeof(double), st);
    double* Vp = V.as<double>();
    // ket blocks by (left sector, in): where their T rows start
    struct KetT { int sr, nr; size_t base; };
    std::vector<KetT> kt((size_t)ketL.nsec() * 16, KetT{-1, 0, 0});
    for (int sk = 0; sk < ketL.nsec(); ++sk)
        for (int in = 0; in < 16; ++in) {
            const int kb = ket.find(sk, in / 4, in % 4);
            if (kb < 0 || toff[panel_of[kb]] < 0) continue;
            const auto& K = ket.blk[kb];
            const int p = panel_of[kb], sr = ket.panels[p].sr;
            const size_t rip = (K.off - ket.panels[p].off) / (size_t)K.cols;
            kt[(size_t)sk * 16 + in] = {sr, rp_rows[sr], (size_t)toff[p] + rip * rp_rows[sr]};
        }
    for (int sl = 0; sl < braL.nsec(); ++sl) {
        if (voff[sl] < 0) continue;
        const int W = wd[sl];
        // column map of the bra left panel -> two-site layout
        std::vector<int> cm;
        int wcol = 0;
        for (int bi : left_blocks[sl]) {
            const auto& B = bra.blk[bi];
            for (int r = 0; r < B.cols; ++r) { cm.push_back((int)(B.off + r)); cm.push_back(B.cols); }
            for (int a = 0; a < na; ++a) {
                const int lc = lcol[(size_t)a * braL.nsec() + sl];
                if (lc < 0) continue;
                const int lb = l_blk[(size_t)a * braL.nsec() + sl];
                const int sk = L.blk[lb].sk, dk = ketL.sec[sk].dim;
                MixTask mt{Vp + voff[sl] + (size_t)lc * W + wcol, dk, B.cols, W, (int)msrc.size(), 0, 0};
                const int o16 = B.s1 * 4 + B.s2;
                for (int q = om.begin(a, o16); q < om.end(a, o16); ++q) {
                    const Omega::E& E = om.e[q];
                    const KetT& k = kt[(size_t)sk * 16 + E.in];
                    if (k.sr < 0) continue;
                    const size_t rq = (size_t)k.sr * nc + E.c;
                    if (rcol[rq] < 0 || rsb[rq] != B.sr) continue;
                    const size_t src = k.base + rcol[rq];
                    if (src + (size_t)(dk - 1) * k.nr + B.cols > tsize) throw Error(MPSPT_ERR_INVALID, "mix source outside T");
                    msrc.push_back({Tp + src, k.nr, 0, E.v});
                }
                mt.s1 = (int)msrc.size();
                mtasks.push_back(mt);
            }
            wcol += B.cols;
        }
        // g2: out(sl, :) = Lpack(sl) V_stack(sl); TC computes the transpose (rows = panel cols)
        const int dl = braL.sec[sl].dim, K = lp_cols[sl];
        if (is_tc(kind)) {
            const long long co = g2.add_cmap(cm);
            int m0 = g2.mark();
            g2.op(Vp + voff[sl], W, Lpp + lp_off[sl], K, K, 1 | 2, 1.0);
            g2.block(out, 0, W, dl, 0, m0, co, 1);
        } else {
            GemmPlan& g = (kind == GEMM_F32 && dl <= 16) ? g2s : g2;
            const long long co = g.add_cmap(cm);
            int m0 = g.mark();
            g.op(Lpp + lp_off[sl], K, Vp + voff[sl], W, K, 0, 1.0);
            g.block(out, 0, dl, W, 0, m0, co, 0);
        }
    }
    // bra blocks whose left panel has no operator: zero them through the mix path
    for (int sl = 0; sl < braL.nsec(); ++sl) {
        if (voff[sl] >= 0) continue;
        for (int bi : left_blocks[sl]) {
            const auto& B = bra.blk[bi];
            mtasks.push_back({out + B.off, B.rows, B.cols, B.cols, (int)msrc.size(), (int)msrc.size(), 0});
        }
    }
    if (checks_enabled()) {
        RangeCheck check;   // (the sources were placed inside T above)
        check(Tp, tsize * sizeof(double), "mix T");
        for (const auto& t : mtasks) check(t.dst, ((size_t)(t.rows - 1) * t.ldd + t.cols) * sizeof(double), "mix dst");
    }
    // Pieces cost the host their list and its copy, so they are made for the
    // low-precision operator alone, which runs tens of times per list and has
    // the large bonds: M = 256 35.3 -> 29.3 ms of block sums a sweep (26.0
    // with every plan in pieces).  A float64 sweep at M = 64 gained 0.2 ms on
    // the device and lost 4.4 ms a pass.
    mpieces.clear();
    if (is_tc(kind)) mix_pieces(mtasks, mpieces);
    mpspt::upload(dmt, mtasks, st);
    if (!mpieces.empty()) mpspt::upload(dmp, mpieces, st);
    mpspt::upload(dms, msrc, st);
    g1.upload(st);
    g2.upload(st);
    g2s.upload(st);
}

void DiagPlan::build(const Omega& om, const TwoT& x, const Bond& Lb, const Bond& Rb,
                     const EnvT& Le, const EnvT& Re, const std::vector<QN>& dqL,
                     const std::vector<QN>& dqR, double* out, cudaStream_t st) {
    (void)Lb; (void)Rb;
    tasks.clear();
    terms.clear();
    for (const auto& b : x.blk) {
        const int o16 = b.s1 * 4 + b.s2;
        int t0 = (int)terms.size();
        for (int a = 0; a < om.Da; ++a) {
            if (!(dqL[a] == QN(0, 0))) continue;
            const int lb = Le.find(a, b.sl);
            if (lb < 0) continue;
            for (int q = om.begin(a, o16); q < om.end(a, o16); ++q) {
                const Omega::E& E = om.e[q];
                if (E.in != o16 || !(dqR[E.c] == QN(0, 0))) continue;
                const int rb = Re.find(E.c, b.sr);
                if (rb < 0) continue;
                terms.push_back({Le.ptr(Le.blk[lb]), Re.ptr(Re.blk[rb]), b.rows, b.cols, E.v});
            }
        }
        tasks.push_back({out + b.off, b.rows, b.cols, t0, (int)terms.size()});
    }
    if (checks_enabled()) {
        RangeCheck check_range;
        for (const auto& t : tasks) {
            check_range(t.out, (size_t)t.rows * t.cols * sizeof(double), "diag out");
            for (int k = t.t0; k < t.t1; ++k) {
                check_range(terms[k].L, ((size_t)(t.rows - 1) * (terms[k].ldL + 1) + 1) * sizeof(double), "diag L");
                check_range(terms[k].R, ((size_t)(t.cols - 1) * (terms[k].ldR + 1) + 1) * sizeof(double), "diag R");
            }
        }
    }
    upload(dt, tasks, st);
    upload(dterm, terms, st);
}

void DiagPlan::run(cudaStream_t st) const {
    launch_diag(dt.as<DiagTask>(), (int)tasks.size(), dterm.as<DiagTerm>(), st);
}

void plan_product(GemmPlan& g, const TwoT& x, double* xd, const Bond& mid, const SiteT& A,
                  const SiteT& B, const Bond& L) {
    for (const auto& b : x.blk) {
        int m0 = g.mark();
        int sm = mid.find(L.sec[b.sl].q + site_qn(b.s1));
        if (sm >= 0) {
            int ia = A.find(b.sl, b.s1), ib = B.find(sm, b.s2);
            if (ia >= 0 && ib >= 0 && B.blk[ib].sr == b.sr) {
                int k = mid.sec[sm].dim;
                g.op(A.ptr(A.blk[ia]), k, B.ptr(B.blk[ib]), b.cols, k, 0, 1.0);
            }
        }
        g.block(xd + b.off, b.cols, b.rows, b.cols, 0, m0);
    }
}

// (The sources were placed inside their buffer by the builders.)
void EnvPlan::upload_mix(cudaStream_t st) {
    if (checks_enabled()) {
        RangeCheck check;
        for (const auto& t : mt) check(t.dst, ((size_t)(t.rows - 1) * t.ldd + t.cols) * sizeof(double), "env mix dst");
    }
    mpspt::upload(dmt, mt, st);
    mpspt::upload(dms, ms, st);
    g1.upload(st);
    g2.upload(st);
}

// L_new[b](sb', sk') = sum_{s,t} A_bra(sl_b, s)^T [sum_a W_ab(s,t) L_a(sl_b, sl_k)] A_ket(sl_k, t)
void EnvPlan::build_left(const MPO& W, int site, const EnvT& L, const SiteT& Abra, const SiteT& Aket,
                         const Bond& braL, const Bond& ketL, const Bond& braR, const Bond& ketR,
                         EnvT& Lnew, cudaStream_t st) {
    g1.clear();
    g2.clear();
    mt.clear();
    ms.clear();
    const int nkb = (int)Aket.blk.size();
    // g1: Y_kb = L_panel(sl_k) A_ket(kb), (panel rows) x dim(sr_k)
    std::vector<long long> yoff(nkb, -1);
    size_t ys = 0;
    for (int kb = 0; kb < nkb; ++kb) {
        const auto& K = Aket.blk[kb];
        if (L.prows[K.sl] == 0) continue;
        yoff[kb] = (long long)ys;
        ys += (size_t)L.prows[K.sl] * ketR.sec[K.sr].dim;
    }
    Y.ensure((ys + 1) * sizeof(double), st);
    double* Yp = Y.as<double>();
    for (int kb = 0; kb < nkb; ++kb) {
        if (yoff[kb] < 0) continue;
        const auto& K = Aket.blk[kb];
        const int kd = ketL.sec[K.sl].dim, nd = ketR.sec[K.sr].dim, P = L.prows[K.sl];
        const int m0 = g1.mark();
        g1.op(L.panel(K.sl), kd, Aket.ptr(K), nd, kd, 0, 1.0);
        g1.block(Yp + yoff[kb], nd, P, nd, 0, m0);
    }
    // mix: Z_(out, s) over the elements (a, s, t -> b)
    const std::vector<MPO::El>& el = W.in_el[site];
    const std::vector<int>& at = W.in_at[site];
    struct ZB { int nb, s, bb; size_t off; int rows, cols; };
    std::vector<ZB> zb;
    size_t zs = 0;
    check_range(Yp, ys * sizeof(double), "env mix Y");
    // left sector and block of every (right sector, local state)
    struct Side { int sl, blk; };
    auto side = [](const Bond& br, const SiteT& A) {
        std::vector<Side> v((size_t)br.nsec() * 4, Side{-1, -1});
        for (int b = 0; b < (int)A.blk.size(); ++b) v[(size_t)A.blk[b].sr * 4 + A.blk[b].s] = {A.blk[b].sl, b};
        return v;
    };
    const std::vector<Side> bside = side(braR, Abra), kside = side(ketR, Aket);
    for (int nbi = 0; nbi < (int)Lnew.blk.size(); ++nbi) {
        const auto& nb = Lnew.blk[nbi];
        const int nd = ketR.sec[nb.sk].dim;
        // ket-side lookups depend on t only
        const int* blk_t[4];
        double* y_t[4];
        for (int t = 0; t < 4; ++t) {
            const Side k = kside[(size_t)nb.sk * 4 + t];
            const bool ok = k.blk >= 0 && yoff[k.blk] >= 0;
            blk_t[t] = ok ? L.row(k.sl) : nullptr;
            y_t[t] = ok ? Yp + yoff[k.blk] : nullptr;
        }
        for (int s = 0; s < 4; ++s) {
            const Side side_b = bside[(size_t)nb.sb * 4 + s];
            if (side_b.blk < 0) continue;
            const int slb = side_b.sl, bb = side_b.blk;
            const int rows = braL.sec[slb].dim;
            const int s0 = (int)ms.size();
            for (int q = at[(size_t)nb.a * 4 + s]; q < at[(size_t)nb.a * 4 + s + 1]; ++q) {
                const MPO::El& E = el[q];
                if (!blk_t[E.t]) continue;
                const int lb = blk_t[E.t][E.x];
                if (lb < 0 || L.blk[lb].sb != slb) continue;
                double* src = y_t[E.t] + (size_t)L.blk[lb].roff * nd;
                if (src + (size_t)rows * nd > Yp + ys) throw Error(MPSPT_ERR_INVALID, "env mix source outside Y");
                ms.push_back({src, nd, 0, E.v});
            }
            if ((int)ms.size() == s0) continue;
            zb.push_back({nbi, s, bb, zs, rows, nd});
            mt.push_back({nullptr, rows, nd, nd, s0, (int)ms.size(), 0});
            zs += (size_t)rows * nd;
        }
    }
    Z.ensure((zs + 1) * sizeof(double), st);
    double* Zp = Z.as<double>();
    for (size_t q = 0; q < zb.size(); ++q) mt[q].dst = Zp + zb[q].off;
    // g2: L_new(out) = sum_s A_bra(sl_b, s)^T Z_(out, s)
    size_t z = 0;
    for (int nbi = 0; nbi < (int)Lnew.blk.size(); ++nbi) {
        const auto& nb = Lnew.blk[nbi];
        const int md = braR.sec[nb.sb].dim, nd = ketR.sec[nb.sk].dim;
        const int m0 = g2.mark();
        for (; z < zb.size() && zb[z].nb == nbi; ++z)
            g2.op(Abra.ptr(Abra.blk[zb[z].bb]), md, Zp + zb[z].off, nd, zb[z].rows, 1, 1.0);
        g2.block(Lnew.ptr(nb), nd, md, nd, 0, m0);
    }
    upload_mix(st);
}

void EnvPlan::build_left_run(const RunMap& T, const EnvT& L, const Bond& bra, const Bond& ket, EnvT& Lnew,
                             cudaStream_t st) {
    g1.clear();
    g2.clear();
    mt.clear();
    ms.clear();
    for (const auto& nb : Lnew.blk) {
        const int rows = bra.sec[nb.sb].dim, cols = ket.sec[nb.sk].dim;
        const int s0 = (int)ms.size();
        for (int q = T.ptr[nb.a]; q < T.ptr[nb.a + 1]; ++q) {
            const int lb = L.find(T.col[q], nb.sk);
            if (lb < 0 || L.blk[lb].sb != nb.sb) continue;
            if (L.blk[lb].off + (size_t)rows * cols > L.n) throw Error(MPSPT_ERR_INVALID, "env mix source outside L");
            ms.push_back({L.ptr(L.blk[lb]), cols, 0, T.val[q]});
        }
        mt.push_back({Lnew.ptr(nb), rows, cols, cols, s0, (int)ms.size(), 0});
    }
    upload_mix(st);
}

// R_new[a](sb, sk) = sum_{s,t} A_bra(sb, s) [sum_b W_ab(s,t) R_b(sr_b, sr_k)] A_ket(sk, t)^T
void EnvPlan::build_right(const MPO& W, int site, const EnvT& R, const SiteT& Abra, const SiteT& Aket,
                          const Bond& braL, const Bond& ketL, const Bond& braR, const Bond& ketR,
                          EnvT& Rnew, cudaStream_t st) {
    g1.clear();
    g2.clear();
    mt.clear();
    ms.clear();
    const int nkb = (int)Aket.blk.size();
    // g1: Y_kb = A_ket(kb) R_panel(sr_k)^T, dim(sl_k) x (panel rows)
    std::vector<long long> yoff(nkb, -1);
    size_t ys = 0;
    for (int kb = 0; kb < nkb; ++kb) {
        const auto& K = Aket.blk[kb];
        if (R.prows[K.sr] == 0) continue;
        yoff[kb] = (long long)ys;
        ys += (size_t)ketL.sec[K.sl].dim * R.prows[K.sr];
    }
    Y.ensure((ys + 1) * sizeof(double), st);
    double* Yp = Y.as<double>();
    for (int kb = 0; kb < nkb; ++kb) {
        if (yoff[kb] < 0) continue;
        const auto& K = Aket.blk[kb];
        const int md = ketL.sec[K.sl].dim, kd = ketR.sec[K.sr].dim, P = R.prows[K.sr];
        const int m0 = g1.mark();
        g1.op(Aket.ptr(K), kd, R.panel(K.sr), kd, kd, 2, 1.0);
        g1.block(Yp + yoff[kb], P, md, P, 0, m0);
    }
    // mix: Z_(out, s) = sum over the elements (a, s, t -> b) of v Y_(b, kb(t)), dim(sk) x dim(sr_b)
    const std::vector<MPO::El>& el = W.out_el[site];
    const std::vector<int>& at = W.out_at[site];
    struct ZB { int nb, s, bb; size_t off; int rows, cols; };
    std::vector<ZB> zb;
    size_t zs = 0;
    check_range(Yp, ys * sizeof(double), "env mix Y");
    for (int nbi = 0; nbi < (int)Rnew.blk.size(); ++nbi) {
        const auto& nbk = Rnew.blk[nbi];
        const int nd = ketL.sec[nbk.sk].dim;
        const int* blk_t[4];   // ket-side lookups depend on t only
        double* y_t[4];
        int ld_t[4];
        for (int t = 0; t < 4; ++t) {
            const int kb = Aket.find(nbk.sk, t);
            const bool ok = kb >= 0 && yoff[kb] >= 0;
            blk_t[t] = ok ? R.row(Aket.blk[kb].sr) : nullptr;
            y_t[t] = ok ? Yp + yoff[kb] : nullptr;
            ld_t[t] = ok ? R.prows[Aket.blk[kb].sr] : 0;
        }
        for (int s = 0; s < 4; ++s) {
            const int bb = Abra.find(nbk.sb, s);
            if (bb < 0) continue;
            const int srb = Abra.blk[bb].sr;
            const int cols = braR.sec[srb].dim;
            const int s0 = (int)ms.size();
            for (int q = at[(size_t)nbk.a * 4 + s]; q < at[(size_t)nbk.a * 4 + s + 1]; ++q) {
                const MPO::El& E = el[q];
                if (!blk_t[E.t]) continue;
                const int rb = blk_t[E.t][E.x];
                if (rb < 0 || R.blk[rb].sb != srb) continue;
                double* src = y_t[E.t] + R.blk[rb].roff;
                if (src + (size_t)(nd - 1) * ld_t[E.t] + cols > Yp + ys)
                    throw Error(MPSPT_ERR_INVALID, "env mix source outside Y");
                ms.push_back({src, ld_t[E.t], 0, E.v});
            }
            if ((int)ms.size() == s0) continue;
            zb.push_back({nbi, s, bb, zs, nd, cols});
            mt.push_back({nullptr, nd, cols, cols, s0, (int)ms.size(), 0});
            zs += (size_t)nd * cols;
        }
    }
    Z.ensure((zs + 1) * sizeof(double), st);
    double* Zp = Z.as<double>();
    for (size_t q = 0; q < zb.size(); ++q) mt[q].dst = Zp + zb[q].off;
    // g2: R_new(out) = sum_s A_bra(sb, s) Z_(out, s)^T
    size_t z = 0;
    for (int nbi = 0; nbi < (int)Rnew.blk.size(); ++nbi) {
        const auto& nbk = Rnew.blk[nbi];
        const int md = braL.sec[nbk.sb].dim, nd = ketL.sec[nbk.sk].dim;
        const int m0 = g2.mark();
        for (; z < zb.size() && zb[z].nb == nbi; ++z)
            g2.op(Abra.ptr(Abra.blk[zb[z].bb]), zb[z].cols, Zp + zb[z].off, zb[z].cols, zb[z].cols, 2, 1.0);
        g2.block(Rnew.ptr(nbk), nd, md, nd, 0, m0);
    }
    upload_mix(st);
}

}  // namespace mpspt
