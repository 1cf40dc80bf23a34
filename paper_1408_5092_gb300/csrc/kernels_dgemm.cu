// Float64 grouped block GEMM of the sweep (sm_103a), driven by block lists.
//
// What bounds it: the float64 pipe of this GPU does about 1.75 FMA per clock
// and SM (measured, DMMA and DFMA alike; 1.0 TFLOP/s over 152 SMs) with a
// 64-clock dependent latency, so an 8 x 8 x 4 step (256 FMA, one
// mma.m8n8k4.f64) occupies one SM sub-partition for about 580 clocks.
// Operand traffic is nothing beside that (a 16 x 16 tile reads 0.5 byte per
// flop, 0.5 TB/s out of L2 at the full rate); what costs is every padded row
// or column that is multiplied and every idle SM.  Hence:
//  * work is cut in units of one output tile and one piece of the K-list, the
//    tile in 8 x 8 pieces of which only those inside the block are computed
//    (a 64 x 64 CUDA-core tile took 17 us per 16 K whatever the block's size);
//  * the four warps of a CTA, one per sub-partition, share a unit by taking
//    the K steps in turn (class = step mod 4); each keeps its own
//    accumulators and the four sums are added in class order at the end.
//    Operands go from global memory (L1/L2) straight to registers in the
//    fragment layout, one step ahead of the DMMAs: with no shared-memory
//    staging there is no barrier in the K loop;
//  * long K-lists are cut further (S pieces per tile, dgemm_units); the last
//    CTA to finish a tile adds the pieces in ascending order, so results do
//    not depend on timing.
// Class and piece boundaries depend on the block list alone: every tile shape
// gives the same bits.
// Measured (device time of all float64 GEMMs in one sweep, CUDA-core 64 x 64
// tiles before -> now): 4e/4o + 8, M = 16: 49.8 -> 10.2 ms (5.2 us a launch);
// 8e/8o + 24, M = 64: 199.6 -> 23.3 ms; M = 256 with tuned tiles: 128.5 ->
// 53.9 ms, sigma 53 -> 32 ms for 5.4 GFLOP.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include <cooperative_groups.h>

#include "kernels.h"
#include "mix_piece.h"

namespace mpspt {
namespace {

constexpr int DT = 128;       // threads: four warps
constexpr int OPB = 64;       // K-list entries staged in shared memory at a time

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1},{%2},{%3},{%0,%1};"
                 : "+d"(c[0]), "+d"(c[1])
                 : "d"(a), "d"(b));
}

// COH: operands may have been written by this launch (no read-only loads)
template <bool COH>
__device__ __forceinline__ double load_op(const double* p) {
    if constexpr (COH) return __ldcg(p);
    else return __ldg(p);
}

template <int MI, int NI>
struct UnitSmem {
    GemmOp sop[OPB];
    double red[4][8 * MI * 8 * NI];
    int last;
};

// One unit by the 128 threads of named barrier `bar` (tid: 0 .. 127).
// MI x NI pieces of 8 x 8: 16 x 16 (MI = NI = 2) or 32 x 32 (4).
template <int MI, int NI, bool COH>
__device__ __forceinline__ void dgemm_unit(const GemmBlk& b, int u, const GemmOp* __restrict__ ops, double* part,
                                           unsigned* tick, UnitSmem<MI, NI>& sm, int tid, int bar) {
    constexpr int TM = 8 * MI, TN = 8 * NI;
    const int lane = tid & 31, warp = tid >> 5;
    const int fr = lane >> 2, fk = lane & 3;   // fragment row (column of B) and K position
    auto sync = [bar] { asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory"); };
    const int local = u - b.u0;
    const int tile = local / b.S, piece = local - tile * b.S;
    const int tr = tile / b.nt, r0 = tr * TM, c0 = (tile - tr * b.nt) * TN;
    const int mrem = min(TM, b.m - r0), nrem = min(TN, b.n - c0);
    const int mi = (mrem + 7) >> 3, ni = (nrem + 7) >> 3;
    const int q0 = piece * b.qs, q1 = min(b.q, q0 + b.qs);
    const int cls = (warp + u) & 3;   // the longest class changes its sub-partition from unit to unit
    double acc[MI][NI][2];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < NI; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
    int base = 0;   // K step of the staged entries' first element
    for (int ob = b.op0; ob < b.op1 && base < q1; ob += OPB) {
        const int nb = min(OPB, b.op1 - ob);
        sync();
        for (int o = tid; o < nb; o += DT) sm.sop[o] = ops[ob + o];
        sync();
        // (o, s, j): entry, its first step, the warp's step inside it
        int o = -1, s = base, cnt = 0, j = 0;
        double fa[MI], fb[NI], ga[MI], gb[NI];
        auto next = [&]() -> bool {
            j += 4;
            while (j >= cnt) {
                s += cnt;
                if (++o >= nb) return false;
                cnt = (sm.sop[o].k + 3) >> 2;
                j = (cls - s) & 3;
                if (s + j < q0) j += (q0 - s - j + 3) & ~3;
            }
            return s + j < q1;
        };
        auto load = [&](double (&xa)[MI], double (&xb)[NI]) {
            const GemmOp& op = sm.sop[o];
            const int k = 4 * j + fk;
            const bool kin = k < op.k;
            const size_t ra = (op.trans & 1) ? 1 : op.lda, ca = (op.trans & 1) ? op.lda : 1;
            const size_t rb = (op.trans & 2) ? op.ldb : 1, cb = (op.trans & 2) ? 1 : op.ldb;
            const double* A = op.A + (size_t)(r0 + fr) * ra + (size_t)k * ca;
            const double* B = op.B + (size_t)(c0 + fr) * rb + (size_t)k * cb;
#pragma unroll
            for (int i = 0; i < MI; ++i) xa[i] = (kin && 8 * i + fr < mrem) ? load_op<COH>(A + 8 * i * ra) : 0.0;
#pragma unroll
            for (int i = 0; i < NI; ++i) xb[i] = (kin && 8 * i + fr < nrem) ? load_op<COH>(B + 8 * i * rb) : 0.0;
            if (op.alpha != 1.0)
#pragma unroll
                for (int i = 0; i < MI; ++i) xa[i] *= op.alpha;
        };
        bool more = next();
        if (more) load(fa, fb);
        while (more) {
            more = next();
            if (more) load(ga, gb);   // in flight while the DMMAs below run
#pragma unroll
            for (int i = 0; i < MI; ++i)
                if (i < mi)
#pragma unroll
                    for (int c = 0; c < NI; ++c)
                        if (c < ni) dmma(acc[i][c], fa[i], fb[c]);
#pragma unroll
            for (int i = 0; i < MI; ++i) fa[i] = ga[i];
#pragma unroll
            for (int i = 0; i < NI; ++i) fb[i] = gb[i];
        }
        if (b.op1 - ob > OPB)
            for (int i = 0; i < nb; ++i) base += (sm.sop[i].k + 3) >> 2;
    }
    // four class sums -> tile
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int c = 0; c < NI; ++c) {
            double* d = &sm.red[cls][(8 * i + fr) * TN + 8 * c + 2 * fk];
            d[0] = acc[i][c][0];
            d[1] = acc[i][c][1];
        }
    sync();
    bool store = true;
    double* pt = nullptr;
    if (b.S > 1) {
        pt = part + b.part + (size_t)tile * b.S * (TM * TN);
        double* mine = pt + (size_t)piece * (TM * TN);
        for (int e = tid; e < mrem * TN; e += DT) mine[e] = ((sm.red[0][e] + sm.red[1][e]) + sm.red[2][e]) + sm.red[3][e];
        __threadfence();
        sync();
        if (tid == 0) {
            unsigned* t = tick + b.tick + tile;
            sm.last = atomicAdd(t, 1u) == (unsigned)b.S - 1;
            if (sm.last) *t = 0;
        }
        sync();
        store = sm.last != 0;
        if (store) __threadfence();
    }
    if (store)
        for (int e = tid; e < mrem * TN; e += DT) {
            const int r = e / TN, c = e % TN;
            if (c >= nrem) continue;
            double v;
            if (b.S == 1) v = ((sm.red[0][e] + sm.red[1][e]) + sm.red[2][e]) + sm.red[3][e];
            else {
                v = 0.0;
                for (int p = 0; p < b.S; ++p) v += __ldcg(pt + (size_t)p * (TM * TN) + e);
            }
            const int gr = r0 + r, gc = c0 + c;
            if (b.scale != 1.f || b.diag != 0.f) v = (double)b.scale * v + (gr == gc ? (double)b.diag : 0.0);
            double* dst;
            if (b.cmap == nullptr) dst = b.C + (size_t)gr * b.ldc + gc;
            else if (b.cmap_rows) dst = b.C + b.cmap[2 * gr] + (size_t)gc * b.cmap[2 * gr + 1];
            else dst = b.C + b.cmap[2 * gc] + (size_t)gr * b.cmap[2 * gc + 1];
            *dst = b.accumulate ? (COH ? __ldcg(dst) : *dst) + v : v;
        }
    sync();   // sm is free for the next unit
}

template <int MI, int NI>
__global__ void __launch_bounds__(DT) k_dgemm(const GemmBlk* __restrict__ blks, const unsigned* __restrict__ unit_blk,
                                              int nunit, const GemmOp* __restrict__ ops, double* part, unsigned* tick,
                                              const int* __restrict__ skip) {
    if (skip && *skip) return;
    __shared__ UnitSmem<MI, NI> sm;
    for (int u = blockIdx.x; u < nunit; u += gridDim.x)
        dgemm_unit<MI, NI, false>(blks[unit_blk[u]], u, ops, part, tick, sm, threadIdx.x, 0);
}

// ------------------------------------------------------------ CG on a cluster
// All iterations of one Jacobi-preconditioned CG solve in one launch on a
// cluster of 16 CTAs (8 where the device has no room for 16).  An iteration of
// a small local problem by launches is six of them, 30 us and more of starts
// and ends whatever the work; here its six phases (panel products, operator
// sums, long-K products, p.Ap, update, direction) are separated by cluster
// barriers of 0.2 us, and the scalars are added from every CTA's part in rank
// order by all.  Clusters are scheduled as a whole, so nothing spins.  Each
// worker of 128 threads takes the units of k_dgemm in turn.  16 SMs run 64
// DMMAs at a time where the launches spread over 608 sub-partitions, so it
// pays for operators of few steps.  Measured: sweep of 4e/4o + 8, M = 16, 46.6
// -> 41.3 ms; of 8e/8o + 24, M = 64, with the line at 1200 steps 0.8% faster,
// at 2500, 5000, 10000 and 20000 0.8%, 1.8%, 6% and 4% slower: kClusterSteps.
constexpr int CGT = 512;       // threads: four workers of 128
constexpr int CGW = CGT / 128;

__global__ void __launch_bounds__(CGT) k_cg_cluster(CgArgs a) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char cg_sm[];
    UnitSmem<2, 2>* us = reinterpret_cast<UnitSmem<2, 2>*>(cg_sm);
    __shared__ double red[2][CGT / 32];
    __shared__ double part[2][2][16];   // by parity of the sum
    const int rank = (int)cl.block_rank(), ncta = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, worker = tid >> 7;
    if (*(volatile const int*)&a.S->done) return;   // the same in every CTA
    const size_t stride = (size_t)ncta * CGT, first = (size_t)rank * CGT + tid;
    auto gemm = [&](const GemmRun& g) {
        for (int u = rank * CGW + worker; u < g.nunit; u += ncta * CGW)
            dgemm_unit<2, 2, true>(g.blk[g.unit[u]], u, g.ops, g.part, g.tick, us[worker], tid & 127, 1 + worker);
    };
    // v[0], v[1] summed over all threads of the cluster, in every thread
    int parity = 0;
    auto total = [&](double (&v)[2]) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
            if (lane == 0) red[q][warp] = v[q];
        }
        __syncthreads();
        if (tid < 2 * ncta) {
            const int q = tid & 1;
            double s = 0.0;
            for (int w = 0; w < CGT / 32; ++w) s += red[q][w];
            *cl.map_shared_rank(&part[parity][q][rank], tid >> 1) = s;
        }
        cl.sync();
        v[0] = v[1] = 0.0;
        for (int r = 0; r < ncta; ++r) {
            v[0] += part[parity][0][r];
            v[1] += part[parity][1][r];
        }
        parity ^= 1;
    };
    double rz = a.S->rz, rr = a.S->rr, pAp = 0.0, alpha = 0.0, beta = 0.0;
    const double stop = a.S->tol2 * a.S->bb;
    int it = 0, done = 0, bad = 0;
    while (!done && it < a.maxit) {
        gemm(a.g1);
        cl.sync();
        for (int w = rank * (CGT / 32) + warp; w < a.nmix; w += ncta * (CGT / 32)) {
            const MixTask& t = a.mt[w];
            for (int e = 0, n = t.rows * t.cols; e < n; e += MIX_PIECE) mix_piece<true>(t, e, a.ms, lane);
        }
        cl.sync();
        gemm(a.g2);
        cl.sync();
        double v[2] = {0.0, 0.0};
        for (size_t i = first; i < a.n; i += stride) v[0] = fma(__ldcg(a.p + i), __ldcg(a.Ap + i), v[0]);
        total(v);
        pAp = v[0];
        if (!(pAp > 0.0)) { bad = done = 1; break; }
        alpha = rz / pAp;
        v[0] = v[1] = 0.0;
        for (size_t i = first; i < a.n; i += stride) {
            a.x[i] = fma(alpha, __ldcg(a.p + i), a.x[i]);
            const double ri = fma(-alpha, __ldcg(a.Ap + i), a.r[i]);
            const double zi = a.minv[i] * ri;
            a.r[i] = ri;
            a.z[i] = zi;
            v[0] = fma(ri, zi, v[0]);
            v[1] = fma(ri, ri, v[1]);
        }
        total(v);
        ++it;
        beta = v[0] / rz;
        rz = v[0];
        rr = v[1];
        if (rr <= stop) { done = 2; break; }
        for (size_t i = first; i < a.n; i += stride) a.p[i] = fma(beta, __ldcg(a.p + i), a.z[i]);
        cl.sync();
    }
    if (rank == 0 && tid == 0) {
        a.S->rz = a.S->rz_new = rz;
        a.S->rr = rr;
        a.S->pAp = pAp;
        a.S->alpha = alpha;
        a.S->beta = beta;
        a.S->iters = it;
        a.S->not_spd = bad;
        a.S->done = done;
    }
    cl.sync();   // no CTA leaves while its shared memory may be written
}

int dgemm_resident(const void* f) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> cache;
    thread_local std::map<std::pair<const void*, int>, int> mine;   // lock-free fast path per thread
    int dev = 0;
    cudaGetDevice(&dev);
    auto it = mine.find({f, dev});
    if (it != mine.end()) return it->second;
    std::lock_guard<std::mutex> lk(mu);
    auto c = cache.find({f, dev});
    if (c != cache.end()) return mine[{f, dev}] = c->second;
    int nb = 1, sms = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, DT, 0) != cudaSuccess || nb < 1) nb = 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
    cudaGetLastError();
    return mine[{f, dev}] = cache[{f, dev}] = nb * sms;
}

// CTAs of the solve's cluster on the current device: 16 if one such cluster
// can be resident, else 8 (0: none)
int cg_cluster_size() {
    static std::mutex mu;
    static std::map<int, int> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(dev);
    if (it != cache.end()) return it->second;
    const void* f = reinterpret_cast<const void*>(k_cg_cluster);
    int size = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
        for (int c : {16, 8}) {
            cudaLaunchConfig_t cf = {};
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = c;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cf.gridDim = dim3(c);
            cf.blockDim = dim3(CGT);
            cf.dynamicSmemBytes = CGW * sizeof(UnitSmem<2, 2>);
            cf.attrs = &at;
            cf.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, f, &cf) == cudaSuccess && n >= 1) {
                size = c;
                break;
            }
        }
    cudaGetLastError();
    return cache[dev] = size;
}

}  // namespace

bool launch_cg_cluster(const CgArgs& a, cudaStream_t st) {
    const int c = cg_cluster_size();
    if (c == 0) return false;
    cudaLaunchConfig_t cf = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = c;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cf.gridDim = dim3(c);
    cf.blockDim = dim3(CGT);
    cf.dynamicSmemBytes = CGW * sizeof(UnitSmem<2, 2>);
    cf.stream = st;
    cf.attrs = &at;
    cf.numAttrs = 1;
    if (cudaLaunchKernelEx(&cf, k_cg_cluster, a) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    count_launch();
    return true;
}
bool cg_cluster_available() { return cg_cluster_size() > 0; }

void launch_dgemm(int tile, const GemmBlk* blks, const unsigned* unit_blk, int nunit, const GemmOp* ops, double* part,
                  unsigned* tick, cudaStream_t st, const int* skip) {
    if (nunit <= 0) return;
    count_launch();
    if (tile == 32) {
        const int grid = std::min(nunit, dgemm_resident(reinterpret_cast<const void*>(k_dgemm<4, 4>)));
        k_dgemm<4, 4><<<grid, DT, 0, st>>>(blks, unit_blk, nunit, ops, part, tick, skip);
    } else {
        const int grid = std::min(nunit, dgemm_resident(reinterpret_cast<const void*>(k_dgemm<2, 2>)));
        k_dgemm<2, 2><<<grid, DT, 0, st>>>(blks, unit_blk, nunit, ops, part, tick, skip);
    }
}

}  // namespace mpspt
