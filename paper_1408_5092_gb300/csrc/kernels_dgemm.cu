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

#include "kernels.h"

namespace mpspt {
namespace {

constexpr int DT = 128;       // threads: four warps
constexpr int OPB = 64;       // K-list entries staged in shared memory at a time

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1},{%2},{%3},{%0,%1};"
                 : "+d"(c[0]), "+d"(c[1])
                 : "d"(a), "d"(b));
}

// MI x NI pieces of 8 x 8: 16 x 16 (MI = NI = 2) or 32 x 32 (4).
template <int MI, int NI>
__global__ void __launch_bounds__(DT) k_dgemm(const GemmBlk* __restrict__ blks, const unsigned* __restrict__ unit_blk,
                                              int nunit, const GemmOp* __restrict__ ops, double* part, unsigned* tick,
                                              const int* __restrict__ skip) {
    if (skip && *skip) return;
    constexpr int TM = 8 * MI, TN = 8 * NI;
    __shared__ GemmOp sop[OPB];
    __shared__ double red[4][TM * TN];
    __shared__ int last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int fr = lane >> 2, fk = lane & 3;   // fragment row (column of B) and K position
    for (int u = blockIdx.x; u < nunit; u += gridDim.x) {
        const GemmBlk b = blks[unit_blk[u]];
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
            __syncthreads();
            for (int o = tid; o < nb; o += DT) sop[o] = ops[ob + o];
            __syncthreads();
            // (o, s, j): entry, its first step, the warp's step inside it
            int o = -1, s = base, cnt = 0, j = 0;
            double fa[MI], fb[NI], ga[MI], gb[NI];
            auto next = [&]() -> bool {
                j += 4;
                while (j >= cnt) {
                    s += cnt;
                    if (++o >= nb) return false;
                    cnt = (sop[o].k + 3) >> 2;
                    j = (cls - s) & 3;
                    if (s + j < q0) j += (q0 - s - j + 3) & ~3;
                }
                return s + j < q1;
            };
            auto load = [&](double (&xa)[MI], double (&xb)[NI]) {
                const GemmOp& op = sop[o];
                const int k = 4 * j + fk;
                const bool kin = k < op.k;
                const size_t ra = (op.trans & 1) ? 1 : op.lda, ca = (op.trans & 1) ? op.lda : 1;
                const size_t rb = (op.trans & 2) ? op.ldb : 1, cb = (op.trans & 2) ? 1 : op.ldb;
                const double* A = op.A + (size_t)(r0 + fr) * ra + (size_t)k * ca;
                const double* B = op.B + (size_t)(c0 + fr) * rb + (size_t)k * cb;
#pragma unroll
                for (int i = 0; i < MI; ++i) xa[i] = (kin && 8 * i + fr < mrem) ? __ldg(A + 8 * i * ra) : 0.0;
#pragma unroll
                for (int i = 0; i < NI; ++i) xb[i] = (kin && 8 * i + fr < nrem) ? __ldg(B + 8 * i * rb) : 0.0;
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
                for (int i = 0; i < nb; ++i) base += (sop[i].k + 3) >> 2;
        }
        // four class sums -> tile
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int c = 0; c < NI; ++c) {
                double* d = &red[cls][(8 * i + fr) * TN + 8 * c + 2 * fk];
                d[0] = acc[i][c][0];
                d[1] = acc[i][c][1];
            }
        __syncthreads();
        bool store = true;
        double* pt = nullptr;
        if (b.S > 1) {
            pt = part + b.part + (size_t)tile * b.S * (TM * TN);
            double* mine = pt + (size_t)piece * (TM * TN);
            for (int e = tid; e < mrem * TN; e += DT) mine[e] = ((red[0][e] + red[1][e]) + red[2][e]) + red[3][e];
            __threadfence();
            __syncthreads();
            if (tid == 0) {
                unsigned* t = tick + b.tick + tile;
                last = atomicAdd(t, 1u) == (unsigned)b.S - 1;
                if (last) *t = 0;
            }
            __syncthreads();
            store = last != 0;
            if (store) __threadfence();
        }
        if (store)
            for (int e = tid; e < mrem * TN; e += DT) {
                const int r = e / TN, c = e % TN;
                if (c >= nrem) continue;
                double v;
                if (b.S == 1) v = ((red[0][e] + red[1][e]) + red[2][e]) + red[3][e];
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
                *dst = b.accumulate ? *dst + v : v;
            }
        __syncthreads();   // red, last and sop are free for the next unit
    }
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

}  // namespace

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
