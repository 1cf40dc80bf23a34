// CUDA-core kernels of the MPS-PT hot path (sm_103a): grouped block GEMM in
// float32 arithmetic driven by task lists, Jacobi diagonal, block copies, and
// the CG vector kernels with deterministic (fixed-order) reductions.
#include "kernels.h"
#include "mix_piece.h"

#include <atomic>
#include <algorithm>
#include <cstdio>
#include <map>
#include <mutex>
#include <set>
#include <utility>

namespace mpspt {
namespace {

std::atomic<long long> g_launches{0};
thread_local long long t_launches = 0;   // this host thread's launches
inline void counted() {
    g_launches.fetch_add(1, std::memory_order_relaxed);
    ++t_launches;
}

constexpr int TK = 16;
constexpr int NT = 256;

// float64 operand -> arithmetic type.  To float32 the rounding is done with
// integer operations: the float64 pipe of this GPU is narrow and the
// conversion instruction would bound the tile staging.  Magnitudes below
// the float32 normal range become signed zero.
__device__ __forceinline__ float d2f_rn(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const int e = (int)((b >> 52) & 0x7FF);
    const unsigned long long m = b & 0xFFFFFFFFFFFFFULL;
    if (e == 0x7FF) return __uint_as_float(sign | 0x7F800000u | (m ? 0x400000u : 0u));
    const int fe = e - 1023 + 127;
    if (fe <= 0) return __uint_as_float(sign);
    if (fe >= 255) return __uint_as_float(sign | 0x7F800000u);
    const unsigned mant = (unsigned)(m >> 29);
    const unsigned rem = (unsigned)(m & 0x1FFFFFFFULL);
    unsigned f = sign | ((unsigned)fe << 23) | mant;
    if (rem > 0x10000000u || (rem == 0x10000000u && (mant & 1u))) f += 1u;
    return __uint_as_float(f);
}
// Grouped GEMM: one CTA per output tile, looping over the tile's K-list.
// 16x16 threads; thread (tx, ty) owns rows ty + 16 i (i < TM/16) and
// cols tx + 16 j (j < TN/16).  Operands and results are float64.
// Persistent: the grid is at most the resident CTAs of the GPU, and CTA b
// takes tasks b, b + gridDim.x, ... (the planner orders tasks longest first).
template <int TM, int TN>
__global__ void __launch_bounds__(NT) k_gemm(const GemmTask* __restrict__ tasks, int ntask,
                                             const GemmOp* __restrict__ ops,
                                             const int* __restrict__ skip) {
    if (skip && *skip) return;
    constexpr int RI = TM / 16, RJ = TN / 16;
    __shared__ float As[TK][TM + 1];
    __shared__ float Bs[TK][TN + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  for (int ti = blockIdx.x; ti < ntask; ti += gridDim.x) {
    const GemmTask t = tasks[ti];
    float acc[RI][RJ];
#pragma unroll
    for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int j = 0; j < RJ; ++j) acc[i][j] = 0.f;
    const int mrem = min(TM, t.m - t.r0);
    const int nrem = min(TN, t.n - t.c0);
    int kbase = 0;   // position of op o's first K index in the concatenated K-list
    for (int o = t.op0; o < t.op1; ++o) {
        const GemmOp op = ops[o];
        const int kb = max(0, t.kb - kbase), ke = min(op.k, t.ke - kbase);
        kbase += op.k;
        if (kb >= ke) continue;
        const bool ta = op.trans & 1, tb = op.trans & 2;
        const float alpha = d2f_rn(op.alpha);
        for (int k0 = kb; k0 < ke; k0 += TK) {
            const int krem = min(TK, ke - k0);
            for (int e = threadIdx.x; e < TM * TK; e += NT) {
                int i, kk;
                if (ta) { i = e % TM; kk = e / TM; }
                else { kk = e % TK; i = e / TK; }
                float v = 0.f;
                if (i < mrem && kk < krem) {
                    const int row = t.r0 + i, kg = k0 + kk;
                    v = d2f_rn(ta ? op.A[(size_t)kg * op.lda + row] : op.A[(size_t)row * op.lda + kg]) * alpha;
                }
                As[kk][i] = v;
            }
            for (int e = threadIdx.x; e < TN * TK; e += NT) {
                int j, kk;
                if (tb) { kk = e % TK; j = e / TK; }
                else { j = e % TN; kk = e / TN; }
                float v = 0.f;
                if (j < nrem && kk < krem) {
                    const int col = t.c0 + j, kg = k0 + kk;
                    v = d2f_rn(tb ? op.B[(size_t)col * op.ldb + kg] : op.B[(size_t)kg * op.ldb + col]);
                }
                Bs[kk][j] = v;
            }
            __syncthreads();
#pragma unroll
            for (int kk = 0; kk < TK; ++kk) {
                float a[RI], b[RJ];
#pragma unroll
                for (int i = 0; i < RI; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < RJ; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
                for (int i = 0; i < RI; ++i)
#pragma unroll
                    for (int j = 0; j < RJ; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int i = 0; i < RI; ++i) {
        const int r = ty + 16 * i;
        if (r >= mrem) continue;
#pragma unroll
        for (int j = 0; j < RJ; ++j) {
            const int c = tx + 16 * j;
            if (c >= nrem) continue;
            if (t.part) { t.part[r * TN + c] = (double)acc[i][j]; continue; }
            const int gr = t.r0 + r, gc = t.c0 + c;
            double* dst;
            if (t.cmap == nullptr) dst = t.C + (size_t)gr * t.ldc + gc;
            else if (t.cmap_rows) dst = t.C + t.cmap[2 * gr] + (size_t)gc * t.cmap[2 * gr + 1];
            else dst = t.C + t.cmap[2 * gc] + (size_t)gr * t.cmap[2 * gc + 1];
            *dst = t.accumulate ? *dst + (double)acc[i][j] : (double)acc[i][j];
        }
    }
  }
}

// Split-K reduction: partial tiles summed in ascending order (deterministic).
// Bound by the float64 additions of one SM, so a tile is shared by eight CTAs
// (one per tile took 48 us for tiles of 128 x 64).
__global__ void k_splitk_reduce(const SplitRed* __restrict__ tasks, const int* __restrict__ skip) {
    if (skip && *skip) return;
    const SplitRed t = tasks[blockIdx.x];
    const int mrem = min(t.tm, t.m - t.r0), nrem = min(t.tn, t.n - t.c0);
    const size_t tile = (size_t)t.tm * t.tn;
    for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < mrem * nrem; e += gridDim.y * blockDim.x) {
        const int r = e / nrem, c = e % nrem;
        double v = 0.0;
        for (int q = 0; q < t.nparts; ++q) v += t.part[q * tile + (size_t)r * t.tn + c];
        const int gr = t.r0 + r, gc = t.c0 + c;
        double* dst;
        if (t.cmap == nullptr) dst = t.C + (size_t)gr * t.ldc + gc;
        else if (t.cmap_rows) dst = t.C + t.cmap[2 * gr] + (size_t)gc * t.cmap[2 * gr + 1];
        else dst = t.C + t.cmap[2 * gc] + (size_t)gr * t.cmap[2 * gc + 1];
        *dst = t.accumulate ? *dst + v : v;
    }
}

// dst = sum coef * src over the task's source list, in order.  Blocks are
// small (a few to a few hundred values) with up to hundreds of sources, and
// the time is the latency of each descriptor and value load over the warps in
// flight.  k_mix takes a CTA per block, k_mix_pieces a warp per MIX_PIECE
// values of a block, two per lane: the warps that a CTA per block leaves idle
// (three of four in a block of up to 32 values) hold SM slots.
__global__ void k_mix(const MixTask* __restrict__ tasks, const MixSrc* __restrict__ srcs,
                      const int* __restrict__ skip) {
    if (skip && *skip) return;
    const MixTask t = tasks[blockIdx.x];
    const int n = t.rows * t.cols;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int i = e / t.cols, j = e % t.cols;
        double s = 0.0;
        for (int q = t.s0; q < t.s1; ++q) {
            const MixSrc m = srcs[q];
            s += m.coef * m.src[(size_t)i * m.lds + j];
        }
        t.dst[(size_t)i * t.ldd + j] = s;
    }
}
__global__ void __launch_bounds__(128, 8) k_mix_pieces(const MixTask* __restrict__ tasks,
                                                        const unsigned* __restrict__ piece_task, int npiece,
                                                        const MixSrc* __restrict__ srcs, const int* __restrict__ skip) {
    if (skip && *skip) return;
    const int w = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (w >= npiece) return;
    const MixTask& t = tasks[piece_task[w]];
    mix_piece<false>(t, (w - t.p0) * MIX_PIECE, srcs, threadIdx.x & 31);
}

__global__ void k_diag(const DiagTask* __restrict__ tasks, const DiagTerm* __restrict__ terms) {
    const DiagTask t = tasks[blockIdx.x];
    const int n = t.rows * t.cols;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int l = e / t.cols, r = e % t.cols;
        double s = 0.0;
        for (int k = t.t0; k < t.t1; ++k) {
            const DiagTerm d = terms[k];
            s += d.coef * d.L[(size_t)l * (d.ldL + 1)] * d.R[(size_t)r * (d.ldR + 1)];
        }
        t.out[e] = s;
    }
}

__global__ void k_copy(const CopyTask* __restrict__ tasks) {
    const CopyTask t = tasks[blockIdx.x];
    const int n = t.rows * t.cols_n;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int i = e / t.cols_n, j = e % t.cols_n;
        double v;
        if (t.trans) v = t.src[(size_t)j * t.lds + (t.cols ? t.cols[i] : i)];
        else v = t.src[(size_t)i * t.lds + (t.cols ? t.cols[j] : j)];
        t.dst[(size_t)i * t.ldd + j] = v;
    }
}

// ----------------------------------------------------------------- vectors
// Sums over a vector: a float64 addition occupies a warp's sub-partition for
// 64 clocks however few lanes it has, so a block adds its 256 partial values
// with 8 + 5 additions of one warp per sum (a shuffle tree in every warp took
// 5 per warp and sum, and one thread adding the blocks one by one 64 clocks
// and a cache miss each).  Fixed order: deterministic.
constexpr int RB = 256;        // threads per reduction block
constexpr int RG_MAX = 456;    // max reduction blocks (three a SM)

inline int red_grid(size_t n) {
    size_t g = (n + (size_t)RB * 2 - 1) / ((size_t)RB * 2);
    if (g < 1) g = 1;
    if (g > RG_MAX) g = RG_MAX;
    return (int)g;
}

// sum of sh[0 .. n) over the calling warp, in all its lanes
__device__ __forceinline__ double warp_total(const double* x, int n) {
    double v = 0.0;
    for (int i = threadIdx.x & 31; i < n; i += 32) v += __ldcg(x + i);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Every block adds its threads' v[q], q < nv, stores the sums, and the last
// block to finish adds them over the blocks, in block order, into tot (shared
// memory, nv values); returns true in all its threads.  sh: nv x RB doubles
// of shared memory.
template <int NV>
__device__ bool grid_sum(const double (&v)[NV], int nv, double (*sh)[RB], double* tot, double* scratch,
                         unsigned* counter) {
    __shared__ bool is_last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NV; ++q)
        if (q < nv) sh[q][threadIdx.x] = v[q];
    __syncthreads();
    for (int q = warp; q < nv; q += RB / 32) {
        double x = 0.0;
#pragma unroll
        for (int i = 0; i < RB / 32; ++i) x += sh[q][lane + 32 * i];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) scratch[(size_t)q * gridDim.x + blockIdx.x] = x;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
    for (int q = warp; q < nv; q += RB / 32) {
        const double x = warp_total(scratch + (size_t)q * gridDim.x, gridDim.x);
        if (lane == 0) tot[q] = x;
    }
    if (threadIdx.x == 0) *counter = 0;
    __syncthreads();
    return true;
}

__global__ void k_dot(const double* __restrict__ x, const double* __restrict__ y, size_t n,
                      double* out, double* scratch, unsigned* counter) {
    __shared__ double sh[1][RB];
    __shared__ double tot[1];
    double v[1] = {0.0};
    for (size_t i = blockIdx.x * (size_t)RB + threadIdx.x; i < n; i += (size_t)gridDim.x * RB)
        v[0] += x[i] * y[i];
    if (grid_sum<1>(v, 1, sh, tot, scratch, counter) && threadIdx.x == 0) *out = tot[0];
}

__global__ void k_cg_init(double* r, double* z, double* p, const double* __restrict__ b,
                          const double* __restrict__ Ax, const double* __restrict__ minv, size_t n,
                          CgState* S, double tol, double* scratch, unsigned* counter) {
    __shared__ double sh[3][RB];
    __shared__ double tot[3];
    double v[3] = {0.0, 0.0, 0.0};
    for (size_t i = blockIdx.x * (size_t)RB + threadIdx.x; i < n; i += (size_t)gridDim.x * RB) {
        const double ri = b[i] - Ax[i];
        const double zi = minv[i] * ri;
        r[i] = ri;
        z[i] = zi;
        p[i] = zi;
        v[0] += ri * zi;
        v[1] += ri * ri;
        v[2] += b[i] * b[i];
    }
    if (grid_sum<3>(v, 3, sh, tot, scratch, counter) && threadIdx.x == 0) {
        S->rz = tot[0];
        S->rr = tot[1];
        S->bb = tot[2];
        S->tol2 = tol * tol;
        S->iters = 0;
        S->not_spd = 0;
        S->done = (tot[1] <= tol * tol * tot[2]) || tot[2] == 0.0;
    }
}

__global__ void k_cg_pap(const double* __restrict__ p, const double* __restrict__ Ap, size_t n,
                         CgState* S, double* scratch, unsigned* counter) {
    if (S->done) return;
    __shared__ double sh[1][RB];
    __shared__ double tot[1];
    double v[1] = {0.0};
    for (size_t i = blockIdx.x * (size_t)RB + threadIdx.x; i < n; i += (size_t)gridDim.x * RB)
        v[0] += p[i] * Ap[i];
    if (grid_sum<1>(v, 1, sh, tot, scratch, counter) && threadIdx.x == 0) {
        S->pAp = tot[0];
        if (!(tot[0] > 0.0)) { S->not_spd = 1; S->done = 1; }
        else S->alpha = S->rz / tot[0];
    }
}

__global__ void k_cg_update(double* x, double* r, double* z, const double* __restrict__ p,
                            const double* __restrict__ Ap, const double* __restrict__ minv,
                            size_t n, CgState* S, double* scratch, unsigned* counter) {
    if (S->done) return;
    __shared__ double sh[2][RB];
    __shared__ double tot[2];
    const double a = S->alpha;
    double v[2] = {0.0, 0.0};
    for (size_t i = blockIdx.x * (size_t)RB + threadIdx.x; i < n; i += (size_t)gridDim.x * RB) {
        x[i] += a * p[i];
        const double ri = r[i] - a * Ap[i];
        const double zi = minv[i] * ri;
        r[i] = ri;
        z[i] = zi;
        v[0] += ri * zi;
        v[1] += ri * ri;
    }
    if (grid_sum<2>(v, 2, sh, tot, scratch, counter) && threadIdx.x == 0) {
        S->rz_new = tot[0];
        S->rr = tot[1];
        S->beta = tot[0] / S->rz;
        S->rz = tot[0];
        S->iters += 1;
        if (tot[1] <= S->tol2 * S->bb) S->done = 2;
    }
}

__global__ void k_cg_dir(double* p, const double* __restrict__ z, size_t n, const CgState* S) {
    if (S->done) return;
    const double be = S->beta;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        p[i] = z[i] + be * p[i];
}

__global__ void k_axpy(double* y, const double* __restrict__ x, double a, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] += a * x[i];
}
__global__ void k_scale(double* y, const double* __restrict__ x, double a, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = a * x[i];
}
__global__ void k_minv(double* y, const double* __restrict__ d, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = d[i] > 0.0 ? 1.0 / d[i] : 0.0;
}
// ---- Davidson (ground-state DMRG).  Bases V, AV: vectors of n, leading
// dimension n.  One pass over the vectors per step instead of one launch per
// inner product and per update.
constexpr int DAV_MAX = 16;   // basis vectors at most
struct DavY { double y[DAV_MAX]; };

// q < m: out[q] = V_q . t
// MODE 0: t = r / (theta - d), the denominator kept at least 1e-8 max(1,
//         |theta|) away from zero (its sign kept)
// MODE 1: t -= sum_q coef[q] V_q
// MODE 2: the same, and out[0] = t . t instead
// MODE 3: t = src
template <int MODE>
__global__ void __launch_bounds__(RB) k_dav_pass(double* t, const double* __restrict__ V, int m, size_t n,
                                                 const double* __restrict__ src, const double* __restrict__ d,
                                                 double theta, const double* coef, double* out, double* scratch,
                                                 unsigned* counter) {
    constexpr int NV = MODE == 2 ? 1 : DAV_MAX;
    __shared__ double sh[NV][RB];
    __shared__ double tot[NV];
    const double eps = 1e-8 * fmax(1.0, fabs(theta));
    double c[DAV_MAX], v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = 0.0;
    if (MODE == 1 || MODE == 2)
#pragma unroll
        for (int q = 0; q < DAV_MAX; ++q) c[q] = q < m ? coef[q] : 0.0;
    for (size_t i = blockIdx.x * (size_t)RB + threadIdx.x; i < n; i += (size_t)gridDim.x * RB) {
        double x;
        if (MODE == 0) {
            double den = theta - d[i];
            if (fabs(den) < eps) den = den < 0.0 ? -eps : eps;
            x = src[i] / den;
        } else {
            x = MODE == 3 ? src[i] : t[i];
        }
        double b[DAV_MAX];
#pragma unroll
        for (int q = 0; q < DAV_MAX; ++q) b[q] = q < m && MODE != 2 ? V[(size_t)q * n + i] : 0.0;
        if (MODE == 1 || MODE == 2)
#pragma unroll
            for (int q = 0; q < DAV_MAX; ++q)
                if (q < m) x = fma(-c[q], MODE == 2 ? V[(size_t)q * n + i] : b[q], x);
        t[i] = x;
        if (MODE == 2) v[0] = fma(x, x, v[0]);
        else
#pragma unroll
            for (int q = 0; q < NV; ++q)
                if (q < m) v[q] = fma(b[q], x, v[q]);
    }
    const int nv = MODE == 2 ? 1 : m;
    __syncthreads();
    if (grid_sum<NV>(v, nv, sh, tot, scratch, counter) && threadIdx.x < nv) out[threadIdx.x] = tot[threadIdx.x];
}

// p = t = t / sqrt(*norm2)
__global__ void k_dav_unit(double* t, double* p, const double* __restrict__ norm2, size_t n) {
    const double a = 1.0 / sqrt(*norm2);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double v = a * t[i];
        t[i] = v;
        p[i] = v;
    }
}

// Ritz vector x = sum y_q V_q, ax = sum y_q AV_q, z = ax - theta x; *out = z . z
__global__ void __launch_bounds__(RB) k_dav_ritz(double* x, double* ax, double* z, const double* __restrict__ V,
                                                 const double* __restrict__ AV, int m, size_t n, DavY y, double theta,
                                                 double* out, double* scratch, unsigned* counter) {
    __shared__ double sh[1][RB];
    __shared__ double tot[1];
    double v[1] = {0.0};
    for (size_t i = blockIdx.x * (size_t)RB + threadIdx.x; i < n; i += (size_t)gridDim.x * RB) {
        double s = 0.0, w = 0.0;
#pragma unroll
        for (int q = 0; q < DAV_MAX; ++q)
            if (q < m) {
                s = fma(y.y[q], V[(size_t)q * n + i], s);
                w = fma(y.y[q], AV[(size_t)q * n + i], w);
            }
        const double r = fma(-theta, s, w);
        x[i] = s;
        ax[i] = w;
        z[i] = r;
        v[0] = fma(r, r, v[0]);
    }
    if (grid_sum<1>(v, 1, sh, tot, scratch, counter) && threadIdx.x == 0) *out = tot[0];
}

inline int ew_grid(size_t n) {
    size_t g = (n + 255) / 256;
    if (g < 1) g = 1;
    if (g > 152 * 8) g = 152 * 8;
    return (int)g;
}

}  // namespace

long long launch_count() { return g_launches.load(); }
void count_launch() { counted(); }
long long launch_count_thread() { return t_launches; }
void uncount_launches(long long n) {
    g_launches.fetch_sub(n);
    t_launches -= n;
}

void ensure_smem_attr(const void* func, int bytes) {
    static std::mutex mu;
    static std::set<std::pair<const void*, int>> done;
    thread_local std::set<std::pair<const void*, int>> seen;   // lock-free fast path per thread
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    if (seen.count({func, dev})) return;
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count({func, dev})) {
        if (cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return;
        done.insert({func, dev});
    }
    seen.insert({func, dev});
}

namespace {
// Resident CTAs of a kernel on the current device (occupancy x SMs), cached
// per (kernel, device).
int resident_ctas(const void* func, int threads, size_t smem) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> cache;
    thread_local std::map<std::pair<const void*, int>, int> mine;   // lock-free fast path per thread
    int dev = 0;
    cudaGetDevice(&dev);
    auto f = mine.find({func, dev});
    if (f != mine.end()) return f->second;
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find({func, dev});
    if (it != cache.end()) return mine[{func, dev}] = it->second;
    int nb = 1, sms = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, func, threads, smem) != cudaSuccess || nb < 1) nb = 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
    cudaGetLastError();
    return mine[{func, dev}] = cache[{func, dev}] = nb * sms;
}

template <int TM, int TN>
void launch_tile(const GemmTask* tasks, int ntask, const GemmOp* ops, cudaStream_t st, const int* skip) {
    auto* f = k_gemm<TM, TN>;
    const int grid = std::min(ntask, resident_ctas(reinterpret_cast<const void*>(f), NT, 0));
    counted();
    f<<<grid, NT, 0, st>>>(tasks, ntask, ops, skip);
}
}  // namespace

bool gemm_tile_supported(int tm, int tn) {
    return (tm == 64 && tn == 64) || (tm == 32 && tn == 64) || (tm == 64 && tn == 32) || (tm == 16 && tn == 128) ||
           (tm == 32 && tn == 32);
}

void launch_splitk_reduce(const SplitRed* tasks, int ntask, cudaStream_t st, const int* skip) {
    if (ntask > 0) { counted(); k_splitk_reduce<<<dim3(ntask, 8), 128, 0, st>>>(tasks, skip); }
}

void launch_gemm_tile(int tm, int tn, const GemmTask* tasks, int ntask, const GemmOp* ops, cudaStream_t st,
                      const int* skip) {
    if (ntask <= 0) return;
#define MPSPT_TILE(A, B)                                    \
    if (tm == A && tn == B) {                               \
        launch_tile<A, B>(tasks, ntask, ops, st, skip);     \
        return;                                             \
    }
    MPSPT_TILE(64, 64)
    MPSPT_TILE(32, 64)
    MPSPT_TILE(64, 32)
    MPSPT_TILE(16, 128)
    MPSPT_TILE(32, 32)
#undef MPSPT_TILE
}

void launch_mix(const MixTask* tasks, int ntask, const MixSrc* srcs, cudaStream_t st, const int* skip) {
    if (ntask > 0) { counted(); k_mix<<<ntask, 128, 0, st>>>(tasks, srcs, skip); }
}

void launch_mix_pieces(const MixTask* tasks, const unsigned* piece_task, int npiece, const MixSrc* srcs,
                       cudaStream_t st, const int* skip) {
    if (npiece > 0) { counted(); k_mix_pieces<<<(npiece + 3) / 4, 128, 0, st>>>(tasks, piece_task, npiece, srcs, skip); }
}

void launch_diag(const DiagTask* tasks, int ntask, const DiagTerm* terms, cudaStream_t st) {
    if (ntask > 0) { counted(); k_diag<<<ntask, 256, 0, st>>>(tasks, terms); }
}
void launch_copy(const CopyTask* tasks, int ntask, cudaStream_t st) {
    if (ntask > 0) { counted(); k_copy<<<ntask, 256, 0, st>>>(tasks); }
}
void vec_scale_mask(double* y, const double* x, double a, size_t n, cudaStream_t st) {
    if (n) { counted(); k_scale<<<ew_grid(n), 256, 0, st>>>(y, x, a, n); }
}
void vec_axpy(double* y, const double* x, double a, size_t n, cudaStream_t st) {
    if (n) { counted(); k_axpy<<<ew_grid(n), 256, 0, st>>>(y, x, a, n); }
}
void vec_dot(const double* x, const double* y, size_t n, double* out, double* scratch,
             unsigned* counter, cudaStream_t st) {
    counted(); k_dot<<<red_grid(n), RB, 0, st>>>(x, y, n, out, scratch, counter);
}
namespace {
inline int dav_grid(size_t n) {   // scratch: DAV_MAX sums of at most 228 blocks
    return std::min(red_grid(n), 228);
}
}  // namespace
void dav_correct(double* t, const double* r, const double* diag, double theta, const double* V, int m, size_t n,
                 double* coef, double* scratch, unsigned* counter, cudaStream_t st) {
    counted(); k_dav_pass<0><<<dav_grid(n), RB, 0, st>>>(t, V, m, n, r, diag, theta, nullptr, coef, scratch, counter);
}
void dav_project(double* t, const double* V, int m, size_t n, const double* coef, double* next, bool last,
                 double* scratch, unsigned* counter, cudaStream_t st) {
    counted();
    if (last) k_dav_pass<2><<<dav_grid(n), RB, 0, st>>>(t, V, m, n, nullptr, nullptr, 0.0, coef, next, scratch, counter);
    else k_dav_pass<1><<<dav_grid(n), RB, 0, st>>>(t, V, m, n, nullptr, nullptr, 0.0, coef, next, scratch, counter);
}
void dav_unit(double* t, double* p, const double* norm2, size_t n, cudaStream_t st) {
    counted(); k_dav_unit<<<ew_grid(n), 256, 0, st>>>(t, p, norm2, n);
}
void dav_column(double* av, const double* ap, const double* V, int m, size_t n, double* h, double* scratch,
                unsigned* counter, cudaStream_t st) {
    counted(); k_dav_pass<3><<<dav_grid(n), RB, 0, st>>>(av, V, m, n, ap, nullptr, 0.0, nullptr, h, scratch, counter);
}
void dav_ritz(double* x, double* ax, double* z, const double* V, const double* AV, int m, size_t n, const double* y,
              double theta, double* out, double* scratch, unsigned* counter, cudaStream_t st) {
    DavY yy{};
    for (int q = 0; q < m; ++q) yy.y[q] = y[q];
    counted(); k_dav_ritz<<<red_grid(n), RB, 0, st>>>(x, ax, z, V, AV, m, n, yy, theta, out, scratch, counter);
}
void make_minv(double* minv, const double* diag, size_t n, cudaStream_t st) {
    if (n) { counted(); k_minv<<<ew_grid(n), 256, 0, st>>>(minv, diag, n); }
}
void cg_init(double* r, double* z, double* p, const double* b, const double* Ax,
             const double* minv, size_t n, CgState* S, double tol, double* scratch,
             unsigned* counter, cudaStream_t st) {
    counted(); k_cg_init<<<red_grid(n), RB, 0, st>>>(r, z, p, b, Ax, minv, n, S, tol, scratch, counter);
}
void cg_step(double* x, double* r, double* z, double* p, const double* Ap, const double* minv,
             size_t n, CgState* S, double* scratch, unsigned* counter, cudaStream_t st) {
    counted(); k_cg_pap<<<red_grid(n), RB, 0, st>>>(p, Ap, n, S, scratch, counter);
    counted(); k_cg_update<<<red_grid(n), RB, 0, st>>>(x, r, z, p, Ap, minv, n, S, scratch, counter);
    counted(); k_cg_dir<<<ew_grid(n), 256, 0, st>>>(p, z, n, S);
}

}  // namespace mpspt
