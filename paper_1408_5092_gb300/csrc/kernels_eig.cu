// Batched cyclic Jacobi for the density-matrix eigenproblems of the truncation
// step.
//
// The float64 pipe of this GPU (1.75 FMA per clock and SM, 64 clocks of
// latency) is the scarce unit, so the default solver keeps the O(n^3) work of
// the sweeps in float32 and corrects it by float64 GEMMs on all SMs (eig.cpp):
//
// k_jac_mixed (one CTA per matrix): all sweeps of a phase in one launch.  The
// off-diagonal part is float32, the diagonal float32 in the start and float64
// in the polish, both scaled by a power of two.  In a round of the round-robin ordering the m/2 disjoint
// pairs get their rotations, then every 2 x 2 block of slots (k, l) is
// transformed.  Entries are addressed by slot position, not by index: a round
// reads each block from the same four places of one buffer and writes it to
// the four places of the next round's positions in the other, so a thread's
// addresses are computed once per launch and kept in registers.  The update
// moves 32 bytes of shared memory per block, 940 clocks a round at n = 173;
// the pair phase and two barriers are the rest.
// k_jac_rot64: the float64 rotations (jac_rot.h) of the recorded float32 tangents.
// k_jac_apply (a warp per row of V): V <- V R over the recorded lists; a row
// is touched independently of the others, the rotations of a round act on
// disjoint columns and take one lane each.
//
// Measured (device time of the truncations of one M = 256 sweep of 8e/8o + 24,
// sectors up to n = 173): sweeps 240 -> 47 ms, V 159 -> 25 ms against one
// launch per sweep with float64 polish sweeps and 32 rows of V per CTA; a
// batch of ten sectors (173 and down by 0.8) 29.8 -> 6.0 ms a call.  Above n = 236
// (triangles in global memory): n = 260 102 -> 61 ms, 346 369 -> 148, 500 972 ->
// 455, sixteen of 300 183 -> 146.
//
// k_eig_one / k_eig_cl: the plain float64 solver (float64 sweeps from the
// identity), all sweeps in one launch, V included.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "eig_route.h"
#include "jac_lists.h"
#include "jac_rot.h"
#include "jac_tol.h"
#include "jacobi_schedule.h"
#include "kernels.h"

namespace mpspt {
namespace {

constexpr int JAC_SMEM = 200704;     // dynamic shared memory of the float64 solver and of the apply kernel

// Scale of a matrix with an infinity or a NaN (largest exponent 2047).  Such a
// matrix has no eigenvalues, and float32 norms of scaled entries cannot show it
// (an entry 2^-1025 of its value is zero), so it is told by the exponent: flag
// 2 and w (from the float64 solver V too) filled with NaN.
constexpr int kNonFinite = 0x7FF - 1022;

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

// ---------------------------------------------------------------- mixed
constexpr int MIX_SMEM = 230000;
// Shared memory of the mixed kernel: two triangle buffers of `cap` floats at
// fixed offsets (so that a buffer is an immediate offset), then two diagonals,
// (c, s) and (tan, e).  cap of the variants with NB cached blocks per thread:
__host__ __device__ constexpr int mixed_cap(int nb) { return nb <= 2 ? 1040 : nb <= 5 ? 4192 : nb <= 8 ? 16112 : 27736; }
inline size_t mixed_smem(int n, int cap) {
    const size_t m = n + (n & 1);
    return 8 * (size_t)cap + 24 * m + 16;
}

// NT threads, NB blocks per thread with cached addresses (0: any n, triangles
// in global memory, addresses computed).
// The start keeps its diagonal in float32 as well (its V is corrected to
// float64 later): the chain of the pair phase is then 400 clocks instead of
// 1000, a float64 operation being 64.  In the polish the float64 diagonal is
// updated beside the blocks, by the last warps.
template <int NT, int NB, bool POLISH>
__global__ void __launch_bounds__(NT) k_jac_mixed(const JacTask* __restrict__ tasks) {
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int NW = NT / 32, NC = NB > 0 ? NB : 1;
    __shared__ double red[2][NW];
    __shared__ unsigned redm[NW];
    __shared__ int stop, shift;
    __shared__ double sa_sh;
    const JacTask t = tasks[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (POLISH && *(volatile const int*)t.done) {
        if (tid == 0) *t.nsw = 0;
        return;
    }
    const int n = t.n, m = n + (n & 1), half = m / 2, rounds = m - 1;
    const int np = m * (m - 1) / 2, nblk = half * (half - 1) / 2;
    constexpr int CAP = NB > 0 ? mixed_cap(NB) : 0;
    float* E = NB > 0 ? reinterpret_cast<float*>(sm) : static_cast<float*>(t.P);
    unsigned char* rest = sm + (size_t)8 * CAP;
    const int half2 = NB > 0 ? CAP : np;   // the second buffer
    using DT = std::conditional_t<POLISH, double, float>;
    DT* D = reinterpret_cast<DT*>(rest);              // two of m
    float2* cs = reinterpret_cast<float2*>(rest + 16 * (size_t)m);
    float2* te = cs + half;                            // (tan, e) of the round's pairs
    // scale: the exponent of the largest |a_ij| (over the float64 bits)
    {
        unsigned mx = 0;
        for (int i = warp; i < n; i += NW)
            for (int j = i + lane; j < n; j += 32) mx = max(mx, (unsigned)dexp(t.A[(size_t)i * n + j]));
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) redm[warp] = mx;
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < NW; ++w) mx = max(mx, redm[w]);
            shift = mx == 0 ? 0 : (int)mx - 1022;   // largest entry in [1/2, 1)
        }
        __syncthreads();
    }
    const int sh = shift;
    if (sh == kNonFinite) {   // no rotation in the start, so that B is not finite either and the polish says so
        if (tid == 0) {
            *t.nsw = 0;
            if (!POLISH) t.total[0] = t.total[1] = 0;
            *t.done = POLISH ? 2 : 0;
        }
        if (t.w)
            for (int i = tid; i < n; i += NT) t.w[i] = nan("");
        return;
    }
    for (int e = tid; e < np; e += NT) E[e] = 0.f;
    for (int e = tid; e < m; e += NT) D[e] = DT(0);
    __syncthreads();
    for (int i = warp; i < n; i += NW)
        for (int j = i + lane; j < n; j += 32) {
            const double a = t.A[(size_t)i * n + j];
            if (j == i) {
                if constexpr (POLISH) D[i] = ldexp(a, -sh);
                else D[i] = d2f_scaled(a, sh);
            }
            else E[tri(m, i, j)] = d2f_scaled(a, POLISH ? sh + 1 : sh);
        }
    // B's two halves are rounded independently: their mean is nearer (vectors'
    // errors 0.73 of one half's at n = 8, 0.75 at 128)
    if constexpr (POLISH) {
        __syncthreads();
        for (int i = warp; i < n; i += NW)
            for (int j = lane; j < i; j += 32) E[tri(m, j, i)] += d2f_scaled(t.A[(size_t)i * n + j], sh + 1);
    }
    // places of this thread's pair and blocks in a buffer (16 bits each)
    int kl[NC];
    unsigned rd[2][NC], wr[2][NC];
    int pr = 0, pw = 0, pk = 0, pkb = 0;
    if (NB > 0) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const int e = tid + i * NT;
            kl[i] = rd[0][i] = rd[1][i] = wr[0][i] = wr[1][i] = 0;
            if (e < nblk) {
                int k, l;
                block_slots(half, e, k, l);
                const int kb = m - 1 - k, lb = m - 1 - l;
                kl[i] = k | (l << 16);
                rd[0][i] = (unsigned)tri(m, k, l) | ((unsigned)tri(m, k, lb) << 16);
                rd[1][i] = (unsigned)tri(m, l, kb) | ((unsigned)tri(m, lb, kb) << 16);
                wr[0][i] = (unsigned)tri_next(m, k, l) | ((unsigned)tri_next(m, k, lb) << 16);
                wr[1][i] = (unsigned)tri_next(m, l, kb) | ((unsigned)tri_next(m, lb, kb) << 16);
            }
        }
        if (tid < half) {
            pr = tri(m, tid, m - 1 - tid);
            pw = tri_next(m, tid, m - 1 - tid);
            pk = next_pos(m, tid);
            pkb = next_pos(m, m - 1 - tid);
        }
    }
    __syncthreads();
    float* cur = E;
    float* nxt = E + half2;
    DT* Dc = D;
    DT* Dn = D + m;
    double off0 = 0.0, prev = 1e300;   // thread 0
    float nv = 0.f;
    int s = 0;
    for (;; ++s) {
        // |A|_F^2 and the off-diagonal norm without null pairs
        double dd = 0.0;
        for (int i = tid; i < n; i += NT) dd = fma((double)Dc[i], (double)Dc[i], dd);
        float ee = 0.f;
        for (int i = warp; i < n; i += NW)
            for (int j = i + 1 + lane; j < n; j += 32) {
                const float v = cur[tri(m, i, j)];
                ee = fmaf(v, v, ee);
            }
        double e2 = (double)ee;
        for (int o = 16; o > 0; o >>= 1) {
            dd += __shfl_xor_sync(0xffffffffu, dd, o);
            e2 += __shfl_xor_sync(0xffffffffu, e2, o);
        }
        if (lane == 0) { red[0][warp] = dd; red[1][warp] = e2; }
        __syncthreads();
        if (tid == 0) {
            double a = 0.0, b = 0.0;
            for (int w = 0; w < NW; ++w) { a += red[0][w]; b += red[1][w]; }
            sa_sh = a + 2.0 * b;
            red[0][0] = 2.0 * b;
        }
        __syncthreads();
        const double sa = sa_sh;
        double so = red[0][0];
        if constexpr (POLISH) {   // take the null pairs out
            nv = (float)Tol::null * sqrtf((float)sa);
            float nn = 0.f;
            for (int i = warp; i < n; i += NW)
                if (fabsf(d2f_trunc(Dc[i])) < nv)
                    for (int j = i + 1 + lane; j < n; j += 32) {
                        const float v = cur[tri(m, i, j)];
                        if (fabsf(v) < nv && fabsf(d2f_trunc(Dc[j])) < nv) nn = fmaf(v, v, nn);
                    }
            double n2 = (double)nn;
            for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
            __syncthreads();
            if (lane == 0) red[1][warp] = n2;
            __syncthreads();
            if (tid == 0) {
                double b = 0.0;
                for (int w = 0; w < NW; ++w) b += red[1][w];
                so = so - 2.0 * b < 0.0 ? 0.0 : so - 2.0 * b;
            }
        }
        if (tid == 0) {
            if (s == 0) off0 = so;
            const JacStop q = POLISH ? polish_stop(s, so, sa, off0, prev) : start_stop(so, sa, prev);
            prev = so;
            stop = q.stop || n < 2 || s >= (POLISH ? min(t.cap, kPolishSweeps) : t.cap);
            if (stop) {
                *t.nsw = s;
                if (POLISH) *t.total += s;
                else t.total[0] = s, t.total[1] = 0;
                *t.done = POLISH && (q.done || n < 2) ? 1 : 0;
            }
        }
        __syncthreads();
        if (stop) break;
        float2* list = t.rot + (size_t)s * rounds * half;
        for (int r = 0; r < rounds; ++r) {
            auto pair = [&](int k, int kb, int from, int to, int tok, int tokb) {
                const float e = cur[from];
                const DT dx = Dc[k], dy = Dc[kb];
                float d;
                if constexpr (POLISH) d = d2f_trunc(dy - dx);
                else d = dy - dx;
                bool on = fabsf(e) >= 0x1p-126f;   // (a subnormal entry is left alone)
                if constexpr (POLISH) on = on && !(fabsf(e) < nv && fabsf(d2f_trunc(dx)) < nv && fabsf(d2f_trunc(dy)) < nv);
                const float tn = on ? jac_tan(d, e) : 0.f;
                const float x = fmaf(tn, tn, 1.f);
                float c = rsqrtf(x);
                c = fmaf(0.5f * c, fmaf(-x * c, c, 1.f), c);
                const float sn = tn * c;
                cs[k] = make_float2(c, sn);
                nxt[to] = on ? 0.f : e;
                if constexpr (POLISH) {
                    te[k] = make_float2(tn, e);
                    list[k] = make_float2(tn, 0.f);
                } else {
                    Dn[tok] = fmaf(-tn, e, dx);
                    Dn[tokb] = fmaf(tn, e, dy);
                    list[k] = make_float2(c, sn);
                }
            };
            if (NB > 0) {
                if (tid < half) pair(tid, m - 1 - tid, pr, pw, pk, pkb);
            } else {
                for (int k = tid; k < half; k += NT) {
                    const int kb = m - 1 - k;
                    pair(k, kb, tri(m, k, kb), tri_next(m, k, kb), next_pos(m, k), next_pos(m, kb));
                }
            }
            __syncthreads();
            auto block = [&](int k, int l, int r0, int r1, int r2, int r3, int w0, int w1, int w2, int w3) {
                const float2 a = cs[k], b = cs[l];
                const float kl_ = cur[r0], kL = cur[r1], Kl = cur[r2], KL = cur[r3];
                const float x0 = a.x * kl_ - a.y * Kl, y0 = a.y * kl_ + a.x * Kl;
                const float x1 = a.x * kL - a.y * KL, y1 = a.y * kL + a.x * KL;
                nxt[w0] = b.x * x0 - b.y * x1;
                nxt[w1] = b.y * x0 + b.x * x1;
                nxt[w2] = b.x * y0 - b.y * y1;
                nxt[w3] = b.y * y0 + b.x * y1;
            };
            if (NB > 0) {
#pragma unroll
                for (int i = 0; i < NC; ++i)
                    if (tid + i * NT < nblk)
                        block(kl[i] & 0xffff, kl[i] >> 16, rd[0][i] & 0xffff, rd[0][i] >> 16, rd[1][i] & 0xffff,
                              rd[1][i] >> 16, wr[0][i] & 0xffff, wr[0][i] >> 16, wr[1][i] & 0xffff, wr[1][i] >> 16);
            } else {
                for (int e = tid; e < nblk; e += NT) {
                    int k, l;
                    block_slots(half, e, k, l);
                    const int kb = m - 1 - k, lb = m - 1 - l;
                    block(k, l, tri(m, k, l), tri(m, k, lb), tri(m, l, kb), tri(m, lb, kb), tri_next(m, k, l),
                          tri_next(m, k, lb), tri_next(m, l, kb), tri_next(m, lb, kb));
                }
            }
            if constexpr (POLISH)
                for (int k = NT - 1 - tid; k < half; k += NT) {
                    const double u = f2d_exact(te[k].x) * f2d_exact(te[k].y);
                    Dn[next_pos(m, k)] = Dc[k] - u;
                    Dn[next_pos(m, m - 1 - k)] = Dc[m - 1 - k] + u;
                }
            __syncthreads();
            float* x = cur; cur = nxt; nxt = x;
            DT* d = Dc; Dc = Dn; Dn = d;
            list += half;
        }
    }
    if (t.w)
        for (int i = tid; i < n; i += NT) t.w[i] = ldexp((double)Dc[i], sh);
}

__global__ void k_jac_rot64(const JacTask* __restrict__ tasks) {
    const JacTask t = tasks[blockIdx.y];
    const int m = t.n + (t.n & 1);
    const size_t tot = (size_t)*t.nsw * (m - 1) * (m / 2);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (size_t)gridDim.x * blockDim.x) {
        const float tn = t.rot[i].x;
        double s = (double)tn, h = 0.5 * s;
        if (fabsf(tn) > 1e-9f) {   // below, they round to these
            h = jac_half64(tn, 0.f);
            s = jac_sine64(h);
        }
        t.rot64[i] = make_double2(h, s);
    }
}

// A warp per row of V.  The lane of slot k of a round rotates the row's
// entries of that slot's two columns; the next round's list entries are
// fetched while the present ones are applied.  Float64: four operations per
// rotation and row on the float64 pipe, spread over n / 4 CTAs (32 rows per
// warp, as before, left it on n / 32 SMs).
template <class T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

template <class T>
__global__ void __launch_bounds__(32 * JAC_APPLY_ROWS) k_jac_apply(const JacTask* __restrict__ tasks,
                                                                  const JacRows* __restrict__ rb, int ident) {
    extern __shared__ __align__(16) unsigned char sm[];
    using T2 = typename Vec2<T>::type;
    const JacRows b = rb[blockIdx.x];
    const JacTask t = tasks[b.task];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nsw = *(volatile const int*)t.nsw;
    if (warp >= b.rows || (nsw == 0 && !ident)) return;
    const int n = t.n, m = n + (n & 1), half = m / 2, rounds = m - 1, row = b.r0 + warp;
    T* R = reinterpret_cast<T*>(sm) + (size_t)warp * m;
    double* Vr = t.V + (size_t)row * n;
    for (int j = lane; j < m; j += 32) R[j] = j >= n ? T(0) : ident ? T(j == row ? 1 : 0) : (T)Vr[j];
    __syncwarp();
    const T2* list;
    if constexpr (sizeof(T) == 8) list = t.rot64; else list = t.rot;
    constexpr int PF = 4;   // list entries per lane fetched ahead
    T2 nx[PF];
    const size_t total = (size_t)nsw * rounds;
    auto fetch = [&](size_t g) {
#pragma unroll
        for (int q = 0; q < PF; ++q)
            if (g < total && lane + 32 * q < half) nx[q] = list[g * half + lane + 32 * q];
    };
    auto rotate = [&](int k, int r, T2 cs) {
        if (cs.y == T(0)) return;
        int pa = k - 1 + r, pb = m - 2 - k + r;
        pa = k == 0 ? 0 : (pa >= rounds ? pa - rounds : pa) + 1;
        pb = (pb >= rounds ? pb - rounds : pb) + 1;
        const T x = R[pa], y = R[pb];
        if constexpr (sizeof(T) == 8) {
            R[pa] = rot_first(cs.y, cs.x, x, y);
            R[pb] = rot_second(cs.y, cs.x, x, y);
        } else {
            R[pa] = cs.x * x - cs.y * y;
            R[pb] = cs.y * x + cs.x * y;
        }
    };
    fetch(0);
    int r = 0;
    for (size_t g = 0; g < total; ++g) {
        T2 cs[PF];
#pragma unroll
        for (int q = 0; q < PF; ++q) cs[q] = nx[q];
        fetch(g + 1);
#pragma unroll
        for (int q = 0; q < PF; ++q)
            if (lane + 32 * q < half) rotate(lane + 32 * q, r, cs[q]);
        for (int k = lane + 32 * PF; k < half; k += 32) rotate(k, r, list[g * half + k]);
        __syncwarp();
        if (++r == rounds) r = 0;
    }
    for (int j = lane; j < n; j += 32) Vr[j] = (double)R[j];
}

// -------------------------------------------------------------- float64
// All float64 sweeps of one matrix in one launch, on C CTAs (a cluster of 8,
// or one CTA for small matrices).  The packed upper triangle is spread over
// the CTAs' shared memories (entry e in CTA e mod C, slot e / C; with a_sm
// false it is the upper part of t.A, which is then destroyed), the rows of V
// likewise (row i in CTA i mod C; with v_sm false in t.V).  A round: every CTA
// computes all rotations from the distributed entries; barrier; it transforms
// its share of the 2 x 2 blocks of slots and its rows of V; barrier.  Bound by
// the float64 pipes of the C SMs (4 n^2 operations a round) and, for small n,
// by the chain rotation - barrier - update - barrier.  A float64 instruction
// occupies a sub-partition for 64 clocks however few lanes are active, so what
// counts is their number per warp.  Measured against the one-CTA kernel with
// divisions and square roots: twelve 13 x 13 458 -> 230 us a call, sectors of 90
// and down 20.6 -> 5.5 ms; against the launch-per-sweep cluster form n = 240 531 ->
// 53 ms, 346 1664 -> 153, 500 5007 -> 579.
constexpr int JC = 8;

struct EigFit { size_t head, a, v; };   // shared memory of one CTA: head, triangle share, V rows
__host__ __device__ constexpr EigFit eig_fit(int n, int C) {
    EigFit f{};
    const size_t half = (size_t)(n + 1) / 2;
    // rowoff, slots, (s, h) and the rotated pairs' blocks, the diagonal
    f.head = align16((size_t)n * 4) + align16(half * 8) + align16(half * 40) + align16((size_t)n * 8);
    f.a = align16(((size_t)n * (n + 1) / 2 + C - 1) / C * 8);
    f.v = align16(((size_t)n + C - 1) / C * n * 8);
    return f;
}
__host__ __device__ constexpr bool eig_a_sm(int n, int C) { const EigFit f = eig_fit(n, C); return f.head + f.a <= (size_t)JAC_SMEM; }
__host__ __device__ constexpr bool eig_v_sm(int n, int C) { const EigFit f = eig_fit(n, C); return f.head + f.a + f.v <= (size_t)JAC_SMEM; }
static_assert(eig_a_sm(kEigOneMaxN, 1) && !eig_a_sm(kEigOneMaxN + 5, 1), "largest matrix of one CTA");
inline size_t eig_smem(int n, int C) {
    const EigFit f = eig_fit(n, C);
    return f.head + (eig_a_sm(n, C) ? f.a : 0) + (eig_v_sm(n, C) ? f.v : 0);
}

// h of a pair whose e is below 2^-80 of the largest entry: the Newton steps'
// float32 residuals leave their range there, so by division and square roots.
// Zero where the tangent rounds to zero or e is below 2^-960.
__device__ __noinline__ double jac_half64_tiny(double d, double e) {
    if (abs_below(e, 0x1p-960)) return 0.0;
    const double th = d / (2.0 * e);
    const double t = (th < 0.0 ? -1.0 : 1.0) / (fabs(th) + sqrt(fma(th, th, 1.0)));
    return t / (1.0 + sqrt(fma(t, t, 1.0)));
}

template <int C, int NT, bool A_SM>
__device__ __forceinline__ void eig_body(const EigTask& t, double nullrel, int maxs, int* flag, int rank) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int NW = NT / 32, NBC = 4;
    __shared__ float red[2][NW];
    __shared__ float part[2][C];
    const int n = t.n, m = n + (n & 1), half = m / 2, rounds = m - 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool v_sm = A_SM && eig_v_sm(n, C);
    const EigFit fit = eig_fit(n, C);
    int* rowoff = reinterpret_cast<int*>(sm);
    int2* slots = reinterpret_cast<int2*>(sm + align16((size_t)n * 4));   // (p, q); q < 0: not rotated
    double* Ss = reinterpret_cast<double*>(sm + align16((size_t)n * 4) + align16((size_t)half * 8));
    double *Hh = Ss + half, *Xa = Hh + half, *Xe = Xa + half, *Xb = Xe + half;
    double* dg = reinterpret_cast<double*>(sm + align16((size_t)n * 4) + align16((size_t)half * 8) +
                                           align16((size_t)half * 40));
    double* Ploc = reinterpret_cast<double*>(sm + fit.head);
    const int nrow = (n - rank + C - 1) / C;          // this CTA's rows of V
    double* Vl = v_sm ? reinterpret_cast<double*>(sm + fit.head + fit.a) : t.V + (size_t)rank * n;
    const size_t vld = v_sm ? n : (size_t)C * n;
    auto sync = [&] {
        if constexpr (C > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    auto at = [&](int a, int b) -> double& {   // any order
        const int e = rowoff[min(a, b)] + max(a, b);
        if constexpr (!A_SM) return t.A[e];
        else if constexpr (C > 1) return cg::this_cluster().map_shared_rank(Ploc, e % C)[e / C];
        else return Ploc[e];
    };
    // scaled by a power of two so that the largest entry is in [1/2, 1)
    unsigned mx = 0;
    for (int i = warp; i < n; i += NW)
        for (int j = i + lane; j < n; j += 32) mx = max(mx, (unsigned)dexp(t.A[(size_t)i * n + j]));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) red[0][warp] = __uint_as_float(mx);
    for (int i = tid; i < n; i += NT) rowoff[i] = A_SM ? i * n - i * (i + 1) / 2 : i * n;
    sync();   // (in place: nobody scales an entry before all have looked)
    for (int w = 0; w < NW; ++w) mx = max(mx, __float_as_uint(red[0][w]));
    const int sh = mx == 0 ? 0 : (int)mx - 1022;
    if (sh == kNonFinite) {   // the same in every CTA
        for (int i = rank * NT + tid; i < n; i += C * NT) t.w[i] = nan("");
        for (size_t e = (size_t)rank * NT + tid; e < (size_t)n * n; e += (size_t)C * NT) t.V[e] = nan("");
        if (flag && rank == 0 && tid == 0) *flag = 2;
        return;
    }
    for (int i = warp; i < n; i += NW)
        for (int j = i + lane; j < n; j += 32) {
            const int e = rowoff[i] + j;
            if (A_SM ? e % C != rank : i % C != rank) continue;
            const double v = ldexp(t.A[(size_t)i * n + j], -sh);
            if (A_SM) Ploc[e / C] = v;
            else t.A[e] = v;
        }
    for (int i = warp; i < nrow; i += NW)
        for (int j = lane; j < n; j += 32) Vl[i * vld + j] = j == rank + i * C ? 1.0 : 0.0;
    // this thread's first blocks (all of them up to n = 256 on a cluster)
    const int nblk = half * (half - 1) / 2;
    int bk[NBC];
#pragma unroll
    for (int i = 0; i < NBC; ++i) {
        const int blk = rank + C * (tid + i * NT);
        int k = 0, l = 0;
        if (blk < nblk) block_slots(half, blk, k, l);
        bk[i] = k | (l << 16);
    }
    int ek = 0, el = 0;   // this thread's block when every entry has a thread
    if (C == 1 && 4 * nblk <= NT && tid < 4 * nblk) block_slots(half, tid >> 2, ek, el);
    const unsigned hinv = 0xFFFFFFFFu / (unsigned)half + 1u;   // e / half = umulhi(e, hinv) for e < 2^20
    sync();   // every CTA of the cluster is running and has its share before any remote access
    double nullv = 0.0;
    float prev = 3e38f;
    for (int sweep = 0;; ++sweep) {
        // off-norm without null pairs, and |A|_F^2, in float32 (they decide
        // when to stop, to no more than a few digits); the partial sums of all
        // CTAs are added in rank order by everyone
        for (int i = tid; i < n; i += NT) dg[i] = at(i, i);
        __syncthreads();
        float off = 0.f, all = 0.f;
        for (int i = warp; i < n; i += NW)
            for (int j = i + lane; j < n; j += 32) {
                if (A_SM ? (rowoff[i] + j) % C != rank : i % C != rank) continue;
                const double v = at(i, j);
                const float f = d2f_trunc(v);
                if (j == i) all = fmaf(f, f, all);
                else if (abs_below(v, nullv) && abs_below(dg[i], nullv) && abs_below(dg[j], nullv))
                    all = fmaf(2.f * f, f, all);
                else off = fmaf(2.f * f, f, off);
            }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        if (lane == 0) { red[0][warp] = off; red[1][warp] = all; }
        __syncthreads();
        if (tid < 2 * C) {
            const int which = tid & 1, to = tid >> 1;
            float y = 0.f;
            for (int w = 0; w < NW; ++w) y += red[which][w];
            float* p = &part[which][rank];
            if constexpr (C > 1) p = cg::this_cluster().map_shared_rank(p, to);
            *p = y;
        }
        sync();
        float so = 0.f, sd = 0.f;
        for (int r = 0; r < C; ++r) { so += part[0][r]; sd += part[1][r]; }
        const float sa = so + sd;
        if (sweep == 0) nullv = nullrel * (double)sqrtf(sa);   // the first test counts every pair
        const bool conv = so <= (float)Tol::stop * sa || sa == 0.f || (so <= (float)Tol::stall * sa && so > 0.81f * prev) || n < 2;
        prev = so;
        if (conv || sweep >= maxs) {
            if (flag && rank == 0 && tid == 0) *flag = conv ? 1 : 2;
            break;
        }
        for (int r = 0; r < rounds; ++r) {
            for (int k = tid; k < half; k += NT) {
                int x = k - 1 + r, y = m - 2 - k + r;
                x = k == 0 ? 0 : (x >= rounds ? x - rounds : x) + 1;
                y = (y >= rounds ? y - rounds : y) + 1;
                const int p = min(x, y), q = max(x, y);
                bool on = q < n;
                if (on) {
                    const double a = at(p, p), e = at(p, q), b = at(q, q);
                    const float fd = d2f_trunc(b - a), fe = d2f_trunc(e);
                    on = !is_zero(e) && !jac_negligible(e, a, b) &&
                         !(abs_below(e, nullv) && abs_below(a, nullv) && abs_below(b, nullv));
                    double h = 0.0;
                    if (on && fabsf(fe) >= 0x1p-80f) {
                        const float tn = jac_tan(fd, fe);
                        h = jac_half64(tn, jac_newton(b - a, e, fd, fe, tn));
                    } else if (on) {
                        h = jac_half64_tiny(b - a, e);
                        on = !is_zero(h);
                    }
                    if (on) {
                        Hh[k] = h;
                        Ss[k] = jac_sine64(h);
                        Xa[k] = a; Xe[k] = e; Xb[k] = b;
                    }
                }
                if (!on) { Ss[k] = 0.0; Hh[k] = 0.0; }
                slots[k] = make_int2(p | (on ? 1 << 16 : 0), q < n ? q : -1);
            }
            sync();   // every CTA has read the pair entries before any is updated
            auto block = [&](int k, int l) {
                const int2 sk_ = slots[k], sl_ = slots[l];
                if (((sk_.x | sl_.x) >> 16) == 0) return;
                const double sk = Ss[k], hk = Hh[k], sl = Ss[l], hl = Hh[l];
                const int p = sk_.x & 0xffff, q = sk_.y, u = sl_.x & 0xffff, v = sl_.y;
                const bool hq = q >= 0, hv = v >= 0;
                // a missing partner (odd n) reads the pair's own entry with s = 0
                double& pu = at(p, u);
                double& pv = at(p, hv ? v : u);
                double& qu = at(hq ? q : p, u);
                double& qv = at(hq ? q : p, hv ? v : u);
                const double a_pu = pu, a_pv = pv, a_qu = qu, a_qv = qv;
                const double r_pu = rot_first(sk, hk, a_pu, a_qu), r_qu = rot_second(sk, hk, a_pu, a_qu);
                const double r_pv = rot_first(sk, hk, a_pv, a_qv), r_qv = rot_second(sk, hk, a_pv, a_qv);
                if (hq && hv) qv = rot_second(sl, hl, r_qu, r_qv);
                if (hq) qu = rot_first(sl, hl, r_qu, r_qv);
                if (hv) pv = rot_second(sl, hl, r_pu, r_pv);
                pu = rot_first(sl, hl, r_pu, r_pv);
            };
            if (C == 1 && 4 * nblk <= NT) {
                // few blocks: a thread per entry (six operations instead of
                // sixteen; a float64 instruction takes a warp's sub-partition
                // 64 clocks however few lanes it has)
                double out = 0.0;
                double* dst = nullptr;
                if (tid < 4 * nblk) {
                    const int2 sk_ = slots[ek], sl_ = slots[el];
                    const int p = sk_.x & 0xffff, q = sk_.y, u = sl_.x & 0xffff, v = sl_.y;
                    const bool lo = tid & 1, ro = tid & 2;
                    if ((!lo || q >= 0) && (!ro || v >= 0) && ((sk_.x | sl_.x) >> 16)) {
                        const double sk = lo ? Ss[ek] : -Ss[ek], hk = lo ? -Hh[ek] : Hh[ek];
                        const double sl = ro ? Ss[el] : -Ss[el], hl = ro ? -Hh[el] : Hh[el];
                        const int q_ = q >= 0 ? q : p, v_ = v >= 0 ? v : u;
                        const int p1 = lo ? q_ : p, p2 = lo ? p : q_;   // the entry's own row and the other
                        const double xu = at(p1, u), xv = at(p1, v_), yu = at(p2, u), yv = at(p2, v_);
                        const double ru = fma(sk, fma(hk, xu, yu), xu), rv = fma(sk, fma(hk, xv, yv), xv);
                        const double own = ro ? rv : ru, other = ro ? ru : rv;
                        out = fma(sl, fma(hl, own, other), own);
                        dst = &at(lo ? q : p, ro ? v : u);
                    }
                }
                __syncwarp();   // the four lanes of a block have read it
                if (dst) *dst = out;
            } else
#pragma unroll
                for (int i = 0; i < NBC; ++i)
                    if (rank + C * (tid + i * NT) < nblk) block(bk[i] & 0xffff, bk[i] >> 16);
            for (int blk = rank + C * (tid + NBC * NT); blk < nblk; blk += C * NT) {
                int k, l;
                block_slots(half, blk, k, l);
                block(k, l);
            }
            for (int k = NT - 1 - tid; k < half; k += NT)
                if (k % C == rank && (slots[k].x >> 16)) {   // the rotated pairs' own blocks
                    const int p = slots[k].x & 0xffff, q = slots[k].y;
                    double a = Xa[k], e = Xe[k], b = Xb[k];
                    jac_block64(Ss[k], Hh[k], a, e, b);
                    at(p, p) = a;
                    at(p, q) = e;
                    at(q, q) = b;
                }
            for (int e = tid; e < nrow * half; e += NT) {
                const int i = half > 1 && nrow * half < (1 << 20) ? (int)__umulhi((unsigned)e, hinv) : e / half, k = e - i * half;
                const int2 sk_ = slots[k];
                if (!(sk_.x >> 16)) continue;
                const double s = Ss[k], h = Hh[k];
                double* v = Vl + i * vld;
                const double x = v[sk_.x & 0xffff], y = v[sk_.y];
                v[sk_.x & 0xffff] = rot_first(s, h, x, y);
                v[sk_.y] = rot_second(s, h, x, y);
            }
            sync();   // updates visible to every CTA before the next pair phase
        }
    }
    // the diagonal was gathered by the last test
    for (int i = rank + C * tid; i < n; i += C * NT) t.w[i] = ldexp(dg[i], sh);
    if (v_sm)
        for (int i = warp; i < nrow; i += NW)
            for (int j = lane; j < n; j += 32) t.V[(size_t)(rank + i * C) * n + j] = Vl[(size_t)i * n + j];
    if constexpr (C > 1) cg::this_cluster().sync();   // no CTA leaves while its shared memory may be read
}

template <int NT>
__global__ void __launch_bounds__(NT) k_eig_one(const EigTask* __restrict__ tasks, double nullrel, int maxs, int* flags) {
    eig_body<1, NT, true>(tasks[blockIdx.x], nullrel, maxs, flags ? flags + blockIdx.x : nullptr, 0);
}
__global__ void __cluster_dims__(JC, 1, 1) __launch_bounds__(256)
    k_eig_cl(const EigTask* __restrict__ tasks, double nullrel, int maxs, int* flags) {
    const EigTask t = tasks[blockIdx.x / JC];
    int* flag = flags ? flags + blockIdx.x / JC : nullptr;
    const int rank = (int)cooperative_groups::this_cluster().block_rank();
    if (eig_a_sm(t.n, JC)) eig_body<JC, 256, true>(t, nullrel, maxs, flag, rank);
    else eig_body<JC, 256, false>(t, nullrel, maxs, flag, rank);
}

}  // namespace

template <int NT, int NB>
static void launch_mixed(const JacTask* tasks, int ntask, size_t smem, bool polish, cudaStream_t st) {
    count_launch();
    if (polish) {
        ensure_smem_attr(reinterpret_cast<const void*>(k_jac_mixed<NT, NB, true>), MIX_SMEM);
        k_jac_mixed<NT, NB, true><<<ntask, NT, smem, st>>>(tasks);
    } else {
        ensure_smem_attr(reinterpret_cast<const void*>(k_jac_mixed<NT, NB, false>), MIX_SMEM);
        k_jac_mixed<NT, NB, false><<<ntask, NT, smem, st>>>(tasks);
    }
}

// The number of threads follows the largest matrix (half (half - 1) / 2
// blocks): enough that a round's update is a few blocks per thread, few
// enough that its barriers stay cheap (21 clocks at 128 threads, 45 at 512).
// n up to 46: at most 253 blocks; 92: 1035; 180: 4005; 236 (shared memory): 6903.
void launch_jac_mixed(const JacTask* tasks, int ntask, int nmax, bool polish, cudaStream_t st) {
    if (ntask <= 0) return;
    if (nmax <= 46) launch_mixed<128, 2>(tasks, ntask, mixed_smem(nmax, mixed_cap(2)), polish, st);
    else if (nmax <= 92) launch_mixed<256, 5>(tasks, ntask, mixed_smem(nmax, mixed_cap(5)), polish, st);
    else if (nmax <= 180) launch_mixed<512, 8>(tasks, ntask, mixed_smem(nmax, mixed_cap(8)), polish, st);
    else if (nmax <= 236) launch_mixed<512, 14>(tasks, ntask, mixed_smem(nmax, mixed_cap(14)), polish, st);
    else launch_mixed<1024, 0>(tasks, ntask, mixed_smem(nmax, 0), polish, st);
}

void launch_jac_rot64(const JacTask* tasks, int ntask, cudaStream_t st) {
    for (int i = 0; i < ntask; i += 65535) {
        count_launch();
        k_jac_rot64<<<dim3(16, ntask - i < 65535 ? ntask - i : 65535), 256, 0, st>>>(tasks + i);
    }
}

bool eig_in_place(int n) { return !eig_a_sm(n, JC); }

void order_eig_tasks(EigTask* tasks, int ntask) {
    std::stable_sort(tasks, tasks + ntask, [](const EigTask& x, const EigTask& y) { return x.n > y.n; });
}

template <int NT>
static void launch_eig_one(const EigTask* tasks, int ntask, size_t smem, double nullrel, int maxs, int* flags,
                           cudaStream_t st) {
    ensure_smem_attr(reinterpret_cast<const void*>(k_eig_one<NT>), JAC_SMEM);
    k_eig_one<NT><<<ntask, NT, smem, st>>>(tasks, nullrel, maxs, flags);
}

void launch_eig(const EigTask* tasks, const EigTask* host, int ntask, bool null_rule, int maxs, int* flags,
                cudaStream_t st) {
    const double nullrel = null_rule ? Tol::null : 0.0;
    const int mid = eig_mid_threads_of(ntask, [host](int i) { return host[i].n; });
    for (int i = 0, j; i < ntask; i = j) {   // matrices i to j - 1 take the same kernel
        const int nt = eig_threads(host[i].n, mid);
        const int C = nt == 0 ? JC : 1;
        size_t smem = 0;
        for (j = i; j < ntask && eig_threads(host[j].n, mid) == nt; ++j) smem = std::max(smem, eig_smem(host[j].n, C));
        int* fl = flags ? flags + i : nullptr;
        count_launch();
        if (nt == 0) {
            ensure_smem_attr(reinterpret_cast<const void*>(k_eig_cl), JAC_SMEM);
            k_eig_cl<<<(j - i) * JC, 256, smem, st>>>(tasks + i, nullrel, maxs, fl);
        } else if (nt == 512) {
            launch_eig_one<512>(tasks + i, j - i, smem, nullrel, maxs, fl, st);
        } else if (nt == 256) {
            launch_eig_one<256>(tasks + i, j - i, smem, nullrel, maxs, fl, st);
        } else {
            launch_eig_one<128>(tasks + i, j - i, smem, nullrel, maxs, fl, st);
        }
    }
}

void launch_jac_apply(const JacTask* tasks, const JacRows* rows, int nblocks, int nmax, bool f32, bool ident,
                      cudaStream_t st) {
    if (nblocks <= 0) return;
    const size_t smem = (size_t)JAC_APPLY_ROWS * (nmax + (nmax & 1)) * (f32 ? 4 : 8);
    count_launch();
    if (f32) {
        ensure_smem_attr(reinterpret_cast<const void*>(k_jac_apply<float>), JAC_SMEM);
        k_jac_apply<float><<<nblocks, 32 * JAC_APPLY_ROWS, smem, st>>>(tasks, rows, ident ? 1 : 0);
    } else {
        ensure_smem_attr(reinterpret_cast<const void*>(k_jac_apply<double>), JAC_SMEM);
        k_jac_apply<double><<<nblocks, 32 * JAC_APPLY_ROWS, smem, st>>>(tasks, rows, ident ? 1 : 0);
    }
}

}  // namespace mpspt
