// Device kernels of the MPS-PT hot path and their task descriptors.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace mpspt {

// One K-contribution of a grouped block GEMM: C_tile += alpha * op(A) op(B).
// trans bit 0: A is stored k x m (use A^T); bit 1: B is stored n x k (use B^T).
struct GemmOp {
    const double* A;
    const double* B;
    int lda, ldb, k, trans;
    double alpha;
};

// One output tile (rows [r0, r0+TM) x cols [c0, c0+TN) of an m x n block C).
// With cmap set, element (i, j) of the block is stored at
//   C + cmap[2j] + i * cmap[2j+1]          (cmap_rows == 0, per-column map)
//   C + cmap[2i] + j * cmap[2i+1]          (cmap_rows == 1, per-row map)
// which scatters a panel GEMM straight into a block-sparse layout.
struct GemmTask {
    double* C;
    const int* cmap;
    int ldc, m, n;
    int r0, c0;
    int op0, op1;      // range of GemmOp
    int accumulate;    // 1: C += sum, 0: C = sum
    int cmap_rows;
    // split-K: the task sums the positions
    // [kb, ke) of the concatenated K-list of its ops and, with part set,
    // writes its tm x tn partial tile there (dense, row-major) instead of C;
    // a reduction task then adds the partials in order
    double* part;
    int kb, ke;
};
// Sum of the nparts partial tiles at part + q * tm * tn (q ascending) into
// the tile (r0, c0) of C, with the GemmTask addressing (cmap, accumulate).
struct SplitRed {
    const double* part;
    double* C;
    const int* cmap;
    int nparts, tm, tn;
    int ldc, m, n, r0, c0;
    int accumulate, cmap_rows;
};

// One output block of the float64 grouped GEMM (kernels_dgemm.cu): an m x n
// block C = sum of its K-list ops[op0, op1), addressed as GemmTask's.  Its
// units are numbered u0, u0 + 1, ...: tiles row by row, `nt` to a row, the S
// pieces of a tile's K-list together.  The K-list counts q steps of four K
// (each entry rounded up), a piece has qs of them.  With S > 1 the pieces of
// tile t meet at part + part_off + t * S * tile and tick + tick_off + t.
struct GemmBlk {
    double* C;
    const int* cmap;
    size_t part;
    int tick;
    int ldc, m, n;
    int op0, op1;
    int accumulate, cmap_rows;
    int q, qs, S, nt, u0;
    float scale = 1.f, diag = 0.f;   // stored: scale * sum, plus diag where row = column
};

constexpr int GEMM_TM = 64;
constexpr int GEMM_TN = 64;

// dst block (rows x cols, leading dim ldd) = sum_k coef_k * src_k (leading dim lds_k)
struct MixSrc {
    const double* src;
    int lds;
    int pad;
    double coef;
};
// For k_mix_pieces a block's values are cut, row by row, in pieces of MIX_PIECE;
// p0 is the number of its first piece in the launch, piece_task[p] the task of p.
constexpr int MIX_PIECE = 64;
struct MixTask {
    double* dst;
    int rows, cols, ldd;
    int s0, s1;
    int p0;
};

// Jacobi diagonal of A_loc: out[l, r] += sum coef * L[l*(ldL+1)] * R[r*(ldR+1)]
struct DiagTerm {
    const double* L;
    const double* R;
    int ldL, ldR;
    double coef;
};
struct DiagTask {
    double* out;
    int rows, cols;
    int t0, t1;
};

// Symmetric eigenproblem of one dense n x n row-major block, float64 sweeps.
struct EigTask {
    double* A;      // n*n; read only, or destroyed where eig_in_place(n)
    double* V;      // n*n eigenvectors (columns)
    double* w;      // n eigenvalues (unsorted)
    int n;
    int pad;
};
// One matrix of the sweep kernels (kernels_eig.cu).  Rotation lists hold, for
// every sweep of the last launch, m - 1 rounds of m / 2 slots (m = n rounded
// up to even): the rotation of slot k of round r acts on columns (x, y) of
// the round-robin schedule's slot as x' = c x - s y, y' = s x + c y.
struct JacTask {
    const double* A;   // n x n symmetric input, row-major
    double* V;         // n x n eigenvectors (columns), row-major
    double* w;         // n eigenvalues (unsorted), or null
    void* P;           // scratch for n beyond shared memory: the two float32 triangles
    float2* rot;       // mixed sweeps: (c, s), or (tan, 0) in the polish
    double2* rot64;    // float64 (tangent of the half angle, s)
    int* done;         // 1: converged
    int* nsw;          // sweeps in the lists of the last launch
    int* total;        // sweeps of the phase so far: [0] of the start, whose [1] is [0] of the polish
    int n;
    int cap;           // sweeps the lists have room for
};
struct JacRows {       // rows [r0, r0 + rows) of task's V for one apply block
    int task, r0, rows, pad;
};

// Block copy with optional column selection and transpose:
//   trans 0: dst[i*ldd + j] = src[i*lds + col(j)]
//   trans 1: dst[i*ldd + j] = src[j*lds + col(i)]      col(x) = cols ? cols[x] : x
struct CopyTask {
    const double* src;
    double* dst;
    const int* cols;
    int rows, cols_n;   // shape of dst
    int lds, ldd;
    int trans;
    int pad;
};

// CG scalar block living in device memory.
struct CgState {
    double rz, rz_new, pAp, alpha, beta, rr, bb, tol2;
    int done, iters, not_spd, pad;
};

// Number of kernels launched by this library in this process.
long long launch_count();
void count_launch();
long long launch_count_thread();      // launches made by the calling host thread
void uncount_launches(long long n);   // launches that went into a captured graph (this thread's)
// Raises a kernel's dynamic shared-memory limit to `bytes` on the current
// device.  The attribute belongs to the device's context, so it is set once
// per (kernel, device); thread-safe.  A failure is not remembered: the
// launch that follows then fails and its error check reports it.
void ensure_smem_attr(const void* func, int bytes);

// Split-bfloat16 tcgen05 variant of the grouped GEMM (tiles 128 x 64; same
// task format); f16: split-float16 terms instead.  *err is set to 1 if a
// bounded mbarrier wait gave up.
int tc_tile_m();
int tc_tile_n();
void launch_gemm_tc(const GemmTask* tasks, int ntask, const GemmOp* ops, int* err, cudaStream_t st,
                    const int* skip = nullptr, bool f16 = false);
// Float64 grouped GEMM over the units of a block list (see GemmBlk), output
// tile 16 x 16 or 32 x 32; unit_blk[u] is the block of unit u.  part holds the
// partial tiles and tick one zeroed counter per split tile (left at zero).
void launch_dgemm(int tile, const GemmBlk* blks, const unsigned* unit_blk, int nunit, const GemmOp* ops, double* part,
                  unsigned* tick, cudaStream_t st, const int* skip = nullptr);
// A grouped GEMM's device lists, 16 x 16 units (see launch_dgemm).
struct GemmRun {
    const GemmBlk* blk;
    const unsigned* unit;
    const GemmOp* ops;
    double* part;
    unsigned* tick;
    int nunit;
};
// One CG solve (state after cg_init in *S): the operator as g1, operator sums,
// g2 from p to Ap, the vectors of n, at most maxit iterations.
struct CgArgs {
    GemmRun g1, g2;
    const MixTask* mt;
    const MixSrc* ms;
    int nmix, maxit;
    double *x, *r, *z, *p;
    const double *Ap, *minv;
    size_t n;
    CgState* S;
};
// The whole solve in one launch on one cluster; false: not available here, or
// the launch was refused (nothing runs).
bool launch_cg_cluster(const CgArgs& a, cudaStream_t st);
bool cg_cluster_available();
// Float32 arithmetic on float64 data: grouped GEMM with output tile tm x tn
// (64x64, 32x64, 64x32, 16x128, 32x32).  Persistent: at most the resident
// CTAs are launched and each walks a stride of the task list.
bool gemm_tile_supported(int tm, int tn);
void launch_splitk_reduce(const SplitRed* tasks, int ntask, cudaStream_t st, const int* skip = nullptr);
void launch_gemm_tile(int tm, int tn, const GemmTask* tasks, int ntask, const GemmOp* ops, cudaStream_t st,
                      const int* skip = nullptr);
void launch_mix(const MixTask* tasks, int ntask, const MixSrc* srcs, cudaStream_t st, const int* skip = nullptr);
void launch_mix_pieces(const MixTask* tasks, const unsigned* piece_task, int npiece, const MixSrc* srcs,
                       cudaStream_t st, const int* skip = nullptr);
void launch_diag(const DiagTask* tasks, int ntask, const DiagTerm* terms, cudaStream_t st);
// Float64 Jacobi of every matrix, at most maxs sweeps.  host: the same task
// list on the host, in the order of order_eig_tasks (largest first, so that
// each kernel gets one launch; which kernel: eig_route.h).  null_rule: pairs below
// 1e-14 |A|_F are left alone; flags (nullable): 1 converged, 2 stopped by the
// cap.
void order_eig_tasks(EigTask* tasks, int ntask);
void launch_eig(const EigTask* tasks, const EigTask* host, int ntask, bool null_rule, int maxs, int* flags,
                cudaStream_t st);
bool eig_in_place(int n);
// The solver reads A while it writes V and w: a call whose outputs overlap its
// input (V = A) needs a work copy of it.  tot: sum of n^2, totw: sum of n.
inline bool eig_overlap(const double* A, const double* V, const double* w, size_t tot, size_t totw) {
    return (V < A + tot && A < V + tot) || (w < A + tot && A < w + totw);
}
constexpr int kEighSweeps = 40;   // sweep cap of the calls that report no flags
// Mixed sweeps (float32 off-diagonal, float64 diagonal) of every matrix, up
// to its cap in the launch; polish: see k_jac_mixed.  nmax: the largest n.
void launch_jac_mixed(const JacTask* tasks, int ntask, int nmax, bool polish, cudaStream_t st);
// rot64 <- the float64 rotations of the tangents in rot
void launch_jac_rot64(const JacTask* tasks, int ntask, cudaStream_t st);
// V <- V R over the lists (ident: V starts as the identity)
constexpr int JAC_APPLY_ROWS = 4;
void launch_jac_apply(const JacTask* tasks, const JacRows* rows, int nblocks, int nmax, bool f32, bool ident,
                      cudaStream_t st);
void launch_copy(const CopyTask* tasks, int ntask, cudaStream_t st);

// Vector kernels (n doubles).  Reductions are deterministic (fixed order).
void vec_scale_mask(double* y, const double* x, double a, size_t n, cudaStream_t st);  // y = a*x
void vec_axpy(double* y, const double* x, double a, size_t n, cudaStream_t st);       // y += a*x
// out[slot] = x.y  (partial sums in scratch: 4096 doubles, for all of these)
void vec_dot(const double* x, const double* y, size_t n, double* out, double* scratch,
             unsigned* counter, cudaStream_t st);

// Preconditioned CG building blocks on device scalars.
// r = b - Ax ; z = Minv r ; p = z ; rz = r.z ; rr = r.r ; bb = b.b
void cg_init(double* r, double* z, double* p, const double* b, const double* Ax,
             const double* minv, size_t n, CgState* S, double tol, double* scratch,
             unsigned* counter, cudaStream_t st);
// pAp = p.Ap ; alpha = rz / pAp ; x += alpha p ; r -= alpha Ap ; z = Minv r ;
// rz_new = r.z ; rr = r.r ; done if rr <= tol2 bb ; p = z + (rz_new/rz) p
void cg_step(double* x, double* r, double* z, double* p, const double* Ap, const double* minv,
             size_t n, CgState* S, double* scratch, unsigned* counter, cudaStream_t st);
void make_minv(double* minv, const double* diag, size_t n, cudaStream_t st);
// Davidson passes over a basis V (and AV) of m <= 16 vectors of n:
//  dav_correct: t = r / (theta - diag), denominators kept away from zero, and coef[q] = V_q . t
//  dav_project: t -= sum coef[q] V_q, and next[q] = V_q . t (last: next[0] = t . t)
//  dav_unit:    p = t = t / sqrt(*norm2)
//  dav_column:  av = ap and h[q] = V_q . av
//  dav_ritz:    x = sum y_q V_q, ax = sum y_q AV_q, z = ax - theta x, *out = z . z
void dav_correct(double* t, const double* r, const double* diag, double theta, const double* V, int m, size_t n,
                 double* coef, double* scratch, unsigned* counter, cudaStream_t st);
void dav_project(double* t, const double* V, int m, size_t n, const double* coef, double* next, bool last,
                 double* scratch, unsigned* counter, cudaStream_t st);
void dav_unit(double* t, double* p, const double* norm2, size_t n, cudaStream_t st);
void dav_column(double* av, const double* ap, const double* V, int m, size_t n, double* h, double* scratch,
                unsigned* counter, cudaStream_t st);
void dav_ritz(double* x, double* ax, double* z, const double* V, const double* AV, int m, size_t n, const double* y,
              double theta, double* out, double* scratch, unsigned* counter, cudaStream_t st);

// ---- learned preconditioner (kernels_mlp.cu)
struct BlockRef {      // one QN block of a two-site vector
    size_t off;
    int len;
    int pad;
};
constexpr int MLP_NF = 16;   // features per block
void mlp_gemm_bf16w(int M, int N, int K, const float* A, int lda, bool ta, const void* B, int ldb, bool tb,
                    float* C, int ldc, const float* bias, const float* mask, int epi, cudaStream_t st);
// Weight gradient gW (M x N) = dY^T X over K samples and bias gradient gb (M) =
// column sums of dY.  With mlp_wgrad_pieces(K) > 1 the pieces go to part
// (pieces * (M N + M) floats) and mlp_wgrad_sum adds them.
int mlp_wgrad_pieces(int K);
void mlp_wgrad(int M, int N, int K, const float* dY, const float* X, float* gW, float* gb, float* part, cudaStream_t st);
struct MlpSums {
    struct L {
        const float* part;
        float *gW, *gb;
        int wn, bn, pieces;
    } l[3];
    int count;
};
void mlp_wgrad_sum(const MlpSums& s, cudaStream_t st);
void mlp_mse(int B, int N, const float* Y, const float* T, float* dY, float* rowloss, cudaStream_t st);
void mlp_adam(int n, float* w, const float* g, float* m, float* v, void* wb, float lr, int step, cudaStream_t st);
void mlp_to_bf16(int n, const float* w, void* wb, cudaStream_t st);
void block_features(const BlockRef* blocks, int nb, const double* diag, const double* g, const double* xw,
                    const float* meta, float* feats, cudaStream_t st);
void block_combine(const BlockRef* blocks, int nb, const float* coef, const double* xw, const double* minv,
                   const double* bvec, double* x0, cudaStream_t st);
void block_fit(const BlockRef* blocks, int nb, const double* xw, const double* minv, const double* bvec,
               const double* x, double* out, cudaStream_t st);

}  // namespace mpspt
