// Internal declarations shared by the translation units of libamdd.
// Dense matrices are row-major: element (r, c) of a matrix with leading
// dimension ld sits at p[r * ld + c].
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

namespace amdd {

// Bits of the device error word.
enum : int {
    DERR_NOT_SPD = 1,        // Cholesky pivot <= 0 (or NaN) without clamping
    DERR_EIG_NOCONV = 2,     // Jacobi sweep limit reached
    DERR_BOUNDS = 4,         // an index check failed
    DERR_TIMEOUT = 8,        // a bounded device wait (mbarrier) gave up
};

constexpr int CHOL_NB = 32;     // diagonal block of the blocked Cholesky / inverse
constexpr int GEMM_T = 64;      // GEMM output tile
constexpr int PANEL_ROWS = 16;  // rows per CTA of the Cholesky panel solve
constexpr int MAXB = 8;                // right-hand sides per batched apply / PCG pass
constexpr int JAC_CLUSTER = 8;  // CTAs per matrix in the Jacobi solvers
constexpr int JAC_MAX_PAIRS = 64;  // largest sub-round of the shared-memory block Jacobi

// ---------------------------------------------------------------- dense
// C = alpha * op(A) * op(B) + beta * C for m x n outputs, inner dimension k.
// ta = 0: A is m x k (A[r*lda + kk]); ta = 1: A is stored k x m (A[kk*lda + r]).
// tb = 0: B is k x n (B[kk*ldb + c]); tb = 1: B is stored n x k (B[c*ldb + kk]).
// lower = 1: only elements with r >= c are written (tiles above skipped).
// kfrom_row = 1: the k loop starts at the tile's first row (for products whose
// A operand is zero for kk < r, e.g. a lower-triangular Y read transposed).
// beta == 0 means C is not read.
template <typename T>
struct GemmDescT {
    const T* A;
    const T* B;
    T* C;
    int m, n, k;
    int lda, ldb, ldc;
    int ta, tb, lower, kfrom_row;
    T alpha, beta;
};
using GemmDesc = GemmDescT<double>;

struct TileRef {
    int desc, tm, tn;
};

// Blocked Cholesky / inverse-factor descriptors (one per matrix).
template <typename T>
struct CholDescT {
    T* A;            // n x n, lower triangle used and overwritten with L
    int n, ld;
    int stop;        // factor columns [0, stop); stop < n leaves the Schur complement
    const T* clamp;  // per-matrix pivot floor (pivots below are raised to it); NULL = SPD check
    T* Linv;         // ceil(stop/NB) * NB*NB entries: inverses of the diagonal blocks
    int* bad = nullptr;  // with clamp: set to 1 when a computed pivot falls below 0.9 x the floor
                         // (or is not finite): the matrix is not numerically definite at that floor
};
using CholDesc = CholDescT<double>;

struct PanelRef {
    int desc, rt;  // row tile index (PANEL_ROWS rows) below the diagonal block
};

template <typename T>
struct TrtriDescT {
    const T* L;     // n x n lower Cholesky factor (ld)
    T* Y;           // n x n output L^{-1} (ldy), lower triangular
    const T* Linv;  // diagonal-block inverses from the Cholesky
    int n, ld, ldy;
};
using TrtriDesc = TrtriDescT<double>;

struct ChunkRef {
    int desc, ct;  // column chunk (64 columns)
};

// a looser tolerance for long rows (above: squared length, 0: none)
template <typename T>
struct JacLoose {
    T above, tol;
};
template <typename T>
struct JacobiDescT {
    T* A;               // rows x ld, rows orthogonalised in place
    int rows, ld;
    int ncols_dot;      // columns entering the inner products
    int ncols_rot;      // columns rotated (>= ncols_dot)
    T* nrm2;            // rows scratch entries (squared row norms)
    const T* absfloor;  // optional absolute floor on |<p,q>| below which no rotation is made
    // optional f: no rotation either while <p,q>^2 <= u f max(|p|^2, |q|^2) (u the
    // unit roundoff of T).  With f = u |M|^2 (launch_row_maxnorm2) a pair is left
    // alone once its coupling is below the rounding of M itself, u |M|.
    const T* normfloor = nullptr;
    // optional: two rows both longer than sqrt(loose.above) need only be orthogonal
    // to loose.tol (their span, not the rows themselves, is wanted)
    JacLoose<T> loose = {};
};
// squared relative tolerance for the pair of squared lengths a, b
template <typename T>
__host__ __device__ __forceinline__ T jac_tol2(T tol, T a, T b, JacLoose<T> l) {
    const T t = l.above > T(0) && (a < b ? a : b) > l.above ? l.tol : tol;
    return t * t;
}
using JacobiDesc = JacobiDescT<double>;

// Conversion descriptors of the FP32 preconditioning stage of the Jacobi solvers.
struct CvtDesc {
    const double* A;  // rows x L (lda)
    int rows, L, lda;
    float* out32;     // rows x (L + rows), ld32
    int ld32;
    double* Q;        // rows x rows
};

// Symmetric tridiagonal reduction and bisection (eigenvalues only).
template <typename T>
struct TridiagDescT {
    T* A;  // n x n symmetric, full storage (ld); destroyed
    int n, ld;
    T* d;  // n
    T* e;  // n (e[i] = T[i][i-1], e[0] = 0)
    T* p;  // n scratch
};
using TridiagDesc = TridiagDescT<double>;

// Row GEMV descriptors: y[row] = (b ? b[row] : 0) + alpha * sum_{c in [c0(row), c1(row))} M[row][c] x[c].
// mode 0: full row [0, ncols); mode 1: lower [0, row]; mode 2: upper [row, ncols).
template <typename T>
struct GemvDescT {
    const T* M;
    int rows, ncols, ld;
    const T* x;
    T* y;
};
using GemvDesc = GemvDescT<double>;

template <typename T>
void launch_gemm(const GemmDescT<T>* d_descs, const TileRef* d_tiles, int ntiles, int tile, cudaStream_t s);
template <typename T>
void launch_chol_diag(const CholDescT<T>* d, int nmat, int k0, int* err, cudaStream_t s);
template <typename T>
void launch_chol_panel(const CholDescT<T>* d, const PanelRef* tiles, int ntiles, int k0, cudaStream_t s);
template <typename T>
void launch_trtri_diag(const TrtriDescT<T>* d, const ChunkRef* tiles, int ntiles, int k0, cudaStream_t s);
template <typename T>
void launch_set_identity(const TrtriDescT<T>* d, int nmat, int maxn, cudaStream_t s);
// Block-pair variant for matrices of any size (rows in global memory): one
// round of the block round-robin schedule (blocks of 32 rows; tasks[t] =
// {matrix, pair index in the round, blocks of that matrix (even, >= 2), 0});
// rotated[matrix] is set when a pair of it was rotated, rots[matrix] counts
// plane rotations, stats[6] accumulates pair tasks, rotated pairs, the SM
// cycles of the three phases (Gram matrix, small eigensolve, rotation of the
// rows) and the inner sweeps.  The host runs the rounds of a sweep and the sweeps.
constexpr int JP_ROWS = 32;
// leading dimension with every row on a 128-byte boundary: the tensor-core kernel's
// 16-byte loads need 16, and its stores of 32 columns then fill whole lines
inline int jacobi_ld(int ncols) { return (ncols + 31) / 32 * 32; }
template <typename T>
size_t jacobi_pair_smem();
template <typename T>
void launch_jacobi_pair_round(const JacobiDescT<T>* d, const int4* tasks, int ntasks, int round, T tol, int inner,
                              int* rotated, unsigned long long* rots, unsigned long long* stats, cudaStream_t s);
// Batched FP32 GEMM on the tensor cores (tcgen05, TF32 with the 3xTF32 split
// for FP32 accuracy), 128 x 128 output tiles (TileRef tm, tn in units of 128);
// a wait that gives up latches DERR_TIMEOUT in *err.
constexpr int TC_GEMM_TILE = 128;
size_t gemm_tc_smem();
// one sweep of the block-pair Jacobi in FP32 with the Gram matrices and the
// rotations on the tensor cores (3xTF32), as one persistent launch: tasks[t] =
// {matrix, pair index in its round, blocks of that matrix, round}, ordered by
// round; CTAs claim tasks through *counter (zero before the launch) and wait
// (bounded) until bdone[bofs[matrix] + block] (zero before the launch) shows
// that both row blocks of the pair have finished the previous round; results
// are those of the round-by-round launches.  DERR_TIMEOUT into *err when a
// wait gives up.  Returns the CTAs launched.
size_t jacobi_pair_tc_smem();
int launch_jacobi_pair_tc_sweep(const JacobiDescT<float>* d, const int4* tasks, int ntasks, int* counter, int* bdone,
                                 const int* bofs, float tol, int inner, int* rotated, unsigned long long* rots,
                                 unsigned long long* stats, int* err, cudaStream_t s);
// one thread waits (bounded, `limit` SM cycles) for *flag >= 1; DERR_TIMEOUT
// into *err when the wait gives up
void launch_wait_selftest(const int* flag, long long limit, int* err, cudaStream_t s);
void launch_gemm_tc(const GemmDescT<float>* d_descs, const TileRef* d_tiles, int ntiles, int* err, cudaStream_t s);
// *p |= bits (one thread)
void launch_or_flag(int* p, int bits, cudaStream_t s);
// Shared-memory-resident block variant; returns false (nothing launched) when
// the two row blocks of the largest matrix do not fit in shared memory.
constexpr size_t JAC_BLOCK_SMEM_MAX = 220 * 1024;
template <typename T>
size_t jacobi_block_smem(int rows, int ncols_rot, int cluster);
// Shared-memory-resident block variant with a cluster of JAC_CLUSTER CTAs per
// matrix, else (blocks too large) 2 * JAC_CLUSTER; returns false, with nothing
// launched, when neither fits (smem8 / smem16: bytes per CTA for the two sizes;
// floors: some matrix has absfloor, normfloor or loose).
template <typename T>
bool launch_jacobi_block(const JacobiDescT<T>* d, int nmat, size_t smem8, size_t smem16, int max_rows,
                         int max_sweeps, T tol, int* sweeps, unsigned long long* rots, int* err, int report_noconv,
                         bool floors, cudaStream_t s);
template <typename T>
void launch_row_maxnorm2(const JacobiDescT<T>* d, int nmat, T eps, T* out, cudaStream_t s);
void launch_to_f32_with_identity(const CvtDesc* d, int nmat, int maxrows, cudaStream_t s);
void launch_extract_q(const CvtDesc* d, int nmat, int maxrows, cudaStream_t s);
// sigma[j] = ||row j|| over ncols_dot (as double); delta[mat] = eps * max_j sigma[j];
// optionally scale row j by 1/sqrt(sigma[j]).
// Robust Schur complement of the splitting (fallback when the clamped
// Cholesky of its [G, D] block is flagged): rows of C = Sigma^{1/2} V^T
// (n_i x nt, columns [C_R | C_I], C_R the first nR) give
//   J = [C_R | I_{n_i}]  (n_i x (nR + n_i), leading dimension ldj), and after
//   the one-sided Jacobi of J's rows (inner products over the first nR
//   columns) each row k of its right part is scaled by 1 / sqrt(s_k^2 + delta)
//   with s_k^2 the squared norm of its left part.
template <typename T>
struct KjacDesc {
    const T* C;  // n_i x nt (ldc)
    T* J;        // n_i x (nR + n_i) (ldj)
    int ni, nR, ldc, ldj;
    const T* delta;
};
// Coarse block of a subdomain whose every eigenvalue is selected: the nI x nI
// rows Zt[k][c] = (k == c) / sqrt(A_II[k][k]) (A_ii dense FP64, leading
// dimension lda).
struct DiagBasisDesc {
    const double* A;
    int lda;
    double* Zt;
    int nI;
};
void launch_diag_basis(const DiagBasisDesc* d, int nmat, int maxn, cudaStream_t s);
// With that basis: AZ[r][c] = A_ii[r][c] / sqrt(A_II[c][c]) (ni x nI, leading
// dimension nI) and the lower triangle of E_ii[r][c] = AZ[r][c] / sqrt(A_II[r][r])
// (leading dimension ldE).
struct DiagScaleDesc {
    const double* A;  // A_ii dense, ni x ni (leading dimension ni)
    int ni, nI;
    double* AZ;
    double* Eii;
    int64_t ldE;
};
void launch_diag_scale(const DiagScaleDesc* d, int nmat, int maxni, cudaStream_t s);
// Matrix-free local eigensolve (eq. (invAii)): from the scaled rows C =
// Sigma^{1/2} V^T of the SVD of X_i (ni x nt, leading dimension ld, the
// Omega_Ii columns from nR on) and the row norms sigma, Cc = C(:, I) and
// Bm = diag(1 / (sigma + delta)) C(:, I), both ni x nI contiguous.
struct MfPrepDesc {
    const double* X1;
    int ld, nR, ni, nI;
    const double* sig;    // sigma_j of row j
    const double* delta;  // sigma_1 eps (one value)
    double* Cc;
    double* Bm;
};
void launch_mf_prepare(const MfPrepDesc* d, int nmat, int maxni, cudaStream_t s);
template <typename T>
void launch_build_kjac(const KjacDesc<T>* d, int nmat, int maxrows, cudaStream_t s);
template <typename T>
void launch_kjac_scale(const KjacDesc<T>* d, int nmat, cudaStream_t s);
template <typename T>
void launch_rownorms(const JacobiDescT<T>* d, int nmat, double* const* sigma_ptrs, T* delta, double eps,
                     int scale_rows, cudaStream_t s);
template <typename T>
void launch_add_diag(T* const* mats, const int* n, const int* ld, const T* delta, int nmat, int maxn, cudaStream_t s);
template <typename T>
void launch_mirror_lower(T* const* mats, const int* n, const int* ld, int nmat, int maxn, cudaStream_t s);
template <typename T>
void launch_gemv_rows(const GemvDescT<T>* d, const int* row_desc, const int* row_local, int64_t nrows,
                      cudaStream_t s);
template <typename T>
void launch_gemv_rows_multi(const GemvDescT<T>* d, const int* row_desc, const int* row_local, int64_t nrows, int nb,
                            int64_t xs, int64_t ys, cudaStream_t s);
// whether a matrix of order n fits the distributed shared memory of a cluster
template <typename T>
bool tridiag_fits(int n);
template <typename T>
void launch_tridiag(const TridiagDescT<T>* d, int nmat, int maxn, cudaStream_t s);
template <typename T>
void launch_bisect(const TridiagDescT<T>* d, int nmat, const int* eig_mat, const int* eig_idx, int64_t total,
                   double* const* out, cudaStream_t s);
// dst[i] = (To)src[i]
template <typename Ti, typename To>
void launch_convert(const Ti* src, To* dst, int64_t n, cudaStream_t s);
template <typename Ti, typename To>
void launch_convert_blocks(const Ti* const* src, const int* lds, To* const* dst, const int* ldd, const int* n,
                           int nmat, int maxn, cudaStream_t s);

// ---------------------------------------------------------------- sparse / vectors
struct PcgScal {
    double rz, pq, rr, bb, alpha, beta;
    int conv, iters;
    unsigned ticket;  // CTAs of the running reduction that have finished (0 between kernels)
    unsigned pad;
};
// A dot product computed at the end of a kernel: nb sums into the scalars sc[k].
// which: 0 -> pq (alpha = rz/pq), 1 -> rz (beta = new rz / old rz), 2 -> rr (conv = rr
// <= tol2 * bb, iters + 1), 3 -> bb, 4 -> rz (initial), 5 -> rr (conv).  part: nb x CTAs
// of the kernel partial sums (at most DOT_MAX_BLOCKS each); skip: a right-hand side
// that has converged keeps its scalars.
struct DotArgs {
    double* part = nullptr;
    PcgScal* sc = nullptr;
    int which = 0;
    double tol2 = 0.0;
    int skip = 0;
};
constexpr int DOT_BLOCKS = 264;            // CTAs of the plain vector kernels
constexpr int DOT_MAX_BLOCKS = 152 * 16;   // CTAs of a kernel with a fused dot product, at most
// Sparse local Cholesky factors: per subdomain its order n, factor entries
// nnz, the offset of its column pointers (n + 1 local offsets), of its entries
// and of its rows in the local vectors.
struct SparseLocalDesc {
    int n, nnz;
    int64_t poff, eoff, xoff;
};
// dst[t] = src[idx[t]] (idx >= 0) or 1 / src[-idx[t] - 1]
template <typename T>
void launch_gather_entries(const T* src, const int64_t* idx, T* dst, int64_t cnt, cudaStream_t s);
// y_i = P^T L^{-T} L^{-1} P r_i with the factors staged in shared memory (smem:
// the largest sparse_local_smem of the batch for nb vectors), nb <= MAXB
// vectors ld apart
template <typename T>
size_t sparse_local_smem(int n, int nnz, int nb);
template <typename T>
void launch_sparse_local_solve(const SparseLocalDesc* d, int nmat, size_t smem, const int32_t* colptr,
                               const uint16_t* rowidx, const T* val, const int32_t* perm, const T* r, T* y, int nb,
                               int64_t ld, cudaStream_t s);

// Host: nested-dissection order of the symmetric pattern of an n x n CSR graph
// (sets of at most `leaf` unknowns not cut) and the column structure of the
// Cholesky factor of P A P^T in that order: perm[k] = old index of new k,
// column j holds rows[colptr[j] .. colptr[j+1]), the diagonal j first, then
// ascending.  False on a malformed graph.
bool nd_factor_pattern(int n, const int64_t* rowptr, const int32_t* colind, int leaf, std::vector<int32_t>& perm,
                       std::vector<int32_t>& colptr, std::vector<int32_t>& rows);

// *flag |= 1 when v[0..n) holds a NaN or an infinity
void launch_nonfinite(const double* v, int64_t n, int* flag, cudaStream_t s);
// y = A x and y = b - A x: every SpMV of the library goes through these two
// launchers, which choose the form from n and nnz alone, so that equal inputs
// give equal bits
void launch_spmv(int64_t n, int64_t nnz, const int64_t* rowptr, const int32_t* col, const double* val,
                 const double* x, double* y, cudaStream_t s);
void launch_spmv_resid(int64_t n, int64_t nnz, const int64_t* rowptr, const int32_t* col, const double* val,
                       const double* x, const double* b, double* y, cudaStream_t s);
// y = A x and x.y into the PCG scalars
void launch_spmv_dot(int64_t n, int64_t nnz, const int64_t* rowptr, const int32_t* col, const double* val,
                     const double* x, double* y, const DotArgs& d, cudaStream_t s);
void launch_gather_values(const int64_t* src, const int64_t* dst, int64_t cnt, const double* val, double* out,
                          cudaStream_t s);
void launch_gather_vec(const int32_t* idx, int64_t cnt, const double* x, double* out, cudaStream_t s);
void launch_gather_vec_multi(const int32_t* idx, int64_t cnt, const double* x, int64_t ldx, double* out, int nb,
                             cudaStream_t s);
void launch_spmv_multi(int64_t n, const int64_t* rowptr, const int32_t* col, const double* val, const double* x,
                       double* y, int nb, int64_t ld, cudaStream_t s, const DotArgs* d = nullptr);
template <typename T>
void launch_gather_rows(const T* src, const int64_t* src_off, T* dst, const int64_t* dst_off, const int32_t* len,
                        int64_t nrows, cudaStream_t s);
template <typename TY>
void launch_scatter_prolong(int64_t n, const int32_t* order_g, const int64_t* sc_ptr, const int32_t* sc_idx,
                            const TY* yloc, const double* zc, double* z, cudaStream_t s, int nb = 1, int64_t ldy = 0,
                            int64_t ldzc = 0, int64_t ldz = 0, const double* r = nullptr,
                            const DotArgs* d = nullptr);
// batched rectangular transposes: dst (cols x rows, leading dimension ldd) = src^T
template <typename T>
struct TransDescT {
    const T* src;
    T* dst;
    int rows, cols, lds, ldd;
};
using TransDesc = TransDescT<double>;
template <typename T>
void launch_transpose_rect(const TransDescT<T>* d, int nmat, int maxdim, cudaStream_t s);
struct EPairRef {
    int i, j;          // block E_ij, i > j
    int64_t list_off;  // entries [list_off, list_off + list_len)
    int list_len;
    int tr, tc;        // 32x32 tile of the p_i x p_j block
};
void launch_e_offdiag(const EPairRef* tiles, int ntiles, const int32_t* la, const int32_t* lpos,
                      const double* Zt, const int64_t* zt_off, const int32_t* nI, const double* AZ,
                      const int64_t* az_off, const int32_t* p, const int64_t* coff, double* E, int64_t ldE,
                      cudaStream_t s);

// ---------------------------------------------------------------------------
// Learned warm start of the local eigensolve and block LOBPCG
// ---------------------------------------------------------------------------
constexpr int PROP_NF = 32;    // features per subdomain
constexpr int PROP_NB = 16;    // Krylov basis vectors
constexpr int PROP_NH = 256;   // hidden width
constexpr int PROP_NO = 256;   // outputs: a 16 x 16 matrix
// parameter layout: W1 (32 x 256), b1, W2 (256 x 256), b2, W3 (256 x 256), b3
constexpr int64_t MLP_OFF_W1 = 0;
constexpr int64_t MLP_OFF_B1 = MLP_OFF_W1 + PROP_NF * PROP_NH;
constexpr int64_t MLP_OFF_W2 = MLP_OFF_B1 + PROP_NH;
constexpr int64_t MLP_OFF_B2 = MLP_OFF_W2 + PROP_NH * PROP_NH;
constexpr int64_t MLP_OFF_W3 = MLP_OFF_B2 + PROP_NH;
constexpr int64_t MLP_OFF_B3 = MLP_OFF_W3 + PROP_NH * PROP_NO;
constexpr int64_t MLP_NPARAM = MLP_OFF_B3 + PROP_NO;

// Features of subdomain i from its dense local matrix A_ii (rows [I, G],
// leading dimension ld, ncols = |Omega_i|):
//  0 log nI, 1 log(1+nG), 2 log(1+nD), 3 nG/nI, 4 nD/nI,
//  5-8 mean/std/min/max of log diag(A_II), 9-12 the same of log|off-diagonal
//  non-zeros of A_II|, 13 max - min of log diag, 14-16 mean/std/max of the
//  off-diagonal non-zeros per row, 17 fraction of rows coupled to Omega_G,
//  18-19 mean/max of sum_G |a_rg| / a_rr, 20-23 mean/std/min/max of
//  sum_{c != r} |a_rc| / a_rr, 24 log(||A_II||_F / nI), 25 log(trace / nI),
//  26 fraction of positive off-diagonal non-zeros, 27 log(max(p,1)/nI),
//  28 log max(p,1), 29 log tau, 30 mean log diag over coupled rows minus
//  the mean over all rows, 31 the constant 1.
struct FeatDesc {
    const double* A;
    int ld, ncols, nI, nG, nD, p;
    double tau;
    float* out;  // 32 entries
};
void launch_features(const FeatDesc* d, int nmat, cudaStream_t s);

struct KrylovDesc {
    const double* A;  // A_II is the leading nI x nI block (leading dimension ld)
    int ld, nI;
    double* Bt;  // PROP_NB x nI, rows = basis vectors
    double* w;   // nI scratch
};
void launch_krylov(const KrylovDesc* d, int nmat, cudaStream_t s);

// mean[f], sd[f] (population; < 1e-6 -> 1) of the columns of an n x PROP_NF matrix
void launch_feature_stats(const float* feat, int n, float* mean, float* sd, cudaStream_t s);
void launch_normalize_features(const float* feat, const float* mean, const float* sd, float* X, int n,
                               cudaStream_t s);
// The proposal network (mlp_kernels.cu): q (n x 256) of n samples; one training
// step (work as amdd_mlp_sizes; lr = 0: gradient and loss only)
void launch_mlp_forward(const float* wb, const float* x, int n, float* q, cudaStream_t s);
void launch_mlp_step(float* w, float* wb, float* m, float* v, int t, float lr, const float* x, const float* qt, int n,
                     float* grad, float* work, float* loss, cudaStream_t s);
void launch_bf16_round(const float* W, float* Wb, int n, cudaStream_t s);
// bfloat16 rounding of binary32: add 0x7FFF plus the lowest kept bit, keep
// the top 16 bits (nearest, ties to even); NaN stays NaN.
__device__ __forceinline__ float bf16_round(float x) {
    if (x != x) return x;
    unsigned u = __float_as_uint(x);
    u = (u + 0x7FFFu + ((u >> 16) & 1u)) & 0xFFFF0000u;
    return __uint_as_float(u);
}

template <typename T>
struct RowsDesc {  // rows [r0, r1) of a row-major matrix (cols entries each)
    T* A;
    int ld, r0, r1, cols, id;
};
template <typename T>
void launch_rng_rows(const RowsDesc<T>* d, int nmat, int maxrows, unsigned long long seed, cudaStream_t s);

template <typename T>
void launch_zero_upper(const RowsDesc<T>* d, int nmat, int maxrows, cudaStream_t s);
// out[t] = dot of the two halves (len[t] entries each) of the row at W + off[t]
template <typename T>
void launch_half_dots(const T* W, const int64_t* off, const int32_t* len, int64_t rows, double* out, cudaStream_t s);

template <typename T>
struct ResidDesc {  // R = TX - diag(theta) X over k rows of n entries; norms of the first `want`
    const T* X;
    const T* TX;
    T* R;
    const T* theta;
    double* norms;
    int ld, n, k, want;
};
template <typename T>
void launch_residual_rows(const ResidDesc<T>* d, int nmat, cudaStream_t s);

template <typename T>
struct ScaleDesc {  // A[r] *= f[r] (or 1 / ||A[r]|| with unit scaling)
    T* A;
    int ld, rows, cols;
    const T* f;
};
template <typename T>
void launch_scale_rows(const ScaleDesc<T>* d, int nmat, int unit, cudaStream_t s);

// Exact solves by substructuring (front_kernels.cu).  One part: its front F
// ((m + nb) x (m + nb), lower triangle, setup only), Ainv (m x m, symmetric,
// full) and W (m x nb), its interior at plan positions i0 .. i0 + m and its
// boundary bnd[b0 .. b0 + nb).
template <typename T>
struct FrontDevT {
    T* F;
    T* Ainv;
    T* W;
    int m, nb;
    int64_t i0, b0;
    int kid0, kid1;  // children (FrontChild) whose Schur complements enter F
};
struct FrontChild {
    const double* S;  // Schur complement on the child's boundary (lower triangle)
    int ld;
    int64_t map, inv;  // offsets of the maps child boundary -> parent row, parent row -> child boundary
};
template <typename T>
struct FrontRefT {  // a row of W^T and the interior it multiplies
    const T* row;
    int64_t i0;
    int m;
};
template <typename T>
struct FrontSolveT {
    int64_t n = 0;
    int stages = 0;
    const int32_t* perm = nullptr;  // caller's index of each plan position (output)
    const int32_t* src = nullptr;   // its index in the input vectors
    const double* scale = nullptr;  // with it, input and output entries are multiplied by scale[plan position]
    const FrontDevT<T>* fr = nullptr;
    const int32_t* row_front = nullptr;
    const int32_t* bnd = nullptr;
    const int32_t* down_rows = nullptr;  // boundary unknowns of each stage's parts
    const int32_t* down_ptr = nullptr;   // their refs (one shared list, nrow + 1 pointers over all stages)
    const FrontRefT<T>* refs = nullptr;
    T* v = nullptr;  // work and solution: as many vectors of n each as a solve is given
    T* e = nullptr;
    std::vector<int64_t> down_off, row_off;  // host: per stage
    double entries = 0.0;                    // host: stored entries (multiply-adds of one solve)
};
// the dense matrix (lower triangle) that a front is gathered from: unknown u is its row u - off
struct FrontSrc {
    const double* A;
    int64_t ld, off;
};
void launch_front_gather(const FrontDevT<double>* fr, const FrontSrc* src, int nfr, const int32_t* bnd,
                         const int32_t* perm, int maxn, cudaStream_t s);
// scale[k] = own[perm[k]] = 1 / sqrt(val[diag[k]]) (val 0 where diag[k] < 0), k < n
void launch_front_scale(const double* val, const int64_t* diag, const int32_t* perm, double* scale, double* own,
                        int64_t n, cudaStream_t s);
// F[dst[t]] = val[src[t]] scale[a[t]] scale[b[t]], t < cnt
void launch_front_scatter(const double* val, const int64_t* src, const int64_t* dst, const int32_t* a,
                          const int32_t* b, const double* scale, double* F, int64_t cnt, cudaStream_t s);
void launch_front_extend_add(const FrontDevT<double>* fr, int nfr, const FrontChild* kids, const int32_t* maps,
                             int maxn, cudaStream_t s);
// the solution for nb <= MAXB vectors (c ldc apart) in a.e (plan order, n apart)
// and, when out is given, in the caller's order (ldo apart)
template <typename T>
void launch_front_solve(const FrontSolveT<T>& a, const double* c, int64_t ldc, T* out, int64_t ldo, int nb,
                        cudaStream_t s);

// Vector operations of PCG on nb right-hand sides stored ld apart; with d.skip (or
// skip_done) a converged right-hand side (sc[k].conv) keeps x, r, p and its scalars.
void launch_dot_partials(int64_t n, const double* x, const double* y, double* partials, cudaStream_t s, int nb = 1,
                         int64_t ld = 0);
void launch_dot(int64_t n, const double* x, const double* y, const DotArgs& d, cudaStream_t s, int nb = 1,
                int64_t ld = 0);
// x += alpha p, r -= alpha q, r.r (d); inside a graph's while-loop (maxit given) also
// alog[k-1] = alpha, blog[k-2] = beta (k = iterations done, entries below *maxit only)
// and the loop's condition !conv && k < *maxit
void launch_pcg_update_xr(int64_t n, double* x, double* r, const double* p, const double* q, const DotArgs& d,
                          cudaStream_t s, int nb = 1, int64_t ld = 0, const int* maxit = nullptr,
                          double* alog = nullptr, double* blog = nullptr, cudaGraphConditionalHandle loop = 0);
void launch_pcg_update_p(int64_t n, double* p, const double* z, const PcgScal* sc, cudaStream_t s, int nb = 1,
                         int64_t ld = 0, int skip_done = 0);
void launch_axpby(int64_t n, double a, const double* x, double b, const double* y, double* out, cudaStream_t s);
// ---------------------------------------------------------------------------
// Deflated / restricted additive Schwarz forms and GMRES(m) (Sec. 4.1)
// ---------------------------------------------------------------------------
// z[order_g[t]] = yloc[own_idx[t]] (+ zc[t] when zc is given)
template <typename TY>
void launch_ras_prolong(int64_t n, const int32_t* order_g, const int32_t* own_idx, const TY* yloc, const double* zc,
                        double* z, cudaStream_t s);
// zg[order_g[t]] = zo[t]
void launch_owner_to_global(int64_t n, const int32_t* order_g, const double* zo, double* zg, cudaStream_t s);
// out[t] = val[src[t]] (64-bit indices)
void launch_gather_idx64(const int64_t* src, int64_t cnt, const double* val, double* out, cudaStream_t s);
constexpr int GM_MAXR = 64;   // largest GMRES restart length
constexpr int GM_CHUNK = 32;  // basis vectors per block row of the fused Gram-Schmidt passes
struct GmState {
    double H[GM_MAXR * (GM_MAXR + 1)];  // Hessenberg matrix, column-major (column j: rows 0..j+1), rotated
    double cs[GM_MAXR], sn[GM_MAXR];    // Givens rotations
    double g[GM_MAXR + 1];              // rotated right-hand side beta e_1
    double y[GM_MAXR];                  // least-squares solution of a cycle
    double hcol[GM_MAXR + 1];           // projections of the current Gram-Schmidt pass
    double bnorm2, beta, hnext, res;    // ||b||^2, ||r_0|| of the cycle, h_{j+1,j}, |g_{j+1}| / ||b||
    int conv;
};
void launch_gm_ortho(int64_t n, const double* V, int64_t ldv, int k, const double* h, const double* w, double* out,
                     double* part, int mode, cudaStream_t s);
void launch_gm_finalize(const double* part, int k, double* hcol, double* Hcol, int add, cudaStream_t s);
void launch_gm_norm(const double* part, GmState* st, int which, cudaStream_t s);
void launch_gm_givens(const double* part, GmState* st, int j, double rtol, cudaStream_t s);
void launch_gm_scale(int64_t n, const double* src, double* dst, const GmState* st, int which, cudaStream_t s);
void launch_gm_trisolve(GmState* st, int k, cudaStream_t s);
void launch_gm_combine(int64_t n, const double* Zp, int64_t ldv, int k, const GmState* st, double* x,
                       cudaStream_t s);

}  // namespace amdd
