// Internal declarations shared by the translation units of libxk.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>
#include <string>

namespace xk {

// Kernel launches issued since load (all translation units), and by the
// calling thread (a graph capture counts its own launches with it).
extern std::atomic<uint64_t> g_launches;
inline thread_local uint64_t t_launches = 0;
inline void count_launch(uint64_t k = 1) {
  g_launches.fetch_add(k, std::memory_order_relaxed);
  t_launches += k;
}

// ---------------------------------------------------------------------------
// FP64 SIMT path (xk_fp64.cu)
// ---------------------------------------------------------------------------

// C[M x N] = alpha * op(A) op(B) (o H) + beta * C, row-major.  op(A)[m,k] is
// A[k*lda + m] when transA else A[m*lda + k]; op(B)[k,n] is B[n*ldb + k] when
// transB else B[k*ldb + n].  H (nullable, ldh) multiplies the result
// element-wise (the Hadamard epilogue).  ksplit > 1 splits K: partial sums
// go to `work` (ksplit * M * N doubles) and are summed in split order, so
// the result does not depend on scheduling.
struct DGemm {
  int M, N, K;
  const double* A; long lda; bool transA;
  const double* B; long ldb; bool transB;
  double* C; long ldc;
  double alpha;
  const double* H; long ldh;
  int ksplit;
  double* work;
  double beta;  // C = alpha op(A) op(B) (o H) + beta C (0: C is not read)
  int* scale;   // nullable: digit_scale_ints(M, N) ints of scratch, with which large
                // products run on the tensor cores (xk_digits.cu)
  int nbatch;   // > 0: the columns of C come in batches of nbatch: column n is stored
  long cskip;   // (n / nbatch) cskip elements further on, and H has column n % nbatch
  bool sym;     // C is symmetric (M = N, no H, beta = 0): one half may be formed and mirrored
  int *rmax, *cmax;          // digit_maxima(g): high words of the largest |C| per row and
                             // column, for products that take C as an operand
  const int *amax, *bmax;    // those of op(A)'s rows / op(B)'s columns, when they are known
  int* status;               // nullable: gets a code when a bounded wait of the digit product gives up
  long long wait;            // limit of those waits in SM cycles (0: the default)
};
// The result overwrites rows of B (M <= 64, one row of tiles, unsplit: every block has read
// its columns of B before it writes them).
__host__ __device__ inline bool in_place(const DGemm& g) {
  return g.C >= g.B && g.C < g.B + (g.transB ? (long)g.N : (long)g.K) * g.ldb;
}
cudaError_t dgemm(const DGemm& g, cudaStream_t s);

// Powers of two.  The digit products (xk_digits.cu) hold an operand's row on one grid, so
// terms of a product lose bits when its two operands are graded in opposite directions
// along K; scaling by powers of two, exact, puts them on one footing.
// The exponents e of the largest |x| of every row (of rows idx[0..rows) of p, idx nullable) or
// column of a matrix, 2^(e-1) <= |x| < 2^e, at most `limit` in size; 0 for rows of zeros or
// with infinities or NaN.
cudaError_t row_exponents_f64(const double* p, long ld, const int32_t* idx, int rows, int cols, int limit,
                              int* out, cudaStream_t s);
cudaError_t col_exponents_f64(const double* p, long ld, long rows, int cols, int limit, int* out,
                              cudaStream_t s);
// A2 = A 2^e, B2 = B 2^-e, row by row, with e such that both have rows of one size.
cudaError_t balance_rows_f64(const double* A, const double* B, int rows, int cols, double* A2, double* B2,
                             cudaStream_t s);
// out[i] = a[i] - b[i].
cudaError_t sub_i32(const int* a, const int* b, int n, int* out, cudaStream_t s);
// dst[r][c] = f (src[r][c] 2^(rm re[r] + cm ce[c])) (re, ce nullable; dst may be src).
cudaError_t scale_f64(const double* src, double* dst, long rows, long cols, const int* re, int rm,
                      const int* ce, int cm, cudaStream_t s, double f = 1.0);

// The product of dgemm on the tensor cores, split into exact digits
// (xk_digits.cu): whether its size calls for it, the K split it wants (at most
// cap), and the launch (ksplit partial sums of kchunk terms each in g.work
// when ksplit > 1).  *g.scale is 0 afterwards, or not when the product has to be
// formed with FP64 FMAs instead (an operand that is not finite).
size_t digit_scale_ints(int M, int N);
bool digit_maxima(const DGemm& g);  // whether the product can leave rmax and cmax
bool digit_gemm_wanted(const DGemm& g);
int digit_ksplit(int M, int N, int K, bool sym, int cap);
cudaError_t digit_gemm(const DGemm& g, int ksplit, int kchunk, cudaStream_t s);
// Split count dgemm picks when DGemm::ksplit == 0 (work needs ksplit*M*N).
int dgemm_ksplit(int M, int N, int K);

// out[r, c] = in[idx[r] * ld_in + c] 2^-re[r] for r < rows, c < cols (row gather; re nullable).
cudaError_t gather_rows_f64(const double* in, long ld_in, const int32_t* idx, int rows, int cols,
                            double* out, long ld_out, cudaStream_t s, const int* re = nullptr);

// K[mu, i] = dV * ((L1[i, mu] + L2[i, mu] - L3[i, mu]) 2^ce[mu]); L* are n x N.
cudaError_t assemble_k_f64(const double* L1, const double* L2, const double* L3, int n, int N,
                           double dV, const int* ce, double* K, cudaStream_t s);

// *out = -sum_j a[j] * b[j] over `len` doubles, fixed summation order.
// `work` holds at least reduce_work_elems() doubles.
cudaError_t neg_dot_f64(const double* a, const double* b, long len, double* work, double* out,
                        cudaStream_t s);
size_t reduce_work_elems();

// Poisson solves on a cubic g^3 grid in the real product basis of its axes
// (xk_fp64.cu).  Tables of one (g, L): poisson_table_elems(g) doubles, filled by
// poisson_tables_f64 (tab stays the caller's; uploads from host memory and
// waits for it).
size_t poisson_table_elems(int g);
cudaError_t poisson_tables_f64(int g, double L, double* tab, cudaStream_t s);
// out = Pois(in) (Eq. cou-1: 4 pi / G^2 on the grid's reciprocal vectors, G = 0
// removed) for nf functions of g^3 values each; in is kept, out and tmp (nf g^3
// each) are not the same memory.  scale: DGemm::scale of the products
// (scale_ints ints), nullable; wst: their DGemm::status.
cudaError_t poisson_f64(const double* in, double* out, double* tmp, long nf, int g,
                        const double* tab, int* scale, size_t scale_ints, int* wst, cudaStream_t s);
// rho[R] = sum_i psi[R][i]^2 for psi (ng x n).
cudaError_t density_f64(const double* psi, long ng, int n, double* rho, cudaStream_t s);
// out[R][nu] = v[R] phi[R][nu].
cudaError_t potential_rows_f64(const double* v, const double* phi, long ng, int N, double* out,
                               cudaStream_t s);
// *out = scale * sum_j a[j] b[j] (fixed order); `work` holds reduce_work_elems() doubles.
cudaError_t dot_f64(const double* a, const double* b, long len, double scale, double* work,
                    double* out, cudaStream_t s);

// K[mu][nu] = dV ((Y[mu][nu] + Y[nu][mu] - Z[mu][nu]) 2^(ce[mu] + ce[nu])) for N x N matrices.
cudaError_t assemble_full_f64(const double* Y, const double* Z, int N, double dV, const int* ce,
                              double* K, cudaStream_t s);

// GPU ISDF set-up (xk_isdf.cu), all FP64: from Phi (ng x N) and Phi_g
// (na x N), X_gg into Xgg (na x na, overwritten by its Cholesky factor),
// chi = X_gg^{-1} X_gR (na x ng), V = Pois(chi) on the cubic grid^3 grid of
// side L (na x ng) and W = V chi^T symmetrised (na x na).  `work` holds the
// split-K work of the products (dgemm_ksplit sizes) and at least na doubles, `dig` is
// DGemm::scale of an na x ng product (dig_ints ints), `wst` DGemm::status of all: where that is set
// afterwards the tables are not to be used.
// A ridge of 1e-14 tr(X_gg)/na is added when the plain factorisation fails
// (*ridge_out); cudaErrorInvalidValue if it still fails.
// phig holds the rows of Phi_g times 2^-u[g] (u: device): the row of a point where the basis
// is small is as large as any in X_gg and in the solves, whose digit products (xk_digits.cu)
// would lose bits otherwise.  X_gg and X_gR then stand times 2^(-2 u) on the side of each g, and
// chi, V and W come out times 2^(2 u).
cudaError_t isdf_tables_f64(const double* phi, long ng, int N, const double* phig, const int* u, int na,
                            int grid, double L, double* Xgg, double* chi, double* V, double* W,
                            double* work, int* dig, size_t dig_ints, int* wst, int* status,
                            double* ridge_out, cudaStream_t s);
// Interpolation points (Sec. III.A) by a greedy complete-pivoting Cholesky of
// X = (F F^T) o (F F^T) for the m candidate rows F (m x N, device): up to
// `want` pivots (indices into F, selection order) into piv (host), stopping
// when the largest remaining diagonal is at most tol_rel times the largest
// initial one; *count = pivots taken.  Holds m N + m want doubles of
// stream-ordered scratch during the call.
cudaError_t select_points_f64(const double* F, int m, int N, int want, double tol_rel,
                              int32_t* piv, int* count, cudaStream_t s);
// In-place blocked Cholesky (lower) of the n x n matrix A (lda); *status = 1
// on a non-positive pivot.  scale, wst (here and below): DGemm::scale and status of the updates.
cudaError_t cholesky_blocked_f64(double* A, int n, long lda, int* status, int* scale, int* wst,
                                 cudaStream_t s);
// B (n x ncols, ldb) := (L L^T)^{-1} B with the lower factor L (ldl), which is overwritten.
cudaError_t cholesky_solve_f64(double* L, int n, long ldl, double* B, long ldb, long ncols,
                               int* scale, int* wst, cudaStream_t s);

// *out = -dV (2 sum_t V[t] P[t]^2 - sum_t W[t] Q[t]^2) over lenA and lenC
// elements, in a fixed order; `work` holds reduce_work_elems() doubles.
cudaError_t closed_form_ex_f64(const double* V, const double* P, long lenA, const double* W,
                               const double* Q, long lenC, double dV, double* work, double* out,
                               cudaStream_t s);

// A <- (A + A^T) / 2 for an n x n matrix.
cudaError_t symmetrize_f64(double* A, int n, cudaStream_t s);

// Kij = (C^T K + K^T C) / 2 for C, K of N x n.
cudaError_t kij_f64(const double* C, const double* K, int N, int n, double* Kij, cudaStream_t s);

// In-place Cholesky A = L L^T (lower, n x n, zeros above).  *status = 0 on
// success, k + 1 if the k-th pivot is not positive (A then holds no factor).
// cholesky_f64: one block (the tensor path's set-up).
cudaError_t cholesky_tiled_f64(double* A, int n, int* status, cudaStream_t s);
cudaError_t cholesky_f64(double* A, int n, int* status, cudaStream_t s);
// One step of it, for a blocked factorisation: the kb x kb block at (k, k), kb <= 64,
// and the panel below it (*status as above, set only on failure).
cudaError_t cholesky_step_f64(double* A, long lda, int k, int kb, int n, int* status, cudaStream_t s);

// X <- B L^{-T} for L lower n x n and B rows x n (row-major): solves
// X L^T = B row by row.  LT: n x n scratch (nullable: the slow general kernel).
cudaError_t trsm_right_lt_f64(const double* L, int n, const double* B, int rows, double* X,
                              cudaStream_t s, double* LT = nullptr);

// Cyclic Jacobi eigendecomposition of the symmetric n x n matrix A (one
// block): on return A holds the eigenvalues on its diagonal and U the
// eigenvectors as columns.  Runs at most max_sweeps sweeps; *sweeps gets the
// number used.
cudaError_t jacobi_eig_f64(double* A, double* U, int n, int max_sweeps, int* sweeps,
                           cudaStream_t s);

// X[r, k] = B[r, k] * f(lambda_k) with f = |lambda|^{-1/2} when
// |lambda| > cut * max|lambda| else 0; sign[k] = sign(lambda) or 0.
cudaError_t scale_eigcols_f64(const double* Adiag_src, int n, const double* B, int rows, double cut,
                              double* X, double* sign, cudaStream_t s);

// Allocation-free E_x = -sum K[t] C[t] with partial sums in a fixed
// file-scope device array (xk_noalloc.cu); count <= noalloc_max_count().
int64_t noalloc_max_count();
cudaError_t exchange_energy_noalloc(const double* K, const double* C, int64_t count, double* Ex,
                                    cudaStream_t s);

}  // namespace xk
