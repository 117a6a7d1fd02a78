// GPU FP64 ISDF set-up (Sec. III.A and IV.C of arXiv 2207.04636): from the
// basis on the grid and the interpolation points, the tables the exchange
// build consumes,
//   X_gg = (Phi_g Phi_g^T) o (Phi_g Phi_g^T),  X_gR = (Phi_g Phi^T) o (Phi_g Phi^T)
//   chi  = X_gg^{-1} X_gR          (Eq. lsqfit; blocked Cholesky, two blocked solves)
//   V    = Pois(chi_g)              (Eq. rpsPot; poisson_f64)
//   W    = V chi^T, symmetrised     (Eq. thcpot)
// all in FP64: the large products on the tensor cores (xk_digits.cu), the
// blocks of the factorisation and the solves on the CUDA cores; with a ridge of
// 1e-14 tr(X_gg) / N_aux added to the diagonal when the plain factorisation
// fails.
#include <algorithm>
#include <cmath>
#include <vector>

#include "tc_common.cuh"
#include "xk_internal.h"

namespace xk {

namespace {

constexpr int NB = 64;  // panel and block width of the factorisation and the solves

int nblocks(long total) { return (int)std::max<long>(1, std::min<long>((total + 255) / 256, 152L * 16)); }

__global__ void square_kernel(double* __restrict__ a, long rows, long cols, long ld) {
  const long count = rows * cols;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < count;
       t += (long)gridDim.x * blockDim.x) {
    const long r = t / cols, c = t % cols;
    const double v = a[r * ld + c];
    a[r * ld + c] = v * v;
  }
}

// d in the units of X_gg's rows and columns.
__global__ void add_diag_kernel(double* __restrict__ a, int n, long ld, double d, const int* __restrict__ u) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    a[(long)i * ld + i] += scalbn(d, -4 * u[i]);
}

__global__ void copy_diag_kernel(const double* __restrict__ a, int n, long ld, double* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = a[(long)i * ld + i];
}

// The triangular solves chi = L^{-T} L^{-1} X_gR run as two sweeps of one product per
// block row (64 rows of chi against every earlier or later one), with the 64 x 64
// diagonal blocks inverted beforehand:
//   forward   Y_k = D_k (B_k - sum_{j<k} L_kj Y_j)        D_k = L_kk^{-1}
//   backward  X_k = D_k^T (Y_k - sum_{j>k} L_jk^T X_j)
// The lower triangle of the factor takes F_kj = -D_k L_kj and D_k, the upper one
// G_kj = -(L_jk D_k)^T, so that each is one product [F_k0 .. D_k] [Y_0 .. B_k] or
// [D_k^T G_k,k+1 ..] [Y_k X_k+1 ..], in place.  Substitution inside the blocks ran at the
// FP64 FMA rate: 17.6 of 62 ms at 1053 functions of 45^3 points, 3.5 ms this way.

// D_k into the diagonal blocks (zeros above), one block of 64 threads per k: thread c
// forms column c by forward substitution.
__global__ void __launch_bounds__(NB) invert_diag_kernel(double* __restrict__ A, int n, long lda) {
  __shared__ double l[NB][NB + 1], rd[NB];
  const int k = blockIdx.x * NB, kb = min(NB, n - k), c = threadIdx.x;
  double* D = A + (long)k * lda + k;
  for (int i = 0; i < kb; ++i) l[i][c] = c <= i && c < kb ? D[(long)i * lda + c] : 0.0;
  __syncthreads();
  if (c < kb) rd[c] = 1.0 / l[c][c];
  __syncthreads();
  if (c >= kb) return;
  double x[NB];
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    if (i < kb) {
      double v = i == c ? 1.0 : 0.0;
#pragma unroll
      for (int j = 0; j < i; ++j) v = fma(-l[i][j], x[j], v);
      x[i] = v * rd[i];
      D[(long)i * lda + c] = i >= c ? x[i] : 0.0;
    } else {
      x[i] = 0.0;
    }
  }
}

// For block rows j > k (blockIdx.x: the pair, blockIdx.y: 16 of the 64 columns or rows):
// upper: G_kj = -(L_jk D_k)^T into block (k, j); else F_jk = -D_j L_jk in place.
__global__ void __launch_bounds__(256) scale_blocks_kernel(double* __restrict__ A, int n, long lda, int upper) {
  __shared__ double l[NB][NB + 1], d[NB][NB + 1];
  int j = (int)((sqrtf(8.0f * blockIdx.x + 1.0f) + 1.0f) * 0.5f);  // pair = j (j - 1) / 2 + k
  while (j * (j - 1) / 2 > (int)blockIdx.x) --j;
  while ((j + 1) * j / 2 <= (int)blockIdx.x) ++j;
  const int k = (int)blockIdx.x - j * (j - 1) / 2;
  const int jr = j * NB, kr = k * NB, jb = min(NB, n - jr);  // block row k < j is whole
  const int q0 = blockIdx.y * 16, dr = upper ? kr : jr, db = upper ? NB : jb;
  // in place: a block reads the 16 columns of L_jk it rewrites (F), or rows for G
  for (int t = threadIdx.x; t < NB * NB; t += 256) {
    const int r = t / NB, c = t % NB;
    d[r][c] = r < db && c <= r ? A[(long)(dr + r) * lda + dr + c] : 0.0;
    const bool mine = upper ? r >= q0 && r < q0 + 16 : c >= q0 && c < q0 + 16;
    l[r][c] = mine && r < jb ? A[(long)(jr + r) * lda + kr + c] : 0.0;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 16 * NB; t += 256) {
    double s = 0.0;
    if (upper) {
      const int r = q0 + t / NB, c = t % NB;  // (L_jk D_k)[r][c]
      for (int p = c; p < NB; ++p) s = fma(l[r][p], d[p][c], s);
      if (r < jb) A[(long)(kr + c) * lda + jr + r] = -s;
    } else {
      const int r = t / 16, c = q0 + t % 16;  // (D_j L_jk)[r][c]
      for (int p = 0; p <= r; ++p) s = fma(d[r][p], l[p][c], s);
      if (r < jb) A[(long)(jr + r) * lda + kr + c] = -s;
    }
  }
}

// The diagonal blocks transposed in place.
__global__ void __launch_bounds__(256) transpose_diag_kernel(double* __restrict__ A, int n, long lda) {
  const int k = blockIdx.x * NB, kb = min(NB, n - k);
  double* D = A + (long)k * lda + k;
  for (int t = threadIdx.x; t < kb * kb; t += 256) {
    const int i = t / kb, j = t % kb;
    if (j >= i) continue;
    const double v = D[(long)i * lda + j];
    D[(long)i * lda + j] = D[(long)j * lda + i];
    D[(long)j * lda + i] = v;
  }
}

// ---------------------------------------------------------------- point selection
// Greedy complete-pivoting Cholesky of X = (F F^T) o (F F^T), left-looking:
// only the diagonal d is kept up to date; each step forms one column, from
// the rows themselves, so X is never stored (m^2 doubles, and a product that
// took half of the time: 10.3 of 21.6 ms for 13824 points).  One launch a step:
// a block first reduces the previous launch's block maxima to the pivot (every
// block the same one), then forms the column for its 32 rows and the maximum of
// their new diagonals.  Its 8 warps take every eighth term of the two dot
// products (lanes along the rows of the transposed F and of L stored by
// columns, so loads are contiguous) and are added up in order.
// State on the device: d[m] (selected rows set to -1), L[want][m], val[t] =
// pivot value, sel[0] = steps taken, pv / pi = block maxima
// (two sets, alternating).

constexpr int PT_ROWS = 32, PT_WARPS = 8;

// Diagonals are compared as their bit patterns: those of non-negative doubles
// order like the numbers, a negative sentinel (-1) lies below them all, and an
// integer comparison takes a sixteenth of an FP64 one here.
__device__ __forceinline__ long long bits(double x) { return __double_as_longlong(x); }

// Largest value and its row (the lowest on ties) over a warp.
__device__ __forceinline__ void warp_argmax(long long& v, int& i) {
  for (int o = 16; o > 0; o >>= 1) {
    const long long ov = __shfl_xor_sync(0xffffffffu, v, o);
    const int oi = __shfl_xor_sync(0xffffffffu, i, o);
    if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
  }
}

// d[i] = X(i, i) and the block maxima; FT: the rows transposed, [N][m].
__global__ void __launch_bounds__(PT_ROWS) diag_init_kernel(const double* __restrict__ FT, int m, int N,
                                                            double* __restrict__ d,
                                                            long long* __restrict__ pv,
                                                            int* __restrict__ pi) {
  const int i = blockIdx.x * PT_ROWS + threadIdx.x;
  double s = 0.0;
  if (i < m)
    for (int k = 0; k < N; ++k) {
      const double f = FT[(long)k * m + i];
      s = fma(f, f, s);
    }
  if (i < m) d[i] = s * s;
  const bool in = i < m && s * s >= 0.0;  // a NaN is never a pivot
  long long v = in ? bits(s * s) : -1;
  int idx = in ? i : 0x7fffffff;
  warp_argmax(v, idx);
  if (threadIdx.x == 0) { pv[blockIdx.x] = v; pi[blockIdx.x] = idx; }
}

// Step t: pivot p = the largest d; stops when it is not above tol (tol_rel
// times the largest initial diagonal).  For every unselected row i,
// L[i][t] = ((F_i . F_p)^2 - sum_{s<t} L[i][s] L[p][s]) / sqrt(val[t]) and
// d[i] -= L[i][t]^2; the pivot row gets L[p][t] = sqrt(val[t]).
__global__ void __launch_bounds__(PT_ROWS * PT_WARPS) point_step_kernel(
    const double* __restrict__ F, const double* __restrict__ FT, int m, int N, int t, double tol_rel,
    int* __restrict__ sel, int32_t* __restrict__ piv, double* __restrict__ val,
    double* __restrict__ tol, double* __restrict__ L, double* __restrict__ d,
    long long* __restrict__ pv, int* __restrict__ pi) {
  __shared__ long long bv[PT_WARPS];
  __shared__ double rsp, sf[PT_WARPS][PT_ROWS], sl[PT_WARPS][PT_ROWS];
  __shared__ int bi[PT_WARPS];
  tc::dep_wait();
  tc::dep_launch();
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nb = gridDim.x;
  long long top = -1;
  int p = 0x7fffffff;
  for (int b = tid; b < nb; b += PT_ROWS * PT_WARPS) {
    const long long x = pv[(t & 1) * nb + b];
    const int q = pi[(t & 1) * nb + b];
    if (x > top || (x == top && q < p)) { top = x; p = q; }
  }
  warp_argmax(top, p);
  if (lane == 0) { bv[w] = top; bi[w] = p; }
  __syncthreads();
  top = bv[0];
  p = bi[0];
  for (int k = 1; k < PT_WARPS; ++k)
    if (bv[k] > top || (bv[k] == top && bi[k] < p)) { top = bv[k]; p = bi[k]; }
  const double v = top >= 0 ? __longlong_as_double(top) : -1.0;
  const double lim = t == 0 ? tol_rel * v : *tol;
  const bool stop = !(v > lim) || p >= m;
  if (blockIdx.x == 0 && tid == 0) {
    if (t == 0) *tol = lim;
    if (!stop) {
      piv[t] = p;
      val[t] = v;
      sel[0] = t + 1;
    }
  }
  if (stop) {
    // every block leaves here, in the later launches too
    if (tid == 0) { pv[((t + 1) & 1) * nb + blockIdx.x] = -1; pi[((t + 1) & 1) * nb + blockIdx.x] = 0x7fffffff; }
    return;
  }
  const int i = blockIdx.x * PT_ROWS + lane;
  const long ii = i < m ? i : m - 1;
  // 1 / sqrt(val): some 60 dependent FP64 instructions, beside the other warps' sums
  if (tid == PT_ROWS * PT_WARPS - 1) rsp = 1.0 / sqrt(v);
  const double di = w == 0 && i < m ? d[i] : -1.0;
  double f = 0.0, l = 0.0;
  const double* fp = F + (long)p * N;
#pragma unroll 4
  for (int k = w; k < N; k += PT_WARPS) f = fma(FT[(long)k * m + ii], __ldg(fp + k), f);
#pragma unroll 8
  for (int s = w; s < t; s += PT_WARPS) l = fma(L[(long)s * m + ii], L[(long)s * m + p], l);
  sf[w][lane] = f;
  sl[w][lane] = l;
  __syncthreads();
  if (w != 0) return;
  for (int k = 1; k < PT_WARPS; ++k) {
    f += sf[k][lane];
    l += sl[k][lane];
  }
  long long nd = -1;
  if (i < m) {
    if (i == p) {
      L[(long)t * m + i] = v * rsp;
      d[i] = -1.0;
    } else if (di >= 0.0) {
      const double x = (f * f - l) * rsp;
      L[(long)t * m + i] = x;
      const double dn = di - x * x;
      d[i] = dn;
      // a diagonal that rounding has taken below zero is out, as a selected row is
      if (dn >= 0.0) nd = bits(dn);
    }
  }
  int q = nd >= 0 ? i : 0x7fffffff;
  warp_argmax(nd, q);
  if (lane == 0) { pv[((t + 1) & 1) * nb + blockIdx.x] = nd; pi[((t + 1) & 1) * nb + blockIdx.x] = q; }
}

// out[c][r] = in[r][c] for rows x cols.
__global__ void transpose_kernel(const double* __restrict__ in, int rows, int cols, double* __restrict__ out) {
  __shared__ double tile[32][33];
  const long r0 = (long)blockIdx.x * 32, c0 = (long)blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += 8)
    if (r0 + i < rows && c0 + threadIdx.x < cols) tile[i][threadIdx.x] = in[(r0 + i) * cols + c0 + threadIdx.x];
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8)
    if (c0 + i < cols && r0 + threadIdx.x < rows) out[(c0 + i) * rows + r0 + threadIdx.x] = tile[threadIdx.x][i];
}

}  // namespace

cudaError_t select_points_f64(const double* F, int m, int N, int want, double tol_rel,
                              int32_t* piv, int* count, cudaStream_t s) {
  if (m <= 0 || want <= 0) {
    *count = 0;
    return cudaSuccess;
  }
  want = std::min(want, m);
  void* buf = nullptr;
  const int nb = (m + PT_ROWS - 1) / PT_ROWS;
  const size_t fb = (size_t)m * N * 8, lb = (size_t)m * want * 8;
  const size_t bytes = fb + lb + ((size_t)m + want + 2 + 2 * (size_t)nb) * 8 +
                       ((size_t)want + 2 * (size_t)nb + 4) * 4;
  cudaError_t e = cudaMallocAsync(&buf, bytes, s);
  if (e != cudaSuccess) return e;
  char* b = static_cast<char*>(buf);
  double* FT = reinterpret_cast<double*>(b);
  double* L = reinterpret_cast<double*>(b + fb);
  double* d = reinterpret_cast<double*>(b + fb + lb);
  double* val = d + m;
  double* tol = val + want;
  long long* pv = reinterpret_cast<long long*>(tol + 2);
  int* sel = reinterpret_cast<int*>(pv + 2 * nb);
  int* pi = sel + 4;
  int32_t* dpiv = pi + 2 * nb;
  e = cudaMemsetAsync(sel, 0, 16, s);
  if (e == cudaSuccess) {
    transpose_kernel<<<dim3((unsigned)nb, (unsigned)((N + 31) / 32)), dim3(32, 8), 0, s>>>(F, m, N, FT);
    diag_init_kernel<<<nb, PT_ROWS, 0, s>>>(FT, m, N, d, pv, pi);
    count_launch(2);
  }
  // each step may be launched while the one before it ends (tc::dep_wait)
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)nb);
  c.blockDim = dim3(PT_ROWS * PT_WARPS);
  c.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  for (int t = 0; e == cudaSuccess && t < want; ++t) {
    e = cudaLaunchKernelEx(&c, point_step_kernel, F, (const double*)FT, m, N, t, tol_rel, sel, dpiv, val,
                           tol, L, d, pv, pi);
    count_launch();
  }
  int got = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&got, sel, 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && got > 0)
    e = cudaMemcpyAsync(piv, dpiv, (size_t)got * 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaError_t e2 = cudaFreeAsync(buf, s);
  if (e == cudaSuccess) e = e2;
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  *count = got;
  return e;
}

cudaError_t cholesky_blocked_f64(double* A, int n, long lda, int* status, int* scale, int* wst,
                                 cudaStream_t s) {
  for (int k = 0; k < n; k += NB) {
    const int kb = std::min(NB, n - k);
    cudaError_t e = cholesky_step_f64(A, lda, k, kb, n, status, s);
    if (e != cudaSuccess) return e;
    if (k + kb < n) {
      const int rest = n - k - kb;
      // A22 -= L21 L21^T (the whole square; only its lower triangle is used)
      DGemm g{rest, rest, kb, A + (long)(k + kb) * lda + k, lda, false,
              A + (long)(k + kb) * lda + k, lda, true, A + (long)(k + kb) * lda + k + kb, lda,
              -1.0, nullptr, 0, 1, nullptr, 1.0, scale};
      g.status = wst;
      e = dgemm(g, s);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

// B := (L L^T)^{-1} B; L (lower) is overwritten.
cudaError_t cholesky_solve_f64(double* L, int n, long ldl, double* B, long ldb, long ncols,
                               int* scale, int* wst, cudaStream_t s) {
  const int nb = (n + NB - 1) / NB;
  const unsigned pairs = (unsigned)(nb * (nb - 1) / 2);
  invert_diag_kernel<<<(unsigned)nb, NB, 0, s>>>(L, n, ldl);
  count_launch();
  if (pairs > 0) {
    scale_blocks_kernel<<<dim3(pairs, NB / 16), 256, 0, s>>>(L, n, ldl, 1);
    scale_blocks_kernel<<<dim3(pairs, NB / 16), 256, 0, s>>>(L, n, ldl, 0);
    count_launch(2);
  }
  auto row = [&](int k, int k0, int k1) {  // B_k := L[k rows, k0:k1] B[k0:k1]
    DGemm g{std::min(NB, n - k), (int)ncols, k1 - k0, L + (long)k * ldl + k0, ldl, false,
            B + (long)k0 * ldb, ldb, false, B + (long)k * ldb, ldb, 1.0, nullptr, 0, 1, nullptr, 0.0,
            scale};
    g.status = wst;
    return dgemm(g, s);
  };
  for (int k = 0; k < n; k += NB) {
    cudaError_t e = row(k, 0, std::min(n, k + NB));
    if (e != cudaSuccess) return e;
  }
  transpose_diag_kernel<<<(unsigned)nb, 256, 0, s>>>(L, n, ldl);
  count_launch();
  for (int k = (nb - 1) * NB; k >= 0; k -= NB) {
    cudaError_t e = row(k, k, n);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t isdf_tables_f64(const double* phi, long ng, int N, const double* phig, const int* u, int na,
                            int grid, double L, double* Xgg, double* chi, double* V, double* W,
                            double* work, int* dig, size_t dig_ints, int* wst, int* status,
                            double* ridge_out, cudaStream_t s) {
  cudaError_t e;
  // scratch of the tensor-core products: W until W itself is formed, when that is the
  // larger (more functions to a Poisson pass)
  int* scale = dig;
  size_t ints = dig_ints;
  if (2 * (size_t)na * na > ints) {
    scale = reinterpret_cast<int*>(W);
    ints = 2 * (size_t)na * na;
  }
  auto gram = [&]() {
    DGemm g{na, na, N, phig, N, false, phig, N, true, Xgg, na, 1.0, nullptr, 0, 0, work};
    g.scale = scale;
    g.status = wst;
    g.sym = true;
    cudaError_t r = dgemm(g, s);
    if (r != cudaSuccess) return r;
    square_kernel<<<nblocks((long)na * na), 256, 0, s>>>(Xgg, na, na, na);
    count_launch();
    return cudaGetLastError();
  };
  // X_gR = (Phi_g Phi^T) o (Phi_g Phi^T) into chi
  {
    DGemm g{na, (int)ng, N, phig, N, false, phi, N, true, chi, ng, 1.0, nullptr, 0, 0, work};
    g.scale = scale;
    g.status = wst;
    e = dgemm(g, s);
    if (e != cudaSuccess) return e;
    square_kernel<<<nblocks((long)na * ng), 256, 0, s>>>(chi, na, ng, ng);
    count_launch();
  }
  e = gram();
  if (e != cudaSuccess) return e;
  double ridge = 0.0;
  int st = 0;
  e = cudaMemsetAsync(status, 0, 4, s);
  if (e == cudaSuccess) e = cholesky_blocked_f64(Xgg, na, na, status, scale, wst, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&st, status, 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  if (st != 0) {  // the factorisation failed: add the ridge and factor again
    e = gram();
    if (e != cudaSuccess) return e;
    std::vector<double> d(na);
    std::vector<int> hu(na);
    e = cudaMemcpyAsync(hu.data(), u, (size_t)na * 4, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    copy_diag_kernel<<<nblocks(na), 256, 0, s>>>(Xgg, na, na, work);
    count_launch();
    e = cudaMemcpyAsync(d.data(), work, (size_t)na * 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    double tr = 0.0;
    for (int i = 0; i < na; ++i) tr += std::ldexp(d[i], 4 * hu[i]);
    ridge = 1e-14 * tr / na;
    add_diag_kernel<<<nblocks(na), 256, 0, s>>>(Xgg, na, na, ridge, u);
    count_launch();
    e = cudaMemsetAsync(status, 0, 4, s);
    if (e == cudaSuccess) e = cholesky_blocked_f64(Xgg, na, na, status, scale, wst, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&st, status, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    if (st != 0) return cudaErrorInvalidValue;  // X_gg is not positive definite
  }
  if (ridge_out) *ridge_out = ridge;
  // chi = X_gg^{-1} X_gR
  e = cholesky_solve_f64(Xgg, na, na, chi, ng, ng, scale, wst, s);
  if (e != cudaSuccess) return e;
  // V = Pois(chi) in batches of functions (the scratch holds one)
  {
    const long g3 = (long)grid * grid * grid;
    long nf = std::max<long>(1, std::min<long>(na, (1L << 28) / (g3 * 8)));
    // the row maxima of a batch go into the scratch of the products
    nf = std::max<long>(1, std::min<long>(nf, ((long)std::min<size_t>(ints, 1u << 30) - grid - 8) /
                                                  ((long)grid * grid)));
    void* buf = nullptr;
    e = cudaMallocAsync(&buf, ((size_t)nf * g3 + poisson_table_elems(grid)) * 8, s);
    if (e != cudaSuccess) return e;
    double* tmp = static_cast<double*>(buf);
    double* tab = tmp + nf * g3;
    e = poisson_tables_f64(grid, L, tab, s);
    for (long r0 = 0; e == cudaSuccess && r0 < na; r0 += nf)
      e = poisson_f64(chi + r0 * ng, V + r0 * ng, tmp, std::min<long>(nf, na - r0), grid, tab, scale,
                      ints, wst, s);
    cudaError_t e2 = cudaFreeAsync(buf, s);
    if (e == cudaSuccess) e = e2;
    if (e != cudaSuccess) return e;
  }
  // W = V chi^T, symmetrised
  {
    DGemm g{na, na, (int)ng, V, ng, false, chi, ng, true, W, na, 1.0, nullptr, 0, 0, work};
    g.scale = dig;
    g.status = wst;
    e = dgemm(g, s);
    if (e == cudaSuccess) e = symmetrize_f64(W, na, s);
  }
  return e;
}

}  // namespace xk
