// FP64 kernels of the exchange build: a tiled SIMT DGEMM with a Hadamard
// epilogue and deterministic split-K, row gathers, the K assembly, the E_x
// reduction, and the small dense FP64 factorisations of the occ-RI K_ij.
//
// On GB300 FP64 runs on the CUDA cores at a small fraction of the tensor
// rate, so a contraction here is bound by the DFMA pipe; the tiles only need
// enough register reuse to keep that pipe fed.  Products of 2e7 multiply-adds and
// more, nearly all of the work, go to the tensor cores instead (xk_digits.cu).
#include "xk_internal.h"

#include <algorithm>
#include <cmath>
#include <vector>

namespace xk {

std::atomic<uint64_t> g_launches{0};

namespace {

constexpr int BM = 64, BN = 64, BK = 16, TPB = 256;

template <bool TA, bool TB, bool HAD>
__global__ void __launch_bounds__(TPB) dgemm_kernel(DGemm g, int kchunk, const int* only_if) {
  // behind a product on the tensor cores: only when that one was left out (a few
  // blocks then walk the tiles; a grid of all of them took 25 us to start and end)
  const int left_out = only_if ? *only_if : 1;
  if (!left_out) return;
  // the maxima it left are not C's: rows that are not split, so that products of C
  // take this kernel too
  if (only_if && g.rmax) {
    for (long i = blockIdx.x * (long)TPB + threadIdx.x; i < g.M; i += (long)gridDim.x * TPB) g.rmax[i] = 0x7ff00000;
    for (long i = blockIdx.x * (long)TPB + threadIdx.x; i < g.N; i += (long)gridDim.x * TPB) g.cmax[i] = 0x7ff00000;
  }
  const long gx = (g.N + BN - 1) / BN, gy = (g.M + BM - 1) / BM, ntiles = gx * gy * g.ksplit;
  __shared__ double As[BK][BM + 1];
  __shared__ double Bs[BK][BN + 1];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  for (long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
  const long bz = tile / (gx * gy);
  const long m0 = (tile / gx % gy) * BM, n0 = (tile % gx) * BN;
  const long kbeg = bz * kchunk, kend = min((long)g.K, kbeg + kchunk);
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;

  for (long k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int e = 0; e < (BM * BK) / TPB; ++e) {
      const int l = tid + TPB * e;
      int m, k;
      if (TA) { k = l / BM; m = l % BM; } else { m = l / BK; k = l % BK; }
      const long gm = m0 + m, gk = k0 + k;
      double v = 0.0;
      if (gm < g.M && gk < kend) v = TA ? g.A[gk * g.lda + gm] : g.A[gm * g.lda + gk];
      As[k][m] = v;
    }
#pragma unroll
    for (int e = 0; e < (BN * BK) / TPB; ++e) {
      const int l = tid + TPB * e;
      int n, k;
      if (TB) { n = l / BK; k = l % BK; } else { k = l / BN; n = l % BN; }
      const long gn = n0 + n, gk = k0 + k;
      double v = 0.0;
      if (gn < g.N && gk < kend) v = TB ? g.B[gn * g.ldb + gk] : g.B[gk * g.ldb + gn];
      Bs[k][n] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long m = m0 + ty + 16 * i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const long n = n0 + tx + 16 * j;
      if (n >= g.N) continue;
      if (g.ksplit > 1) {
        g.work[(bz * g.M + m) * g.N + n] = acc[i][j];
      } else {
        const long q = g.nbatch > 0 ? n / g.nbatch : 0;  // batch of the column
        const long at = m * g.ldc + n + q * g.cskip;
        double v = g.alpha * acc[i][j];
        if (HAD) v *= g.H[m * g.ldh + n - q * g.nbatch];
        if (g.beta != 0.0) v += g.beta * g.C[at];
        // a tensor-core product that gave up half-way has changed C already (it is reported
        // by way of DGemm::status)
        if ((g.beta != 0.0 || in_place(g)) && only_if && left_out == 2) v = nan("");
        g.C[at] = v;
      }
    }
  }
  }
}

// C = alpha * sum_z work[z] (o H), z in increasing order.
__global__ void splitk_reduce_kernel(DGemm g) {
  const long total = (long)g.M * g.N;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
       t += (long)gridDim.x * blockDim.x) {
    const long m = t / g.N, n = t % g.N;
    if (g.sym && n < m) continue;
    double s = 0.0;
    for (int z = 0; z < g.ksplit; ++z) s += g.work[(long)z * total + t];
    double v = g.alpha * s;
    if (g.H) v *= g.H[m * g.ldh + n];
    if (g.beta != 0.0) v += g.beta * g.C[m * g.ldc + n];
    g.C[m * g.ldc + n] = v;
    if (g.sym) g.C[n * g.ldc + m] = v;
  }
}

int choose_ksplit(int M, int N, int K) {
  const long tiles = (long)((M + BM - 1) / BM) * ((N + BN - 1) / BN);
  const long target = 4L * 152;  // about four waves of CTAs over 152 SMs
  if (tiles >= target) return 1;
  long ks = (target + tiles - 1) / tiles;
  ks = std::min<long>(ks, std::max(1, K / 64));
  return (int)std::max<long>(1, std::min<long>(ks, 64));
}

template <bool TA, bool TB>
cudaError_t launch_tt(const DGemm& g, int kchunk, const int* only_if, cudaStream_t s) {
  const long tiles = (long)((g.N + BN - 1) / BN) * ((g.M + BM - 1) / BM) * g.ksplit;
  const unsigned grid = (unsigned)(only_if ? std::min<long>(tiles, 152 * 4) : tiles);
  if (g.H && g.ksplit == 1)
    dgemm_kernel<TA, TB, true><<<grid, TPB, 0, s>>>(g, kchunk, only_if);
  else
    dgemm_kernel<TA, TB, false><<<grid, TPB, 0, s>>>(g, kchunk, only_if);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

int dgemm_ksplit(int M, int N, int K) {
  int ks = choose_ksplit(M, N, K);
  int kchunk = (K + ks - 1) / ks;
  kchunk = ((kchunk + BK - 1) / BK) * BK;
  if (kchunk <= 0) kchunk = BK;
  return std::max(1, (K + kchunk - 1) / kchunk);
}

cudaError_t dgemm(const DGemm& gin, cudaStream_t s) {
  DGemm g = gin;
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (g.nbatch > 0) g.ksplit = 1;  // batched columns are stored unsplit
  const bool digits = digit_gemm_wanted(g);
  if (digits)
    g.ksplit = digit_ksplit(g.M, g.N, g.K, g.sym,
                            !g.work || g.nbatch > 0 ? 1 : g.ksplit > 0 ? g.ksplit : dgemm_ksplit(g.M, g.N, g.K));
  if (g.ksplit <= 0) g.ksplit = choose_ksplit(g.M, g.N, g.K);
  if (g.ksplit > 1 && !g.work) g.ksplit = 1;
  int kchunk = (g.K + g.ksplit - 1) / g.ksplit;
  const int unit = digits ? 32 : BK;
  kchunk = ((kchunk + unit - 1) / unit) * unit;
  if (kchunk <= 0) kchunk = BK;
  g.ksplit = std::max(1, (g.K + kchunk - 1) / kchunk);
  cudaError_t e = digits ? digit_gemm(g, g.ksplit, kchunk, s) : cudaSuccess;
  if (e != cudaSuccess) return e;
  const int* only_if = digits ? g.scale : nullptr;
  if (!g.transA && !g.transB) e = launch_tt<false, false>(g, kchunk, only_if, s);
  else if (g.transA && !g.transB) e = launch_tt<true, false>(g, kchunk, only_if, s);
  else if (!g.transA && g.transB) e = launch_tt<false, true>(g, kchunk, only_if, s);
  else e = launch_tt<true, true>(g, kchunk, only_if, s);
  if (e != cudaSuccess || g.ksplit == 1) return e;
  const long total = (long)g.M * g.N;
  const int blocks = (int)std::min<long>((total + 255) / 256, 152L * 16);
  splitk_reduce_kernel<<<blocks, 256, 0, s>>>(g);
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------

__global__ void gather_rows_kernel(const double* __restrict__ in, long ld_in,
                                   const int32_t* __restrict__ idx, int rows, int cols,
                                   double* __restrict__ out, long ld_out, const int* __restrict__ re) {
  const long total = (long)rows * cols;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
       t += (long)gridDim.x * blockDim.x) {
    const long r = t / cols, c = t % cols;
    const double v = in[(long)idx[r] * ld_in + c];
    out[r * ld_out + c] = re ? scalbn(v, -re[r]) : v;
  }
}

cudaError_t gather_rows_f64(const double* in, long ld_in, const int32_t* idx, int rows, int cols,
                            double* out, long ld_out, cudaStream_t s, const int* re) {
  const long total = (long)rows * cols;
  if (total == 0) return cudaSuccess;
  const int blocks = (int)std::min<long>((total + 255) / 256, 152L * 16);
  gather_rows_kernel<<<blocks, 256, 0, s>>>(in, ld_in, idx, rows, cols, out, ld_out, re);
  count_launch();
  return cudaGetLastError();
}

__device__ __forceinline__ int exponent_of(int hi, int limit) {  // hi: high word of |x|
  return hi <= 0 || hi >= 0x7ff00000 ? 0 : max(-limit, min(limit, (hi >> 20) - 1022));
}

// High word of the largest |x| of a row, over a warp.
__device__ __forceinline__ int row_max_hi(const double* __restrict__ row, int cols) {
  int m = 0;
  for (int c = threadIdx.x & 31; c < cols; c += 32) m = max(m, __double2hiint(row[c]) & 0x7fffffff);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  return m;
}

// One warp per row.
__global__ void row_exponents_kernel(const double* __restrict__ p, long ld, const int32_t* __restrict__ idx,
                                     int rows, int cols, int limit, int* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const long r = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const int m = row_max_hi(p + (idx ? (long)idx[r] : r) * ld, cols);
  if (lane == 0) out[r] = exponent_of(m, limit);
}

cudaError_t row_exponents_f64(const double* p, long ld, const int32_t* idx, int rows, int cols, int limit,
                              int* out, cudaStream_t s) {
  row_exponents_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(p, ld, idx, rows, cols, limit, out);
  count_launch();
  return cudaGetLastError();
}

// One warp per row.
__global__ void balance_rows_kernel(const double* __restrict__ A, const double* __restrict__ B, int rows,
                                    int cols, double* __restrict__ A2, double* __restrict__ B2) {
  const long r = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const double *a = A + r * cols, *b = B + r * cols;
  const int ma = row_max_hi(a, cols), mb = row_max_hi(b, cols), big = max(ma, mb);
  const int e = ma == 0 || mb == 0 || big >= 0x7ff00000
                    ? 0 : (exponent_of(mb, 1022) - exponent_of(ma, 1022)) >> 1;
  for (int c = threadIdx.x & 31; c < cols; c += 32) {
    A2[r * cols + c] = scalbn(a[c], e);
    B2[r * cols + c] = scalbn(b[c], -e);
  }
}

cudaError_t balance_rows_f64(const double* A, const double* B, int rows, int cols, double* A2, double* B2,
                             cudaStream_t s) {
  balance_rows_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(A, B, rows, cols, A2, B2);
  count_launch();
  return cudaGetLastError();
}

__global__ void sub_kernel(const int* a, const int* b, int n, int* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = a[i] - b[i];
}

cudaError_t sub_i32(const int* a, const int* b, int n, int* out, cudaStream_t s) {
  sub_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, b, n, out);
  count_launch();
  return cudaGetLastError();
}

// One thread per column and chunk of rows (blockIdx.y).
__global__ void col_max_kernel(const double* __restrict__ p, long ld, long rows, int cols, long chunk,
                               int* __restrict__ out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  const long r0 = blockIdx.y * chunk, r1 = min(rows, r0 + chunk);
  int m = 0;
  for (long r = r0; r < r1; ++r) m = max(m, __double2hiint(p[r * ld + c]) & 0x7fffffff);
  atomicMax(out + c, m);
}

__global__ void exponents_kernel(int* __restrict__ x, int n, int limit) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = exponent_of(x[i], limit);
}

cudaError_t col_exponents_f64(const double* p, long ld, long rows, int cols, int limit, int* out,
                              cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, (size_t)cols * 4, s);
  if (e != cudaSuccess) return e;
  const long chunk = std::max(64L, (rows + 1023) / 1024);
  col_max_kernel<<<dim3((unsigned)((cols + 127) / 128), (unsigned)((rows + chunk - 1) / chunk)), 128, 0, s>>>(
      p, ld, rows, cols, chunk, out);
  exponents_kernel<<<(unsigned)((cols + 255) / 256), 256, 0, s>>>(out, cols, limit);
  count_launch(2);
  return cudaGetLastError();
}

// x 2^e as scalbn gives it: in integers where x and the result are normal (scalbn and FP64
// products took 1484 us of the 1755 x 91125 V, this with four loads in flight 426).
__device__ __forceinline__ double times_pow2(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  if ((unsigned)(ex - 1) < 2046u && (unsigned)(ex + e - 1) < 2046u)
    return __hiloint2double(hi + e * (1 << 20), __double2loint(x));
  return scalbn(x, e);
}

// I: an index type that holds rows x cols and a few grids' threads beyond.
template <class I>
__global__ void scale_kernel(const double* src, double* dst, I rows, I cols, const int* __restrict__ re,
                             int rm, const int* __restrict__ ce, int cm, double f) {
  const I total = rows * cols, step = (I)gridDim.x * blockDim.x;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += 4 * step) {
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = t + u * step < total ? src[t + u * step] : 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const I at = t + u * step;
      if (at >= total) break;
      const I r = at / cols, c = at - r * cols;
      const double x = times_pow2(v[u], (re ? rm * re[r] : 0) + (ce ? cm * ce[c] : 0));
      dst[at] = f == 1.0 ? x : f * x;
    }
  }
}

cudaError_t scale_f64(const double* src, double* dst, long rows, long cols, const int* re, int rm,
                      const int* ce, int cm, cudaStream_t s, double f) {
  const long total = rows * cols;
  if (total == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)std::min<long>((total + 255) / 256, 152L * 16);
  if (total < 1L << 31)  // (4 grids are 2^21.3 threads)
    scale_kernel<unsigned><<<blocks, 256, 0, s>>>(src, dst, (unsigned)rows, (unsigned)cols, re, rm, ce, cm, f);
  else
    scale_kernel<long><<<blocks, 256, 0, s>>>(src, dst, rows, cols, re, rm, ce, cm, f);
  count_launch();
  return cudaGetLastError();
}

__global__ void assemble_k_kernel(const double* __restrict__ L1, const double* __restrict__ L2,
                                  const double* __restrict__ L3, int n, int N, double dV,
                                  const int* __restrict__ ce, double* __restrict__ K) {
  const long total = (long)n * N;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
       t += (long)gridDim.x * blockDim.x) {
    const long mu = t / n, i = t % n;
    const long src = i * N + mu;
    K[t] = dV * scalbn((L1[src] + L2[src]) - L3[src], ce[mu]);  // (in this order: K's own range)
  }
}

cudaError_t assemble_k_f64(const double* L1, const double* L2, const double* L3, int n, int N,
                           double dV, const int* ce, double* K, cudaStream_t s) {
  const long total = (long)n * N;
  const int blocks = (int)std::min<long>((total + 255) / 256, 152L * 8);
  assemble_k_kernel<<<blocks, 256, 0, s>>>(L1, L2, L3, n, N, dV, ce, K);
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Deterministic two-stage reduction: block b sums the contiguous chunk b in a
// fixed per-thread order and a fixed tree; one block then sums the partials.

constexpr int RED_BLOCKS = 512, RED_TPB = 256;

__device__ double block_sum(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  return sh[0];
}

__global__ void dot_stage1(const double* __restrict__ a, const double* __restrict__ b, long len,
                           double* __restrict__ part) {
  __shared__ double sh[RED_TPB];
  const long chunk = (len + gridDim.x - 1) / gridDim.x;
  const long beg = blockIdx.x * chunk, end = min(len, beg + chunk);
  double s = 0.0;
  for (long t = beg + threadIdx.x; t < end; t += blockDim.x) s = fma(a[t], b[t], s);
  const double tot = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__global__ void dot_stage2(const double* __restrict__ part, int np, double* out) {
  __shared__ double sh[RED_TPB];
  double s = 0.0;
  for (int t = threadIdx.x; t < np; t += blockDim.x) s += part[t];
  const double tot = block_sum(s, sh);
  if (threadIdx.x == 0) *out = -tot;
}

size_t reduce_work_elems() { return RED_BLOCKS; }

cudaError_t neg_dot_f64(const double* a, const double* b, long len, double* work, double* out,
                        cudaStream_t s) {
  dot_stage1<<<RED_BLOCKS, RED_TPB, 0, s>>>(a, b, len, work);
  dot_stage2<<<1, RED_TPB, 0, s>>>(work, RED_BLOCKS, out);
  count_launch(2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Coulomb J on the grid: density, Poisson solve, and J = dV Phi^T diag(v) Phi.

namespace {
int blocks_of(long total) { return (int)std::max<long>(1, std::min<long>((total + 255) / 256, 152L * 16)); }
}  // namespace

// rho[R] = sum_i psi[R][i]^2.
__global__ void density_kernel(const double* __restrict__ psi, long ng, int n, double* __restrict__ rho) {
  for (long r = blockIdx.x * (long)blockDim.x + threadIdx.x; r < ng;
       r += (long)gridDim.x * blockDim.x) {
    const double* row = psi + r * n;
    double s = 0.0;
    for (int i = 0; i < n; ++i) s = fma(row[i], row[i], s);
    rho[r] = s;
  }
}

// Poisson solves.  On a cubic grid 4 pi / G^2 depends on the squares of the three
// frequencies only, and the cosine and the sine of one |m| share it: the solve is
// diagonal in the product of the axes' real Fourier bases (orthonormal columns
// 1/sqrt(g), sqrt(2/g) cos, sqrt(2/g) sin, and (-1)^j / sqrt(g) for even g), with
// no complex arithmetic.  Six passes, each a product of the g x g basis with
// the fastest axis of every function that leaves that axis the slowest:
//   in [f][p][j], p over the other two axes  ->  out [f][k][p] = sum_j B[k][j] in[f][p][j],
// three passes into the basis (the third multiplies by 4 pi / G^2), three back,
// after which the axes are in order again.  Many functions are one large product
// for the tensor cores (xk_digits.cu); a single one (the Coulomb build) takes
// axis_kernel.  1053 functions of 45^3: 6 passes of FP64 complex DFTs on two
// functions each took 112 ms.
//
// Tables: [0, g^2) forward B[k][j], [g^2, 2 g^2) its transpose, then 4 pi / G^2
// as [kx][ky][kz].

__global__ void poisson_kernel_table(double* __restrict__ lam, int g, double L) {
  const long g3 = (long)g * g * g;
  const double w = 6.283185307179586 / L;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < g3;
       t += (long)gridDim.x * blockDim.x) {
    // basis function k belongs to the frequency (k + 1) / 2
    const int m0 = ((int)(t / ((long)g * g)) + 1) / 2, m1 = ((int)((t / g) % g) + 1) / 2,
              m2 = ((int)(t % g) + 1) / 2;
    const double g2 = w * w * ((double)m0 * m0 + (double)m1 * m1 + (double)m2 * m2);
    lam[t] = g2 > 0.0 ? 12.566370614359172 / g2 : 0.0;
  }
}

size_t poisson_table_elems(int g) { return 2 * (size_t)g * g + (size_t)g * g * g; }

cudaError_t poisson_tables_f64(int g, double L, double* tab, cudaStream_t s) {
  std::vector<double> b(2 * (size_t)g * g), c(g), d(g);
  const long double tau = 6.283185307179586476925286766559L, rg = sqrtl((long double)g);
  for (int r = 0; r < g; ++r) {  // sqrt(2/g) cos, sin of 2 pi r / g
    c[r] = (double)(sqrtl(2.0L) * cosl(tau * r / g) / rg);
    d[r] = (double)(sqrtl(2.0L) * sinl(tau * r / g) / rg);
  }
  for (int k = 0; k < g; ++k)
    for (int j = 0; j < g; ++j) {
      const int m = (k + 1) / 2, r = (int)(((long)m * j) % g);
      double v = (k & 1) ? c[r] : d[r];
      if (k == 0) v = (double)(1.0L / rg);
      else if (2 * m == g) v = (double)(((j & 1) ? -1.0L : 1.0L) / rg);
      b[(size_t)k * g + j] = b[(size_t)g * g + (size_t)j * g + k] = v;
    }
  cudaError_t e = cudaMemcpyAsync(tab, b.data(), b.size() * 8, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  poisson_kernel_table<<<blocks_of((long)g * g * g), 256, 0, s>>>(tab + 2 * (size_t)g * g, g, L);
  count_launch();
  e = cudaGetLastError();
  return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}

// One pass for few functions: a thread forms two outputs k of one (f, p) (four left a
// third of the SMs with twice the others' work: 22 us at 45^3 against 15); the
// lanes' rows of `in` stay in L1 over the g terms.  Bound by the FP64 pipe.
__global__ void __launch_bounds__(128) axis_kernel(const double* __restrict__ in, double* __restrict__ out,
                                                   long rows, int g, const double* __restrict__ B,
                                                   const double* __restrict__ lam) {
  const long r = (long)blockIdx.x * 32 + threadIdx.x, g2 = (long)g * g;
  const int k0 = 2 * (blockIdx.y * blockDim.y + threadIdx.y);
  if (r >= rows || k0 >= g) return;
  const double* x = in + r * g;
  const double* b[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) b[i] = B + (long)min(k0 + i, g - 1) * g;
  double acc[2] = {0.0, 0.0};
#pragma unroll 8
  for (int j = 0; j < g; ++j) {
    const double v = x[j];
#pragma unroll
    for (int i = 0; i < 2; ++i) acc[i] = fma(__ldg(b[i] + j), v, acc[i]);
  }
  const long f = r / g2, p = r - f * g2;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (k0 + i < g) {
      const double v = lam ? acc[i] * lam[(k0 + i) * g2 + p] : acc[i];
      out[f * g2 * g + (k0 + i) * g2 + p] = v;
    }
}

cudaError_t poisson_f64(const double* in, double* out, double* tmp, long nf, int g,
                        const double* tab, int* scale, size_t scale_ints, int* wst, cudaStream_t s) {
  const long g2 = (long)g * g;
  const double* lam = tab + 2 * g2;
  const double* src = in;
  for (int pass = 0; pass < 6; ++pass) {
    double* dst = (pass & 1) ? out : tmp;
    const double* B = tab + (pass < 3 ? 0 : g2);
    const double* H = pass == 2 ? lam : nullptr;
    DGemm q{g, (int)(nf * g2), g, B, g, false, src, g, true, dst, g2, 1.0, H, g2, 1, nullptr};
    q.nbatch = (int)g2;
    q.cskip = g2 * (g - 1);
    q.scale = scale && scale_ints >= digit_scale_ints(q.M, q.N) ? scale : nullptr;
    q.status = wst;
    cudaError_t e;
    if (digit_gemm_wanted(q)) {
      e = dgemm(q, s);
    } else {
      axis_kernel<<<dim3((unsigned)((nf * g2 + 31) / 32), (unsigned)((g + 7) / 8)), dim3(32, 4), 0, s>>>(
          src, dst, nf * g2, g, B, H);
      count_launch();
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    src = dst;
  }
  return cudaSuccess;
}

// out[R][nu] = v[R] phi[R][nu].
__global__ void potential_rows_kernel(const double* __restrict__ v, const double* __restrict__ phi,
                                      long ng, int N, double* __restrict__ out) {
  const long count = ng * N;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < count;
       t += (long)gridDim.x * blockDim.x)
    out[t] = v[t / N] * phi[t];
}

__global__ void dot_scaled_stage2(const double* __restrict__ part, int np, double scale, double* out) {
  __shared__ double sh[RED_TPB];
  double s = 0.0;
  for (int t = threadIdx.x; t < np; t += blockDim.x) s += part[t];
  const double tot = block_sum(s, sh);
  if (threadIdx.x == 0) *out = scale * tot;
}

cudaError_t density_f64(const double* psi, long ng, int n, double* rho, cudaStream_t s) {
  density_kernel<<<blocks_of(ng), 256, 0, s>>>(psi, ng, n, rho);
  count_launch();
  return cudaGetLastError();
}

cudaError_t potential_rows_f64(const double* v, const double* phi, long ng, int N, double* out,
                               cudaStream_t s) {
  potential_rows_kernel<<<blocks_of(ng * N), 256, 0, s>>>(v, phi, ng, N, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t dot_f64(const double* a, const double* b, long len, double scale, double* work,
                    double* out, cudaStream_t s) {
  dot_stage1<<<RED_BLOCKS, RED_TPB, 0, s>>>(a, b, len, work);
  dot_scaled_stage2<<<1, RED_TPB, 0, s>>>(work, RED_BLOCKS, scale, out);
  count_launch(2);
  return cudaGetLastError();
}

// Full K: K[mu][nu] = dV ((Y[mu][nu] + Y[nu][mu] - Z[mu][nu]) 2^(ce[mu] + ce[nu])) (N x N).
__global__ void assemble_full_kernel(const double* __restrict__ Y, const double* __restrict__ Z,
                                     int N, double dV, const int* __restrict__ ce,
                                     double* __restrict__ K) {
  const long count = (long)N * N;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < count;
       t += (long)gridDim.x * blockDim.x) {
    const long mu = t / N, nu = t % N;
    K[t] = dV * scalbn((Y[t] + Y[nu * N + mu]) - Z[t], ce[mu] + ce[nu]);
  }
}

cudaError_t assemble_full_f64(const double* Y, const double* Z, int N, double dV, const int* ce,
                              double* K, cudaStream_t s) {
  const long count = (long)N * N;
  const int blocks = (int)std::min<long>((count + 255) / 256, 152L * 16);
  assemble_full_kernel<<<std::max(blocks, 1), 256, 0, s>>>(Y, Z, N, dV, ce, K);
  count_launch();
  return cudaGetLastError();
}

// E_x from its closed form, -dV (2 sum w_A p_A^2 - sum w_C p_C^2) (Eq. exoccri
// contracted with C: line 1 and line 2 each give sum V o P o P, line 3 gives
// sum W o Q o Q).  Stage 1: half of the blocks sum the V term, the other
// half the W term; stage 2 adds the per-block sums in a fixed order.
__global__ void wsq_stage1(const double* __restrict__ wa, const double* __restrict__ pa, long la,
                           const double* __restrict__ wc, const double* __restrict__ pc, long lc,
                           double* __restrict__ part) {
  __shared__ double sh[RED_TPB];
  const int half = gridDim.x / 2;
  const bool c = (int)blockIdx.x >= half;
  const double* w = c ? wc : wa;
  const double* p = c ? pc : pa;
  const long len = c ? lc : la;
  const long blk = c ? blockIdx.x - half : blockIdx.x;
  const long chunk = (len + half - 1) / half;
  const long beg = blk * chunk, end = min(len, beg + chunk);
  double s = 0.0;
  for (long t = beg + threadIdx.x; t < end; t += blockDim.x) s = fma(w[t] * p[t], p[t], s);
  const double tot = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__global__ void closed_ex_stage2(const double* __restrict__ part, int half, double dV, double* out) {
  __shared__ double sa[RED_TPB], sc[RED_TPB];
  double a = 0.0, c = 0.0;
  for (int t = threadIdx.x; t < half; t += blockDim.x) {
    a += part[t];
    c += part[half + t];
  }
  sa[threadIdx.x] = a;
  sc[threadIdx.x] = c;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sa[threadIdx.x] += sa[threadIdx.x + w];
      sc[threadIdx.x] += sc[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = -dV * (2.0 * sa[0] - sc[0]);
}

cudaError_t closed_form_ex_f64(const double* V, const double* P, long lenA, const double* W,
                               const double* Q, long lenC, double dV, double* work, double* out,
                               cudaStream_t s) {
  wsq_stage1<<<RED_BLOCKS, RED_TPB, 0, s>>>(V, P, lenA, W, Q, lenC, work);
  closed_ex_stage2<<<1, RED_TPB, 0, s>>>(work, RED_BLOCKS / 2, dV, out);
  count_launch(2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Small dense FP64 factorisations (n <= a few hundred; one block each).

__global__ void symmetrize_kernel(double* A, int n) {
  const long total = (long)n * n;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
       t += (long)gridDim.x * blockDim.x) {
    const long i = t / n, j = t % n;
    if (j > i) {
      const double v = 0.5 * (A[i * n + j] + A[j * n + i]);
      A[i * n + j] = v;
      A[j * n + i] = v;
    }
  }
}

cudaError_t symmetrize_f64(double* A, int n, cudaStream_t s) {
  symmetrize_kernel<<<64, 256, 0, s>>>(A, n);
  count_launch();
  return cudaGetLastError();
}

// Small products and factorisations (the occ-RI K_ij, the blocks of the ISDF
// Cholesky).  One SM forms 2 FP64 multiply-adds a clock, so even these want many
// SMs: tiles are kept at a few thousand multiply-adds.

// Kij[i][j] = sum_mu (C[mu][i] K[mu][j] + C[mu][j] K[mu][i]) / 2.  A block forms the
// 4 x 4 outputs of one tile pair on or above the diagonal, 16 threads to an output's mu
// (8 x 8 tiles put the whole product on 28 SMs at n = 54: 27 us).  The tiled product (five
// blocks of 64 x 64), its split sum and the symmetrisation took 97 us.
constexpr int KT = 4, KS = 16;
__global__ void __launch_bounds__(KT * KT * KS) kij_kernel(const double* __restrict__ C,
                                                          const double* __restrict__ K, int N, int n,
                                                          double* __restrict__ Kij) {
  __shared__ double part[KS][KT * KT];
  if (blockIdx.x > blockIdx.y) return;
  const int o = threadIdx.x % (KT * KT), sl = threadIdx.x / (KT * KT);
  const int i = blockIdx.x * KT + o / KT, j = blockIdx.y * KT + o % KT;
  double u = 0.0, v = 0.0;
  if (i < n && j < n) {
#pragma unroll 4
    for (long mu = sl; mu < N; mu += KS) {
      const double *c = C + mu * n, *k = K + mu * n;
      u = fma(c[i], k[j], u);
      v = fma(c[j], k[i], v);
    }
  }
  part[sl][o] = 0.5 * u + 0.5 * v;  // halved first: sums of 2 K_ij may overflow where K_ij does not
  __syncthreads();
  if (sl != 0 || i >= n || j >= n) return;
  double s = part[0][o];
  for (int w = 1; w < KS; ++w) s += part[w][o];
  Kij[(long)i * n + j] = Kij[(long)j * n + i] = s;
}

cudaError_t kij_f64(const double* C, const double* K, int N, int n, double* Kij, cudaStream_t s) {
  const unsigned t = (unsigned)((n + KT - 1) / KT);
  kij_kernel<<<dim3(t, t), KT * KT * KS, 0, s>>>(C, K, N, n, Kij);
  count_launch();
  return cudaGetLastError();
}

// 1 / d by Newton's iteration from the hardware's approximation (about 20 bits): every
// FP64 instruction of a warp takes the SM's FP64 pipe for 16 cycles, a division some 30.
__device__ __forceinline__ double fast_recip(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  r = fma(r, fma(-d, r, 1.0), r);
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}

// In-place Cholesky factor L (lower) of the kb x kb block at (k, k) of A by one block of
// 256 threads, the triangle in registers: thread t owns the elements e = t, t + 256, ... of
// an enumeration in which the trailing triangles of all columns are prefixes, so no lane
// idles.  Column c: its owners publish it (unscaled), two warps divide it by the pivot, then
// a[i][j] -= a[i][c] (a[j][c] / a[c][c]); the scaling follows at the end.  *status gets the column (from 1) of the first pivot that is not positive; that pivot
// counts as 1.  The matrix in global memory, two barriers, a square root and a division in
// sequence took 87 us at kb = 54, this 65 us: the chain of dependent FP64 instructions per
// column (about 10) bounds it now.
constexpr int CB = 64;
constexpr int CE = (CB * (CB + 1) / 2 + 255) / 256;  // elements a thread
__global__ void __launch_bounds__(256) chol_block_kernel(double* __restrict__ A, long lda, int k, int kb,
                                                        int* __restrict__ status) {
  __shared__ double col[CB], fcol[CB], rs[CB];
  __shared__ int bad;
  const int tid = threadIdx.x;
  double* D = A + (long)k * lda + k;
  const int total = kb * (kb + 1) / 2;
  double v[CE];
  int ei[CE], ej[CE];
#pragma unroll
  for (int q = 0; q < CE; ++q) {
    // e = j'(j'+1)/2 + i', 0 <= i' <= j', counted from the last row and column
    const int e = tid + 256 * q;
    int jp = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
    while (jp * (jp + 1) / 2 > e) --jp;
    while ((jp + 1) * (jp + 2) / 2 <= e) ++jp;
    ej[q] = kb - 1 - jp;
    ei[q] = kb - 1 - (e - jp * (jp + 1) / 2);
    v[q] = e < total ? D[(long)ei[q] * lda + ej[q]] : 0.0;
  }
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int c = 0; c < kb; ++c) {
    const int m = kb - c, live = m * (m + 1) / 2, next = (m - 1) * m / 2;  // e in [next, live): column c
#pragma unroll
    for (int q = 0; q < CE; ++q) {
      const int e = tid + 256 * q;
      if (e < live && e >= next) col[ei[q]] = v[q];
    }
    __syncthreads();
    if (tid < CB && tid >= c && tid < kb) {
      double d = col[c];
      const long long bits = __double_as_longlong(d);  // d > 0, by integers
      if (bits <= 0 || bits > 0x7ff0000000000000LL) {
        d = 1.0;
        if (tid == c && !bad) bad = c + 1;
      }
      if (tid == c) rs[c] = d;
      const double f = col[tid];
      // a division where the reciprocal would leave the normal range (or d is infinite)
      const int hi = __double2hiint(d);
      const bool far = hi < ((1023 - 1000) << 20) || hi >= ((1023 + 1000) << 20);
      fcol[tid] = far ? f / d : f * fast_recip(d);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < CE; ++q)
      if (tid + 256 * q < next) v[q] = fma(-col[ei[q]], fcol[ej[q]], v[q]);
    __syncthreads();
  }
  __syncthreads();
  if (tid < kb) rs[tid] = 1.0 / sqrt(rs[tid]);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < CE; ++q)
    if (tid + 256 * q < total) D[(long)ei[q] * lda + ej[q]] = v[q] * rs[ej[q]];
  if (tid == 0 && bad) atomicCAS(status, 0, k + bad);
}

// Panel below a factored diagonal block: rows r >= k + kb of A[:, k:k+kb] := row
// L11^{-T}, one warp per row: the row in registers (two columns a lane), L11's
// columns from shared memory; each step broadcasts one finished entry.
__global__ void __launch_bounds__(256) chol_panel_kernel(double* __restrict__ A, long lda, int k, int kb,
                                                        int n) {
  __shared__ double lt[CB][CB];  // lt[c][j] = L11[j][c]
  __shared__ double inv[CB];
  const double* D = A + (long)k * lda + k;
  for (int t = threadIdx.x; t < kb * CB; t += 256) {
    const int c = t / CB, j = t % CB;
    lt[c][j] = j < kb && j >= c ? D[(long)j * lda + c] : 0.0;
    if (j == 0) inv[c] = 1.0 / D[(long)c * lda + c];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long r = k + kb + (long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (r >= n) return;
  double* row = A + r * lda + k;
  double x0 = lane < kb ? row[lane] : 0.0, x1 = lane + 32 < kb ? row[lane + 32] : 0.0;
  for (int c = 0; c < kb; ++c) {
    const double b = __shfl_sync(0xffffffffu, c < 32 ? x0 : x1, c & 31) * inv[c];
    const double* l = lt[c];
    if (lane == (c & 31)) {
      if (c < 32) x0 = b; else x1 = b;
    }
    if (lane > c) x0 = fma(-b, l[lane], x0);
    if (lane + 32 > c) x1 = fma(-b, l[lane + 32], x1);
  }
  if (lane < kb) row[lane] = x0;
  if (lane + 32 < kb) row[lane + 32] = x1;
}

// A[i][j] -= sum_c P[i][c] P[j][c] for i >= j >= k + kb, P the panel A[:, k:k+kb]: 16 x 16 tiles.
__global__ void __launch_bounds__(256) chol_update_kernel(double* __restrict__ A, long lda, int k, int kb,
                                                         int n) {
  __shared__ double pi[16][CB + 1], pj[16][CB + 1];
  if (blockIdx.x > blockIdx.y) return;
  const long i0 = k + kb + (long)blockIdx.y * 16, j0 = k + kb + (long)blockIdx.x * 16;
  for (int t = threadIdx.x; t < 16 * kb; t += 256) {
    const int r = t / kb, c = t % kb;
    pi[r][c] = i0 + r < n ? A[(i0 + r) * lda + k + c] : 0.0;
    pj[r][c] = j0 + r < n ? A[(j0 + r) * lda + k + c] : 0.0;
  }
  __syncthreads();
  const int ti = threadIdx.x >> 4, tj = threadIdx.x & 15;
  double s = 0.0;
  for (int c = 0; c < kb; ++c) s = fma(pi[ti][c], pj[tj][c], s);
  const long i = i0 + ti, j = j0 + tj;
  if (i < n && j <= i) A[i * lda + j] -= s;
}

cudaError_t cholesky_step_f64(double* A, long lda, int k, int kb, int n, int* status, cudaStream_t s) {
  const int rest = n - k - kb;
  chol_block_kernel<<<1, 256, 0, s>>>(A, lda, k, kb, status);
  if (rest > 0) chol_panel_kernel<<<(unsigned)((rest + 7) / 8), 256, 0, s>>>(A, lda, k, kb, n);
  count_launch(rest > 0 ? 2 : 1);
  return cudaGetLastError();
}

// Zeroes the upper triangle.
__global__ void lower_kernel(double* A, int n) {
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < (long)n * n;
       t += (long)gridDim.x * blockDim.x)
    if (t % n > t / n) A[t] = 0.0;
}

cudaError_t cholesky_tiled_f64(double* A, int n, int* status, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(status, 0, 4, s);
  if (e != cudaSuccess) return e;
  for (int k = 0; k < n; k += CB) {
    const int kb = std::min(CB, n - k), rest = n - k - kb;
    e = cholesky_step_f64(A, n, k, kb, n, status, s);
    if (e != cudaSuccess) return e;
    if (rest <= 0) break;
    const unsigned t = (unsigned)((rest + 15) / 16);
    chol_update_kernel<<<dim3(t, t), 256, 0, s>>>(A, n, k, kb, n);
    count_launch();
  }
  lower_kernel<<<blocks_of((long)n * n), 256, 0, s>>>(A, n);
  count_launch();
  return cudaGetLastError();
}

// Cholesky in one block, for the tensor path's set-up only: its Phi' = Phi L^{-T} is
// rounded to FP16 pieces, whose last bits follow those of L and would move the K of a
// geometry by about 1e-9 (relative), so its order of operations is kept.
__global__ void cholesky_kernel(double* A, int n, int* status) {
  __shared__ int fail;
  if (threadIdx.x == 0) fail = 0;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (threadIdx.x == 0) {
      const double d = A[(long)k * n + k];
      if (!(d > 0.0)) fail = k + 1;
      else A[(long)k * n + k] = sqrt(d);
    }
    __syncthreads();
    if (fail) break;
    const double piv = A[(long)k * n + k];
    for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) A[(long)i * n + k] /= piv;
    __syncthreads();
    const long rem = n - k - 1;
    for (long t = threadIdx.x; t < rem * rem; t += blockDim.x) {
      const int i = k + 1 + (int)(t / rem), j = k + 1 + (int)(t % rem);
      if (j <= i) A[(long)i * n + j] -= A[(long)i * n + k] * A[(long)j * n + k];
    }
    __syncthreads();
  }
  if (!fail)
    for (long t = threadIdx.x; t < (long)n * n; t += blockDim.x) {
      const int i = (int)(t / n), j = (int)(t % n);
      if (j > i) A[t] = 0.0;
    }
  if (threadIdx.x == 0) *status = fail;
}

cudaError_t cholesky_f64(double* A, int n, int* status, cudaStream_t s) {
  cholesky_kernel<<<1, 1024, 0, s>>>(A, n, status);
  count_launch();
  return cudaGetLastError();
}

__global__ void trsm_kernel(const double* __restrict__ L, int n, const double* __restrict__ B,
                            int rows, double* __restrict__ X) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x) {
    const double* b = B + (long)r * n;
    double* x = X + (long)r * n;
    for (int k = 0; k < n; ++k) {
      double acc = b[k];
      for (int j = 0; j < k; ++j) acc -= L[(long)k * n + j] * x[j];
      x[k] = acc / L[(long)k * n + k];
    }
  }
}

// X L^T = B, one warp per row for n <= 32 Q: the row in registers (Q columns a
// lane); step c broadcasts x[c] = b[c] / L[c][c] and subtracts its multiple of column c of
// L (lanes along the column: LT is L transposed, with the reciprocals of its diagonal: a
// division a step would be most of the FP64 work) from the entries that follow.
template <int Q>
__global__ void __launch_bounds__(64) trsm_warp_kernel(const double* __restrict__ LT, int n,
                                                       const double* __restrict__ B, int rows,
                                                       double* __restrict__ X) {
  const int lane = threadIdx.x & 31;
  const long r = (long)blockIdx.x * 2 + (threadIdx.x >> 5);
  if (r >= rows) return;
  double x[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) x[q] = 32 * q + lane < n ? B[r * n + 32 * q + lane] : 0.0;
#pragma unroll
  for (int p = 0; p < Q; ++p) {
    const int c1 = min(32, n - 32 * p);
#pragma unroll 4
    for (int c = 0; c < c1; ++c) {
      const double* l = LT + (long)(32 * p + c) * n + lane;
      double f[Q];
#pragma unroll
      for (int q = p; q < Q; ++q) f[q] = 32 * q + lane < n ? __ldg(l + 32 * q) : 0.0;
      const double b = __shfl_sync(0xffffffffu, x[p], c) * __shfl_sync(0xffffffffu, f[p], c);
      // row 32 p + c of LT is zero before its diagonal
      x[p] = lane == c ? b : lane > c ? fma(-b, f[p], x[p]) : x[p];
#pragma unroll
      for (int q = p + 1; q < Q; ++q) x[q] = fma(-b, f[q], x[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (32 * q + lane < n) X[r * n + 32 * q + lane] = x[q];
}

// T = A^T with the reciprocals of the diagonal.
__global__ void transpose_recip_kernel(const double* __restrict__ A, int n, double* __restrict__ T) {
  __shared__ double tile[32][33];
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += 8)
    if (r0 + i < n && c0 + (int)threadIdx.x < n) tile[i][threadIdx.x] = A[(long)(r0 + i) * n + c0 + threadIdx.x];
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8)
    if (c0 + i < n && r0 + (int)threadIdx.x < n) {
      double v = tile[threadIdx.x][i];
      if (c0 + i == r0 + (int)threadIdx.x) v = 1.0 / v;
      T[(long)(c0 + i) * n + r0 + threadIdx.x] = v;
    }
}

cudaError_t trsm_right_lt_f64(const double* L, int n, const double* B, int rows, double* X,
                              cudaStream_t s, double* LT) {
  if (!LT || n > 512) {
    trsm_kernel<<<(rows + 127) / 128, 128, 0, s>>>(L, n, B, rows, X);
    count_launch();
    return cudaGetLastError();
  }
  const unsigned t = (unsigned)((n + 31) / 32);
  transpose_recip_kernel<<<dim3(t, t), dim3(32, 8), 0, s>>>(L, n, LT);
  const unsigned blocks = (unsigned)((rows + 1) / 2);
  if (n <= 64) trsm_warp_kernel<2><<<blocks, 64, 0, s>>>(LT, n, B, rows, X);
  else if (n <= 128) trsm_warp_kernel<4><<<blocks, 64, 0, s>>>(LT, n, B, rows, X);
  else if (n <= 256) trsm_warp_kernel<8><<<blocks, 64, 0, s>>>(LT, n, B, rows, X);
  else trsm_warp_kernel<16><<<blocks, 64, 0, s>>>(LT, n, B, rows, X);
  count_launch(2);
  return cudaGetLastError();
}

// Cyclic Jacobi: rotations (p, q) in row order; each rotation updates the
// two columns, then the two rows of A and the two columns of U in parallel.
__global__ void jacobi_kernel(double* A, double* U, int n, int max_sweeps, int* sweeps) {
  __shared__ double cs[2];
  __shared__ double off_sh[1024];
  __shared__ int done;
  for (long t = threadIdx.x; t < (long)n * n; t += blockDim.x)
    U[t] = (t / n == t % n) ? 1.0 : 0.0;
  if (threadIdx.x == 0) done = 0;
  __syncthreads();
  int sw = 0;
  for (; sw < max_sweeps; ++sw) {
    double off = 0.0, tot = 0.0;
    for (long t = threadIdx.x; t < (long)n * n; t += blockDim.x) {
      const double v = A[t] * A[t];
      tot += v;
      if (t / n != t % n) off += v;
    }
    off_sh[threadIdx.x] = off;
    __syncthreads();
    if (threadIdx.x == 0) {
      double o = 0.0;
      for (int i = 0; i < (int)blockDim.x; ++i) o += off_sh[i];
      off_sh[0] = o;
    }
    __syncthreads();
    const double offn = off_sh[0];
    __syncthreads();
    off_sh[threadIdx.x] = tot;
    __syncthreads();
    if (threadIdx.x == 0) {
      double o = 0.0;
      for (int i = 0; i < (int)blockDim.x; ++i) o += off_sh[i];
      done = (offn <= 1e-30 * o) ? 1 : 0;
    }
    __syncthreads();
    if (done) break;
    for (int p = 0; p < n - 1; ++p)
      for (int q = p + 1; q < n; ++q) {
        if (threadIdx.x == 0) {
          const double apq = A[(long)p * n + q];
          double c = 1.0, s = 0.0;
          if (fabs(apq) > 1e-300) {
            const double theta = (A[(long)q * n + q] - A[(long)p * n + p]) / (2.0 * apq);
            const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
            c = 1.0 / sqrt(t * t + 1.0);
            s = t * c;
          }
          cs[0] = c;
          cs[1] = s;
        }
        __syncthreads();
        const double c = cs[0], s = cs[1];
        if (s != 0.0) {
          for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const double akp = A[(long)k * n + p], akq = A[(long)k * n + q];
            A[(long)k * n + p] = c * akp - s * akq;
            A[(long)k * n + q] = s * akp + c * akq;
            const double ukp = U[(long)k * n + p], ukq = U[(long)k * n + q];
            U[(long)k * n + p] = c * ukp - s * ukq;
            U[(long)k * n + q] = s * ukp + c * ukq;
          }
          __syncthreads();
          for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const double apk = A[(long)p * n + k], aqk = A[(long)q * n + k];
            A[(long)p * n + k] = c * apk - s * aqk;
            A[(long)q * n + k] = s * apk + c * aqk;
          }
          __syncthreads();
          if (threadIdx.x == 0) {
            A[(long)p * n + q] = 0.0;
            A[(long)q * n + p] = 0.0;
          }
        }
        __syncthreads();
      }
  }
  if (threadIdx.x == 0) *sweeps = sw;
}

cudaError_t jacobi_eig_f64(double* A, double* U, int n, int max_sweeps, int* sweeps,
                           cudaStream_t s) {
  jacobi_kernel<<<1, 256, 0, s>>>(A, U, n, max_sweeps, sweeps);
  count_launch();
  return cudaGetLastError();
}

__global__ void scale_eigcols_kernel(const double* __restrict__ A, int n,
                                     const double* __restrict__ B, int rows, double cut,
                                     double* __restrict__ X, double* __restrict__ sign) {
  __shared__ double lmax;
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int k = 0; k < n; ++k) m = fmax(m, fabs(A[(long)k * n + k]));
    lmax = m;
  }
  __syncthreads();
  const double thr = cut * lmax;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < (long)rows * n;
       t += (long)gridDim.x * blockDim.x) {
    const int k = (int)(t % n);
    const double lam = A[(long)k * n + k];
    X[t] = fabs(lam) > thr ? B[t] / sqrt(fabs(lam)) : 0.0;
  }
  if (blockIdx.x == 0)
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const double lam = A[(long)k * n + k];
      sign[k] = fabs(lam) > thr ? (lam > 0 ? 1.0 : -1.0) : 0.0;
    }
}

cudaError_t scale_eigcols_f64(const double* Adiag_src, int n, const double* B, int rows, double cut,
                              double* X, double* sign, cudaStream_t s) {
  scale_eigcols_kernel<<<64, 256, 0, s>>>(Adiag_src, n, B, rows, cut, X, sign);
  count_launch();
  return cudaGetLastError();
}

}  // namespace xk
