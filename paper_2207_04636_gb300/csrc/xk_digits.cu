// FP64 products on the tensor cores by splitting both operands into exact
// 8-bit digits (the scheme of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms
// 59 (2012), and its tensor-core form by Ootomo, Ozaki and Yokota, IJHPCA 38
// (2024)).
//
// Every operand row (the K direction) has a power-of-two scale 2^e > max|row|;
// an element becomes the integer X = round(x 2^(55 - e)), |X| < 127 2^48, and
// X = sum_i d_i 2^(8 (6 - i)) with seven signed digits |d_i| <= 128, exact in
// FP16; Y, the operand with fewer rows, has an eighth, to 2^(e - 63).  A product of two digits
// is an integer <= 2^14, and tcgen05.mma adds such integers exactly in its FP32 accumulator
// while the sum stays below 2^24.  The products d_i d'_j of one weight l = i + j share an
// accumulator; levels 0 to 7 are formed (35 of the 56 products), every 256 terms they are
// drained into an integer accumulator of 64 + 20 bits, whose last bit weighs 2^-58 of the
// largest product.  Levels 0 to 3 never exceed 2^24 in 256 terms and are exact.  Levels 4 to 7
// have 5 to 8 pairs and can pass it, where an addition may lose a unit: at most some 20 units
// of level 4, 2^-50 of 256 largest products, and that only when all digits are near their limit
// with one sign in every pair (256 FMAs of such terms are allowed 2^-46).  The result is
// rounded to FP64 once, so its error is in practice that of the 55-bit
// operands and the dropped levels: 5e-17 to 3e-16 of the 2-norm on the
// products of a build, where a chain of FP64 FMAs leaves 1.4e-16 to 9e-15.  The 55 bits
// count from the largest element of the row, so the callers see to it that the two operands
// are not graded in opposite directions along K (units of powers of two: xk_api.cu).
//
// What Y loses it loses alike for all rows of X, hence its eighth digit: C rounded to 55 bits
// moved Psi = Phi C by one smooth function per orbital, which sums over the grid do not average
// out as they do the roundings of Phi's rows, or those of FMAs.  J's error on three cells of 8
// centres (coefficients up to 570, against extended precision): 2.2e-14 to 3.5e-14 with seven
// digits, 5.9e-15 to 1.6e-14 with eight; 2.9e-15 to 5.7e-15 with FMAs.  It costs 0.9 % of an
// FP64 build.  Rounding ties by turns (low_offsets) makes it 1.6e-15 to 3.4e-15.
//
// What bounds it: a 128 x 64 tile takes 35 digit products per K = 16 step, 1120
// clocks of the tensor cores.  One instruction forms up to four of them: the digits of Y
// lie one after another in shared memory and the levels in TMEM, so N = 256 rows of
// Y's digits j .. j + 3 against one digit of X give levels i + j .. i + j + 3, and the
// operands are read 114 KB at a time instead of 210 (890 clocks instead of 1640).  Beside
// them run the workers: about 13 integer operations an element (64 a clock and SM),
// their loads, and the drains.  Measured with parts left out (1053 x 1053 x 91125,
// 6.6 ms): matrix instructions and drains 4.5, workers alone 5.4, workers without loads
// 4.2 ms; refilling a register pair as soon as its digits are formed, to have loads in
// flight longer, made it 7.0.
// FP64 FMAs on the CUDA cores run at 2 a clock and SM.  Measured on random operands
// (GB300, us, with seven digits of Y; FP64 FMA kernel before): 1755 x 54 x 91125: 814
// (14500), 54 x 91125 x 1755: 821 (17500), 1755 x 91125 x 54 (taking and storing the results
// bounds it): 1270 (17700), 351 x 351 x 91125: 816 (26600), 1053 x 1053 x 91125: 6630.  A 27-centre
// FP64 build went from 64.7 to 3.69 ms, its Coulomb matrix from 30.6 to 1.14 ms.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "tc_common.cuh"
#include "xk_internal.h"

namespace xk {

namespace {

using namespace tc;

constexpr int kDig = 7;             // digits of X
constexpr int kDigY = 8;            // digits of Y
constexpr int kLev = 8;             // accumulator levels (i + j)
constexpr int DK = 32;              // K per block: 64-byte rows, 64-byte swizzle
constexpr int DX = 128, DY = 64;    // tile: X rows (MMA M) by Y rows (MMA N)
constexpr int DX_PLANE = DX * DK * 2, DY_PLANE = DY * DK * 2;
constexpr int D_STAGE = kDig * DX_PLANE + kDigY * DY_PLANE;  // 88 KB
constexpr int D_STAGES = 2;
constexpr int D_SMEM = D_STAGES * D_STAGE + 1024;
constexpr int D_GROUP = 256 / DK;   // K blocks between drains
// 16 worker warps turn operands into digits and take accumulators out; one
// more issues the MMAs.  It sits in a warpgroup of its own whose registers go
// to the workers (setmaxnreg: 640 threads launch with 96; 512 x 112 + 128 x 32 =
// 640 x 96).
constexpr int D_WORK = 16;
constexpr int D_THREADS = 32 * (D_WORK + 4);

// Tiles of a symmetric product that reach y <= x: 2 (i + 1) of X tile i, the last
// X tile's all.
int sym_tiles(int tiles_x, int tiles_y) { return (tiles_x - 1) * tiles_x + tiles_y; }

// One operand: element (row, k) at p[row ld + k] (kc) or p[k ld + row].
struct DOperand {
  const double* p;
  long ld;
  int rows;
  int kc;
  const int* scale;  // per row: high word of max |row|
};

struct DArgs {
  DOperand x, y;
  int K, kchunk, ksplit;
  int tiles_x, tiles_y;
  int tiles;         // of one K split: tiles_x * tiles_y, or those that reach y <= x (sym)
  int sym;
  int swapped;       // X rows are the columns of C (else its rows)
  int M, N;          // C is M x N
  double* C; long ldc;
  double alpha, beta;
  int careful;        // added to C, or in place
  int scaled, added;  // alpha != 1, beta != 0 (an FP64 comparison per result would cost more)
  const double* H; long ldh;
  int *xmax, *ymax;  // digit_maxima: largest |C| per X and Y row (nullable)
  double* work;      // ksplit > 1: partial sums [ksplit][M][N]
  int nbatch; long cskip;  // swapped only: batches of C's columns (DGemm)
  int* flag;         // set to 1 when a row cannot be split (row_unfit), to 2 when a bounded
                     // wait gave up: the product is then left to the FP64 FMAs
  int* status;       // nullable: gets a code when a wait gave up, for the call to report
  long long wait;    // limit of the pipeline waits when shortened (kShort)
};

// Scale exponent e of a row from the high word of its largest |x|:
// |x| 2^-e <= 1 - 2^-7.  A row of zeros gets 0.
__device__ __forceinline__ int row_exp(int hi) { return hi ? ((hi + (1 << 14)) >> 20) - 1022 : 0; }

__device__ __forceinline__ uint32_t row_e21(int hi) {
  return ((uint32_t)(row_exp(hi) + 1022) << 21) | 0x1fffffu;
}

// Rows whose largest |x| is infinite, NaN or below 2^-900 (where an element's
// subnormals would count) are not split.
__device__ __forceinline__ bool row_unfit(int hi) {
  return hi >= 0x7ff00000 || (hi > 0 && hi < ((1023 - 900) << 20));
}

// The eight digits of |x| on the grid 2^(e - 63), each plus 128 (most significant digit in
// byte 7; the upper seven are |x| rounded to the grid 2^(e - 55)).  e21 = (e + 1022) 2^21 +
// 2^21 - 1.  Integer operations run at 64 a clock and SM here, so they are what the split
// costs: |x| = m 2^(ex - 1085) with m of 63 bits (a subnormal x, taken for a normal one, is
// below the grid) is shifted by t = e + 1022 - ex >= 0 to the finer grid, t being what is left
// of e21 - 2 high word (one multiply-add, on the other pipe; the doubling drops the sign)
// above its mantissa bits; one sum then adds the offsets 128 2^(8 i) of the digits, the
// lowest being half a step of the coarser grid (low: 0x80808080, or less one, which
// rounds ties to seven digits down).
__device__ __forceinline__ uint2 digits_of(double x, uint32_t e21, uint32_t low) {
  const uint32_t xh = __double2hiint(x), xl = __double2loint(x);
  const uint32_t t = (e21 - 2u * xh) >> 21;
  const uint32_t mh = (xh & 0xfffffu) | 0x100000u;
  const unsigned long long m =
      ((unsigned long long)__funnelshift_l(xl, mh, 10) << 32) | (xl << 10);
  unsigned long long y;
  asm("shr.u64 %0, %1, %2;" : "=l"(y) : "l"(m), "r"(t));  // t > 63 gives 0
  y += 0x8080808000000000ull + low;
  return make_uint2((uint32_t)y, (uint32_t)(y >> 32));
}

// FP16 pairs (digit of x, digit of y), most significant first: byte + 1024 = 0x64xx,
// less 1024 + 128, times the element's sign (+-1 from the high words' sign bits).
template <int D>
__device__ __forceinline__ void digit_pairs(double x, double y, uint32_t e21, uint32_t low, uint32_t (&o)[D]) {
  const uint2 a = digits_of(x, e21, low), b = digits_of(y, e21, low);
  const uint32_t c = 0x64646464u;
  const uint32_t w0 = __byte_perm(a.y, b.y, 0x7632), w1 = __byte_perm(a.y, b.y, 0x5410),
                 w2 = __byte_perm(a.x, b.x, 0x7632), w3 = __byte_perm(a.x, b.x, 0x5410);
  o[0] = __byte_perm(w0, c, 0x4341); o[1] = __byte_perm(w0, c, 0x4240);
  o[2] = __byte_perm(w1, c, 0x4341); o[3] = __byte_perm(w1, c, 0x4240);
  o[4] = __byte_perm(w2, c, 0x4341); o[5] = __byte_perm(w2, c, 0x4240);
  o[6] = __byte_perm(w3, c, 0x4341);
  if constexpr (D == 8) o[7] = __byte_perm(w3, c, 0x4240);
  const uint32_t sg =
      (__byte_perm(__double2hiint(x), __double2hiint(y), 0x7632) & 0x80008000u) | 0x3c003c00u;
  const __half2 s = *reinterpret_cast<const __half2*>(&sg);
  const __half2 off = __hmul2(s, __half2half2(__ushort_as_half(0xe480)));  // -1152
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const __half2 r = __hfma2(*reinterpret_cast<__half2*>(&o[i]), s, off);
    o[i] = *reinterpret_cast<const uint32_t*>(&r);
  }
}

// A block of one operand passes through the registers of the 512 workers, n
// elements each, n = 8 (X, 128 rows) or 4 (Y, 64 rows).  Position 2 j of the
// block's K order holds term j and position 2 j + 1 term j + 16, in both operands:
//  * K contiguous in memory: lane l holds the pairs k = l % 16, + 16 of the rows
//    n w + l / 16 + 2 i of warp w, so that a load reads whole 128-byte pieces of two rows
//    (on any alignment) and a store writes whole 128-byte lines (one 4-byte digit
//    pair per lane);
//  * rows contiguous: a thread holds n successive positions of one row (lanes along
//    the rows) and stores 2 n bytes of each digit.
// Rows past the operand's last are read as that one (nothing of them is stored).
template <int n, bool KC>
__device__ __forceinline__ void load_block(const DOperand& o, int row0, long k0, long kend, int tid,
                                           double (&v)[n]) {
  constexpr int R = 16 * n;  // rows of the block
  const bool whole = k0 + DK <= kend;
  if constexpr (KC) {
    const int r = row0 + (tid >> 5) * n + ((tid >> 4) & 1);
    const long k = k0 + (tid & 15);
    const double* p = o.p + k;
    if (whole) {
#pragma unroll
      for (int i = 0; i < n / 2; ++i) {
        const double* q = p + (long)min(r + 2 * i, o.rows - 1) * o.ld;
        v[2 * i] = __ldg(q);
        v[2 * i + 1] = __ldg(q + 16);
      }
    } else {
#pragma unroll
      for (int i = 0; i < n / 2; ++i) {
        const double* q = p + (long)min(r + 2 * i, o.rows - 1) * o.ld;
        v[2 * i] = k < kend ? __ldg(q) : 0.0;
        v[2 * i + 1] = k + 16 < kend ? __ldg(q + 16) : 0.0;
      }
    }
  } else {
    const long k = k0 + n / 2 * (tid / R);
    const double* p = o.p + k * o.ld + min(row0 + tid % R, o.rows - 1);
    const long half = 16 * o.ld;
    if (whole) {
#pragma unroll
      for (int i = 0; i < n / 2; ++i, p += o.ld) {
        v[2 * i] = __ldg(p);
        v[2 * i + 1] = __ldg(p + half);
      }
    } else {
#pragma unroll
      for (int i = 0; i < n / 2; ++i, p += o.ld) {
        v[2 * i] = k + i < kend ? __ldg(p) : 0.0;
        v[2 * i + 1] = k + i + 16 < kend ? __ldg(p + half) : 0.0;
      }
    }
  }
}

// Row of the block whose exponent lane l of warp w looks up for its warp.
template <int n, bool KC>
__device__ __forceinline__ int block_row(int w, int l) {
  return KC ? w * n + l % n : (32 * w + l) % (16 * n);
}

// Ties of X's rounding to seven digits go up and down by turns along rows and K.  They are
// frequent (an element between 1/16 and 1/8 of 2^e has one bit below the grid), and
// rounded up all, they added 2^-61 of the largest to every element of one sign (Coulomb
// matrix of 8 centres: a third to four fifths of its error).
__device__ __forceinline__ uint32_t low_offsets(int odd) { return 0x80808080u - (odd & 1); }

// Digits of the block into the stage; ex: e21 (digits_of) of the rows block_row(w, 0..31).
template <int n, bool KC>
__device__ __forceinline__ void store_block(uint8_t* st, const uint32_t* ex, int tid, const double (&v)[n]) {
  constexpr int R = 16 * n, PLANE = R * DK * 2, D = n == 8 ? kDig : kDigY;
  if constexpr (KC) {
    // rows r0 + 2 i: the swizzle's chunk is that of r0 with bit 1 of r, i.e. bit 0 of i, flipped
    const int r0 = (tid >> 5) * n + ((tid >> 4) & 1), l = tid & 15;
    const uint32_t low = low_offsets(D == kDig ? (tid >> 4) ^ tid : 0);
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const int r = r0 + 2 * i;
      const uint32_t e = ex[((tid >> 4) & 1) + 2 * i];
      uint32_t o[D];
      digit_pairs(v[2 * i], v[2 * i + 1], e, low, o);
      uint32_t* d = reinterpret_cast<uint32_t*>(st + r * 64 + (((l >> 2) ^ ((r >> 1) & 3)) << 4) + (l & 3) * 4);
#pragma unroll
      for (int q = 0; q < D; ++q) d[q * (PLANE / 4)] = o[q];
    }
  } else {
    const int r = tid % R, q = tid / R;  // q: which n of the 32 k
    const uint32_t e = ex[tid & 31];
    uint32_t o[n / 2][D];
#pragma unroll
    for (int i = 0; i < n / 2; ++i)
      digit_pairs(v[2 * i], v[2 * i + 1], e, low_offsets(D == kDig ? tid ^ i : 0), o[i]);
    const int byte = q * n * 2;  // within the row's 64 bytes
    uint8_t* d = st + r * 64 + (((byte >> 4) ^ ((r >> 1) & 3)) << 4) + (byte & 15);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      if constexpr (n == 8)
        *reinterpret_cast<uint4*>(d + b * PLANE) = make_uint4(o[0][b], o[1][b], o[2][b], o[3][b]);
      else
        *reinterpret_cast<uint2*>(d + b * PLANE) = make_uint2(o[0][b], o[1][b]);
    }
  }
}

// (hi + lo 2^-20) 2^E rounded to FP64, 0 <= lo < 2^20: the 96-bit number
// hi : lo is normalised and rounded in 32-bit words (an FP64 operation costs 64
// times an integer one here).
__device__ __forceinline__ double pack_f64(long long hi, uint32_t lo, int E) {
  uint32_t w0 = lo << 12, w1 = (uint32_t)hi, w2 = (uint32_t)((unsigned long long)hi >> 32);
  const uint32_t sign = w2 & 0x80000000u;
  if (sign) {
    w0 = 0u - w0;
    const unsigned long long m = ~(unsigned long long)hi + (w0 == 0);
    w1 = (uint32_t)m;
    w2 = (uint32_t)(m >> 32);
  }
  int ex = 1023 + 63 + E;  // biased exponent when the top bit of w2 is set
  if (w2 == 0) {
    w2 = w1; w1 = w0; w0 = 0; ex -= 32;
    if (w2 == 0) { w2 = w1; w1 = 0; ex -= 32; }
    if (w2 == 0) return 0.0;
  }
  const int z = __clz(w2);
  ex -= z;
  const uint32_t h = __funnelshift_l(w1, w2, z), l = __funnelshift_l(w0, w1, z);
  // 53 bits: h[31:0] l[31:11], rounded by bit 10; the leading one adds to the exponent
  const unsigned long long m =
      (((unsigned long long)(h >> 11) << 32) | __funnelshift_r(l, h, 11)) + ((l >> 10) & 1);
  if ((uint32_t)(ex - 1) < 2045u)
    return __longlong_as_double(
        (long long)(m + ((unsigned long long)(sign | ((uint32_t)(ex - 1) << 20)) << 32)));
  const double d = (double)m;
  return scalbn(sign ? -d : d, ex - 1075);
}

// The block after the one being loaded, into L2: one 128-byte line per thread
// (256 lines of X, 128 of Y; lines that straddle are left to the loads).
template <bool XK, bool YK>
__device__ __forceinline__ void prefetch_block(const DArgs& g, long x0, long y0, long k0, long kend, int tid) {
  const bool isx = tid < 256;
  const DOperand& o = isx ? g.x : g.y;
  const int i = isx ? tid : tid - 256;
  if (i >= 256 - (isx ? 0 : 128)) return;
  const bool kc = isx ? XK : YK;
  // K contiguous: two lines a row; rows contiguous: 8 (X) or 4 (Y) lines a k
  const long r = (isx ? x0 : y0) + (kc ? i >> 1 : (i & (isx ? 7 : 3)) * 16);
  const long k = k0 + (kc ? (i & 1) * 16 : i >> (isx ? 3 : 2));
  if (r >= o.rows || k >= kend) return;
  asm volatile("prefetch.global.L2 [%0];" ::"l"(o.p + (kc ? r * o.ld + k : k * o.ld + r)));
}

template <bool XK, bool YK, bool kShort>
__global__ void __launch_bounds__(D_THREADS, 1) digit_gemm_kernel(const __grid_constant__ DArgs g) {
  extern __shared__ uint8_t d_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(d_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full[D_STAGES], empty[D_STAGES], set_ready, free_lo, free_hi, drain;
  __shared__ uint32_t tslot;
  __shared__ volatile int abort_flag;
  __shared__ int skip;
  // exponents of the rows a warp turns into digits (X, then Y), of two tiles
  __shared__ uint32_t exps[D_WORK][2][64];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform: the register split needs it
  // A product that is added to C, or overwrites an operand, must not be left out half-way:
  // every CTA looks at every row first.  Any other is formed again as a whole when a
  // tile meets such a row.
  if (tid == 0) skip = 0;
  __syncthreads();
  if (g.careful) {
    bool bad = false;
    for (int i = tid; i < g.x.rows; i += D_THREADS) bad |= row_unfit(__ldg(g.x.scale + i));
    for (int i = tid; i < g.y.rows; i += D_THREADS) bad |= row_unfit(__ldg(g.y.scale + i));
    if (bad) skip = 1;
  }
  __syncthreads();
  if (skip) {
    if (tid == 0) *g.flag = 1;
    return;
  }
  if (tid == 0) {
    for (int s = 0; s < D_STAGES; ++s) {
      mbar_init(&full[s], D_WORK);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&set_ready, 1);
    mbar_init(&free_lo, D_WORK);
    mbar_init(&free_hi, D_WORK);
    mbar_init(&drain, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == D_WORK) {
    tmem_alloc(&tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = tslot;
  const int ntiles = g.tiles * g.ksplit;
  auto wait = [&](uint64_t* bar, uint32_t parity) __attribute__((always_inline)) {
    if constexpr (!kShort) return mbar_wait_warp(bar, parity);
    // (inline: a call would take more registers than the workers have)
    __syncwarp();
    const long long t0 = clock64();
    bool ok;
    while (!(ok = mbar_test(bar, parity)) && clock64() - t0 <= g.wait) {}
    return __all_sync(0xffffffffu, ok) != 0;
  };
  auto gave_up = [&](int code) __attribute__((always_inline)) {
    if (lane == 0) {
      atomicExch(g.flag, 2);
      if (g.status) atomicExch(g.status, code);
      abort_flag = 1;
    }
    __syncwarp();
  };
  // tile t: X tile fastest, then Y tile, then the K split (symmetric: Y fastest)
  auto place = [&](int t, int& xt, int& yt, int& z) __attribute__((always_inline)) {
    z = t / g.tiles;
    const int r = t - z * g.tiles;
    if (g.sym) {
      xt = min((int)((sqrtf(4.0f * r + 1.0f) - 1.0f) * 0.5f), g.tiles_x - 1);
      while (xt > 0 && xt * (xt + 1) > r) --xt;
      while (xt < g.tiles_x - 1 && (xt + 1) * (xt + 2) <= r) ++xt;
      yt = r - xt * (xt + 1);
    } else {
      xt = r % g.tiles_x;
      yt = r / g.tiles_x;
    }
  };
  auto kblocks = [&](int z) {
    const long k0 = (long)z * g.kchunk, k1 = min((long)g.K, k0 + g.kchunk);
    return (int)((k1 - k0 + DK - 1) / DK);
  };

  if (warp >= D_WORK) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp == D_WORK) {
      // per block 35 products of two K = 16 steps, the low levels first: their
      // accumulators are taken out first
      const uint64_t d0 = sdesc_sw64(smem_u32(sm), 16, 512);
      int it = 0, G = 0;
      bool good = true;
      auto fail = [&]() {
        gave_up(51);
        good = false;
      };
      for (int t = blockIdx.x; good && t < ntiles; t += gridDim.x) {
        const int nkb = kblocks(t / g.tiles);
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          if (__shfl_sync(0xffffffffu, (int)abort_flag, 0)) { good = false; break; }
          const int s = it % D_STAGES;
          const bool first = (kb % D_GROUP) == 0;
          const bool last = (kb % D_GROUP) == D_GROUP - 1 || kb == nkb - 1;
          if (!wait(&full[s], (it / D_STAGES) & 1)) { fail(); break; }
          if (first && G >= 1 && !wait(&free_lo, (G - 1) & 1)) { fail(); break; }
          tc_fence_after();
          const uint64_t dx = d0 + (uint64_t)((s * D_STAGE) >> 4);
          const uint64_t dy = dx + (uint64_t)((kDig * DX_PLANE) >> 4);
          // digit i of X by digits j0 .. j0 + c - 1 of Y, whose planes follow one another, gives
          // levels i + j0 onward, whose columns do
          auto run = [&](int i, int j0, int c, bool acc) __attribute__((always_inline)) {
            mma_ss_run2(tbase + 64 * (i + j0), dx + (uint64_t)((i * DX_PLANE) >> 4),
                        dy + (uint64_t)((j0 * DY_PLANE) >> 4), 2, 2,
                        idesc_f16(128, DY * c, false, false, false), acc ? 1u : 0u);
          };
          // levels 4 to 7; digit 1 reaches all four
          run(1, 3, 4, !first);
          run(0, 4, 4, true);
          run(2, 2, 4, true);
          run(3, 1, 4, true);
          run(4, 0, 4, true);
          run(5, 0, 3, true);
          run(6, 0, 2, true);
          if (first && G >= 1) {
            if (!wait(&free_hi, (G - 1) & 1)) { fail(); break; }
            tc_fence_after();
          }
          // levels 0 to 3
          run(0, 0, 4, !first);
          run(1, 0, 3, true);
          run(2, 0, 2, true);
          run(3, 0, 1, true);
          if (elect_one()) {
            mma_commit(&empty[s]);
            if (last) mma_commit(&set_ready);
          }
          __syncwarp();
          if (last) ++G;
        }
      }
      if (elect_one()) mma_commit(&drain);
      __syncwarp();
      mbar_wait_warp(&drain, 0);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    // workers
    const int quad = warp & 3, cg = warp >> 2;  // accumulator rows and columns of this warp
    const uint32_t tacc = tbase + (static_cast<uint32_t>(quad * 32) << 16) + 16 * cg;
    bool ok = true;
    auto lost = [&]() __attribute__((always_inline)) {
      gave_up(52);
      ok = false;
    };
    long long hi[16];  // levels 0-3, in units of level 3
    uint32_t lo[16];   // levels 4-7: 20 bits below level 3
    int G = 0;  // groups taken
    // the K block being fetched: tile ft, block fkb
    int ft = blockIdx.x, fkb = 0, fn = 0, fz = 0;
    int fx0 = 0, fy0 = 0;
    int fpar = 1;  // which half of exps the tile being fetched uses
    // A tile of as many blocks as there are stages finds block kb in stage kb; when
    // this CTA's tile before it had the same Y rows, their digits are there already (the
    // products of 33 to 64 terms, a third of their conversions: 1755 x 91125 x 54 1440 ->
    // 1270 us)
    bool fkeep = false, vkeep = false;  // tile being fetched; block in vx, vy
    auto open_tile = [&]() __attribute__((always_inline)) {
      if (ft >= ntiles) { fn = 0; return; }
      int xt, yt;
      place(ft, xt, yt, fz);
      const int pn = fn, py = fy0;
      fx0 = xt * DX;
      fy0 = yt * DY;
      fn = kblocks(fz);
      fkeep = g.ksplit == 1 && fn == D_STAGES && pn == fn && py == fy0;
      fpar ^= 1;
      const long rx = fx0 + block_row<8, XK>(warp, lane), ry = fy0 + block_row<4, YK>(warp, lane);
      const int hx = __ldg(g.x.scale + min(rx, g.x.rows - 1l)), hy = __ldg(g.y.scale + min(ry, g.y.rows - 1l));
      if (row_unfit(hx) || row_unfit(hy)) *g.flag = 1;
      // with one block a tile this half held the exponents of the block stored just now:
      // every lane has read its own
      __syncwarp();
      exps[warp][fpar][lane] = row_e21(hx);
      exps[warp][fpar][32 + lane] = row_e21(hy);
      __syncwarp();
    };
    double vx[8], vy[4];
    auto fetch = [&]() __attribute__((always_inline)) {
      const long k0 = (long)fz * g.kchunk + (long)fkb * DK;
      const long kend = min((long)g.K, (long)(fz + 1) * g.kchunk);
      load_block<8, XK>(g.x, fx0, k0, kend, tid, vx);
      vkeep = fkeep;
      if (!fkeep) load_block<4, YK>(g.y, fy0, k0, kend, tid, vy);
      prefetch_block<XK, YK>(g, fx0, fy0, k0 + DK, kend, tid);
      if (++fkb == fn) { fkb = 0; ft += gridDim.x; open_tile(); }
    };
    // adds a finished group of accumulators to hi, lo (zeroed at a tile's first
    // group); levels 5 to 7 are added up in FP32 first: up to 2^28.6 units of lo, so half an
    // ulp is 2^4 of them, 2^-62 of the group's 256 largest products, and the rounding to an
    // integer half a unit more
    auto take_group = [&](bool fresh) __attribute__((always_inline)) {
      if (!wait(&set_ready, G & 1)) { lost(); return; }
      tc_fence_after();
      auto level = [](uint32_t a) { return __float2int_rn(__uint_as_float(a)); };
      auto mad = [](int a, int b, long long c) {  // one instruction, off the busy pipe
        long long r;
        asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
        return r;
      };
#pragma unroll
      for (int c = 0; c < 16; c += 8) {
        uint32_t a[8], b[8], d[8];
        tmem_ld8(tacc + 64 * 5 + c, a);
        tmem_ld8(tacc + 64 * 6 + c, b);
        tmem_ld8(tacc + 64 * 7 + c, d);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float f = fmaf(__uint_as_float(d[j]), 0x1p-12f, __uint_as_float(b[j]) * 0x1p-4f);
          a[j] = (uint32_t)__float2int_rn(fmaf(__uint_as_float(a[j]), 0x1p4f, f));
        }
        tmem_ld8(tacc + 64 * 4 + c, b);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          // (int)a < 2^29
          const long long t = mad(level(b[j]), 1 << 12, (int)a[j] + (fresh ? 0 : (int)lo[c + j]));
          lo[c + j] = (uint32_t)t & 0xfffffu;
          hi[c + j] = (fresh ? 0 : hi[c + j]) + (t >> 20);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&free_lo);
#pragma unroll
      for (int c = 0; c < 16; c += 8) {
        uint32_t a[8], b[8];
        tmem_ld8(tacc + c, a);
        tmem_ld8(tacc + 64 + c, b);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) hi[c + j] = mad(level(b[j]), 1 << 16, mad(level(a[j]), 1 << 24, hi[c + j]));
        tmem_ld8(tacc + 64 * 2 + c, a);
        tmem_ld8(tacc + 64 * 3 + c, b);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) hi[c + j] = mad(level(b[j]), 1, mad(level(a[j]), 1 << 8, hi[c + j]));
      }
      ++G;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&free_hi);
    };
    // writes the 16 results of this thread for tile t
    auto put_tile = [&](int t) __attribute__((always_inline)) {
      int xt, yt, z;
      place(t, xt, yt, z);
      const long x = (long)xt * DX + quad * 32 + lane;
      const long y0 = (long)yt * DY + 16 * cg;
      // columns of this warp inside C (symmetric: those up to x)
      const int left = (int)min(16l, (g.sym ? min((long)g.y.rows, x + 1) : (long)g.y.rows) - y0);
      const bool in = x < g.x.rows;
      const int e = row_exp(in ? __ldg(g.x.scale + x) : 0) - 38;
      // the 16 rows' exponents: lane j holds that of row j
      const int ye = row_exp(y0 + (lane & 15) < g.y.rows ? __ldg(g.y.scale + y0 + (lane & 15)) : 0);
      const bool split = g.ksplit > 1;
      const long ld = split ? g.N : g.ldc;
      double* c = (split ? g.work + (long)z * g.M * g.N : g.C) +
                  (g.swapped ? y0 * ld + x : x * ld + y0);
      const long step = g.swapped ? ld : 1;
      const double* h = g.H + (g.swapped ? y0 * g.ldh + x : x * g.ldh + y0);
      if (g.nbatch > 0) {
        const long q = x / g.nbatch;
        c += q * g.cskip;
        h -= q * g.nbatch;
      }
      const long hstep = g.swapped ? g.ldh : 1;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        hi[j] = __double_as_longlong(pack_f64(hi[j], lo[j], e + __shfl_sync(0xffffffffu, ye, j)));
      // with H; the maxima are what rowmax_*_kernel would find in C (in this form of the
      // kernel alone: the others' registers, and 2 % of their time, are spared)
      if (XK && YK && g.xmax) {
        const int mine = in ? left : 0;
        uint32_t mx = 0, my = 0;
        double w[4];
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = j + i < mine ? h[(j + i) * hstep] : 0.0;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t b = 0;
            if (j + i < mine) {
              const double v = __longlong_as_double(hi[j + i]) * w[i];
              c[(j + i) * step] = v;
              b = (uint32_t)__double2hiint(v) & 0x7fffffffu;
            }
            mx = max(mx, b);
            b = __reduce_max_sync(0xffffffffu, b);
            if (lane == j + i) my = b;
          }
        }
        if (in) atomicMax(g.xmax + x, (int)mx);
        if (lane < left) atomicMax(g.ymax + y0 + lane, (int)my);
        return;
      }
      if (!in) return;
      // branches around the FP64 operations: one that is only predicated off
      // would still take its 16 cycles of the FP64 pipe
      if (!split && g.sym) {  // and its mirror image
        double* cm = g.C + x * ld + y0;
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (j < left) {
            double v = __longlong_as_double(hi[j]);
            if (g.scaled) v *= g.alpha;
            c[j * step] = v;
            cm[j] = v;
          }
      } else if (!split && (g.scaled || g.added)) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (j < left) {
            double v = __longlong_as_double(hi[j]) * g.alpha;
            if (g.H) v *= h[j * hstep];
            if (g.added) v += g.beta * c[j * step];
            c[j * step] = v;
          }
      } else if (!split && g.H) {
        double w[4];
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = j + i < left ? h[(j + i) * hstep] : 0.0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (j + i < left) c[(j + i) * step] = __longlong_as_double(hi[j + i]) * w[i];
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (j < left) c[j * step] = __longlong_as_double(hi[j]);
      }
    };

    open_tile();
    if (fn) fetch();
    int it = 0, done = -1;  // done: tile whose results wait in hi, lo
    int dt = -1;            // tile of the block produced last
    int dkb = 0, dn = 0;
    bool due = false;       // the block produced last ended a group
    int par = 1;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const int nkb = kblocks(t / g.tiles);
      par ^= 1;
      for (int kb = 0; kb < nkb && ok; ++kb, ++it) {
        const int s = it % D_STAGES, use = it / D_STAGES;
        if (__shfl_sync(0xffffffffu, (int)abort_flag, 0) ||
            (use > 0 && !wait(&empty[s], (use - 1) & 1))) { lost(); break; }
        uint8_t* st = sm + s * D_STAGE;
        store_block<8, XK>(st, exps[warp][par], tid, vx);
        if (!vkeep) store_block<4, YK>(st + kDig * DX_PLANE, exps[warp][par] + 32, tid, vy);
        auto arrive = [&]() {
          fence_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[s]);
        };
        // the next block's loads fly during the wait above; after a group they
        // follow its taking (registers)
        if (due || done >= 0) {
          arrive();
          if (done >= 0) { put_tile(done); done = -1; }
          if (due) {  // the group that ended with the block before this one
            take_group(dkb < D_GROUP);
            if (dkb == dn - 1) done = dt;
          }
          if (fn) fetch();
        } else {
          if (fn) fetch();
          arrive();
        }
        due = (kb % D_GROUP) == D_GROUP - 1 || kb == nkb - 1;
        dt = t;
        dkb = kb;
        dn = nkb;
      }
    }
    if (ok && done >= 0) put_tile(done);
    if (ok && due) {
      take_group(dkb < D_GROUP);
      if (ok && dkb == dn - 1) put_tile(dt);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == D_WORK) tmem_dealloc(tbase, 512);
}

// Per row: high word of max |x| (the largest of all for infinities and NaN).
// K contiguous: one warp per row and K chunk (blockIdx.y).
__global__ void rowmax_kc_kernel(const double* __restrict__ p, long ld, int rows, int K, int kchunk,
                                 int* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const long r = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const int k0 = blockIdx.y * kchunk, k1 = min(K, k0 + kchunk);
  const double* row = p + r * ld;
  int m = 0;
  for (int k = k0 + lane; k < k1; k += 32) m = max(m, __double2hiint(row[k]) & 0x7fffffff);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) atomicMax(out + r, m);
}

// Rows contiguous (element (r, k) at p[k ld + r]): one thread per row and K chunk.
__global__ void rowmax_rc_kernel(const double* __restrict__ p, long ld, int rows, int K, int kchunk,
                                 int* __restrict__ out) {
  const long r = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  const int k0 = blockIdx.y * kchunk, k1 = min(K, k0 + kchunk);
  int m = 0;
#pragma unroll 4
  for (int k = k0; k < k1; ++k) m = max(m, __double2hiint(p[k * ld + r]) & 0x7fffffff);
  atomicMax(out + r, m);
}

void launch_rowmax(const DOperand& o, int K, int* out, cudaStream_t s) {
  // chunks of K so that about 8 blocks per SM read the operand
  const int rb = o.kc ? (o.rows + 7) / 8 : (o.rows + 255) / 256;
  const int want = std::max(1, (8 * 152 + rb - 1) / rb);
  const int kchunk = std::max(o.kc ? 256 : 64, (K + want - 1) / want);
  const dim3 grid((unsigned)rb, (unsigned)((K + kchunk - 1) / kchunk));
  if (o.kc)
    rowmax_kc_kernel<<<grid, 256, 0, s>>>(o.p, o.ld, o.rows, K, kchunk, out);
  else
    rowmax_rc_kernel<<<grid, 256, 0, s>>>(o.p, o.ld, o.rows, K, kchunk, out);
  count_launch();
}

}  // namespace

size_t digit_scale_ints(int M, int N) { return (size_t)M + N + 8; }

// 2e7 multiply-adds take the FP64 pipe 35 us with every SM at work; the row
// maxima, the launches and a tile here take about 25 us.
bool digit_gemm_wanted(const DGemm& g) {
  return g.scale && g.K >= 16 && std::min(g.M, g.N) >= 8 &&
         (double)g.M * g.N * g.K >= 2e7;
}

// One K group: the product is not split, so its epilogue has every final result.
bool digit_maxima(const DGemm& g) {
  return digit_gemm_wanted(g) && !g.transA && g.transB && g.H && g.K <= 256 && g.alpha == 1.0 && g.beta == 0.0 && !g.sym &&
         g.nbatch == 0 && !in_place(g);
}

// K split (at most cap) of least time: waves of tiles over the SMs times the
// 256-term groups of a tile, with one group's time for a tile's start and end.
int digit_ksplit(int M, int N, int K, bool sym, int cap) {
  const int X = std::max(M, N), Y = std::min(M, N), tx = (X + DX - 1) / DX, ty = (Y + DY - 1) / DY;
  const long tiles = sym ? sym_tiles(tx, ty) : (long)tx * ty;
  const int groups = (K + 255) / 256;
  int best = 1;
  long cost = 0;
  for (int ks = 1; ks <= std::min(cap, groups); ++ks) {
    const long c = ((tiles * ks + 151) / 152) * ((groups + ks - 1) / ks + 1);
    if (ks == 1 || c < cost) { best = ks; cost = c; }
  }
  return best;
}

cudaError_t digit_gemm(const DGemm& g, int ksplit, int kchunk, cudaStream_t s) {
  DArgs a{};
  int* sc = g.scale;  // [flag, 7 unused, M rows of op(A), N columns of op(B)]
  cudaError_t e = cudaMemsetAsync(sc, 0, ((size_t)g.M + g.N + 8) * 4, s);
  if (e != cudaSuccess) return e;
  const DOperand A{g.A, g.lda, g.M, g.transA ? 0 : 1, g.amax ? g.amax : sc + 8};
  const DOperand B{g.B, g.ldb, g.N, g.transB ? 1 : 0, g.bmax ? g.bmax : sc + 8 + g.M};
  if (!g.amax) launch_rowmax(A, g.K, sc + 8, s);
  if (!g.bmax) launch_rowmax(B, g.K, sc + 8 + g.M, s);
  // the longer side of C takes the 128-row side of the tile; as columns of C
  // it also makes the stores contiguous over the lanes
  a.swapped = g.N >= g.M || g.nbatch > 0 ? 1 : 0;
  a.x = a.swapped ? B : A;
  a.y = a.swapped ? A : B;
  a.K = g.K; a.kchunk = kchunk; a.ksplit = ksplit;
  a.tiles_x = (a.x.rows + DX - 1) / DX;
  a.tiles_y = (a.y.rows + DY - 1) / DY;
  a.M = g.M; a.N = g.N; a.C = g.C; a.ldc = g.ldc; a.alpha = g.alpha; a.beta = g.beta;
  a.scaled = g.alpha != 1.0; a.added = g.beta != 0.0; a.careful = a.added || in_place(g);
  if (g.rmax) {
    e = cudaMemsetAsync(g.rmax, 0, (size_t)g.M * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(g.cmax, 0, (size_t)g.N * 4, s);
    if (e != cudaSuccess) return e;
    a.xmax = a.swapped ? g.cmax : g.rmax;
    a.ymax = a.swapped ? g.rmax : g.cmax;
  }
  a.H = g.H; a.ldh = g.ldh; a.work = g.work; a.flag = sc; a.status = g.status; a.wait = g.wait;
  a.nbatch = g.nbatch; a.cskip = g.cskip;
  a.sym = g.sym;
  a.tiles = g.sym ? sym_tiles(a.tiles_x, a.tiles_y) : a.tiles_x * a.tiles_y;
  const long tiles = (long)a.tiles * ksplit;
  const unsigned ctas = (unsigned)std::min<long>(tiles, 152);
  auto launch = [&](auto kernel) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, D_SMEM);
    if (e != cudaSuccess) return e;
    kernel<<<ctas, D_THREADS, D_SMEM, s>>>(a);
    count_launch();
    return cudaGetLastError();
  };
  auto pick = [&](auto s_) {
    constexpr bool S = decltype(s_)::value;
    if (a.x.kc) return a.y.kc ? launch(digit_gemm_kernel<true, true, S>) : launch(digit_gemm_kernel<true, false, S>);
    return a.y.kc ? launch(digit_gemm_kernel<false, true, S>) : launch(digit_gemm_kernel<false, false, S>);
  };
  return short_wait(a.wait) ? pick(std::true_type{}) : pick(std::false_type{});
}

}  // namespace xk
