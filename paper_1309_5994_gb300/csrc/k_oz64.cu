// FP64 series sweep of App. C (and the FP64 Dyson residual) on the BF16 tensor cores:
//     out = B + (Lambda W) X,   X_i(n, k) = sum_{j in NN(i)} J_ij(k) G_j(n, k).
//
// GB300's FP64 pipe does 2 FMA per SM and clock (1.1 TFLOP/s measured), its BF16 tensor cores
// three orders more, so the contraction is done in integer slices (the Ozaki scheme): every
// row of A = [[Re, -Im], [Im, Re]] of Lambda W and every column of X is scaled by a power of two
// below 1 and cut into S = 8 signed 7-bit digits, v = 2^e sum_s q_s 2^{-7 s}, the first 56 bits
// below the row's (column's) largest value.  The digits are small integers, exact in BF16, and
// the products of digits s and t of one diagonal d = s + t accumulate in FP32 in a TMEM block of
// their own: the eight blocks d = 2..9 hold integers.  With |q_1| <= 128, |q_s| <= 64 and at
// most 512 terms (a K segment) the sums of diagonals 2..7 stay within 2^24 and are exact; a sum
// of diagonals 8 and 9 that passed 2^24 would be rounded at 2^-24 of itself, 2^-65 of the
// largest product.  The 36 products with s + t <= 9 leave out terms below 2^-58 of
// max|A_row| max|X_col| each.  The epilogue adds the blocks in int64 at 2^-53 of
// max|A_row| max|X_col| and rounds once to FP64.
//
// Both embeddings are interleaved (row 2 z + part, column 2 z' + part'): an FP64 chunk state
// [i][n][z] complex128 is then a plain real column of 2 Nc entries, the epilogue's stores are
// coalesced, and the two parts of one entry sit in neighbouring lanes (the update norm is the
// complex modulus).
//
// Kernels: k_oz64_aprep (once per Lambda), k_oz64_xprep (gather, scale, digits of X),
// k_oz64_gemm (persistent: bulk copies + tcgen05.mma kind::f16, 128 x 64 tiles); k_oz64_tslice slices the
// operands of a batched complex product (the adjoint's site contraction) for the same kernel.
#include <algorithm>
#include <type_traits>

#include <cuda_bf16.h>

#include "common.cuh"
#include "detail.cuh"
#include "oz64.cuh"
#include "ptx.cuh"

namespace {

constexpr int S = 8;                                      // digits of 7 bits
constexpr int FIX = 7 * S;
constexpr int BM = 128, BN = 64, BK = 32;                 // 32 bf16 = 64-byte rows (64-byte swizzle)
constexpr int ROW_BYTES = BK * 2;
constexpr int A_TILE = BM * BK * 2;                       // 8 KB per A slice
constexpr int X_TILE = BN * BK * 2;                       // 4 KB per X slice
constexpr int STAGE_BYTES = S * (A_TILE + X_TILE);        // 96 KB
constexpr int STAGES = 2;
constexpr int HALF = S / 2;                               // accumulator blocks of a group
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
constexpr int SEG_KB = 512 / BK;                          // k-blocks of one exact K segment
constexpr int THREADS = 640;                              // warp 0 TMA, warp 1 MMA, warps 4-19 epilogue
constexpr int COLS_PER_WARP = BN / 4;
constexpr uint32_t TMEM_COLS = S * BN;                    // one block of 64 columns per diagonal
constexpr int E_BAD = 1 << 20;                            // scale exponent of a row or column with inf or NaN

// kind::f16, D = F32, A = B = BF16, K-major, M = 128 (N set per MMA)
constexpr uint32_t IDESC0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BM >> 4) << 24);

// The slices are stored as the GEMM's shared memory holds them, so that a stage arrives in one or a few bulk
// copies: per site, tile of BT rows (the last one with the R rows that are left) and k-block the S slice
// tiles, R rows of 64 bytes each, 16-byte pieces swizzled as SWIZZLE_64B does.  (Tensor-map copies of
// 64-byte rows delivered 96 KB in 3000 to 6000 cycles, the MMAs on it take 2600.)
struct SliceRow {
  __nv_bfloat162* p;
  size_t block;                                            // pairs of a k-block's S slice tiles
  int slice, sw;                                           // pairs of a slice tile; the row's swizzle
  __device__ __forceinline__ SliceRow(__nv_bfloat16* base, size_t site, int rows, int BT, int row, int Kp) {
    const int t = row / BT, R = min(BT, rows - t * BT), in = row - t * BT;
    slice = R * (BK / 2);
    block = (size_t)S * slice;
    sw = (in >> 1) & 3;
    p = reinterpret_cast<__nv_bfloat162*>(base) + (site * rows + (size_t)t * BT) * ((size_t)Kp / 2 * S) + in * (BK / 2);
  }
  // pair k (elements 2 k, 2 k + 1) of slice 1; slice s lies (s - 1) * slice further
  __device__ __forceinline__ __nv_bfloat162* at(int k) const {
    return p + (size_t)(k / (BK / 2)) * block + ((((k >> 2) & 3) ^ sw) << 2) + (k & 3);
  }
};

struct Oz64State {
  __nv_bfloat16* as = nullptr;        // tiles of the 2 Nc rows of every site (SliceRow)
  int* esig = nullptr;                // [Nr][2Nc] row scale exponents
  size_t a_bytes = 0, sig_bytes = 0;
  bool a_ready = false;
  __nv_bfloat16* xs = nullptr;        // tiles of the ncol columns of every site
  int* etau = nullptr;                // [Nr][ncol] column scale exponents
  size_t x_bytes = 0, tau_bytes = 0;
  int* d_err = nullptr;
  int num_sms = 1;
  bool smem_set = false;
};

int k_pad(int Nc) { return (2 * Nc + BK - 1) / BK * BK; }

// digits of |x| 2^{FIX - e} (|x| < 2^e) in one pass: with 64 added in every digit position below
// the top, digit s of the sum in base 128, less 64, is the balanced digit in [-64, 63]
__device__ __forceinline__ unsigned long long biased_digits(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF);
  const unsigned long long M = E == 0 ? 0 : ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52));
  const int sh = E - 1075 + FIX - e;                       // <= 3
  unsigned long long v;
  if (sh >= 0) {
    v = M << min(sh, 8);
  } else {
    const int r = min(-sh, 63);
    v = (M + ((1ull << r) >> 1)) >> r;
  }
  constexpr unsigned long long BIAS = [] {
    unsigned long long s = 0;
    for (int k = 2; k <= S; ++k) s += 64ull << (7 * (S - k));
    return s;
  }();
  return v + BIAS;
}
// Digit s (1..S) of two values as packed bf16 integers, signs applied.  The bits 0x4300 + j are
// the bf16 number 128 + j for j = 0..128, so one exact packed FMA by +-1 subtracts the offset
// (128 for the top digit, 128 + 64 for the balanced ones) and sets the sign: six instructions a
// pair, where integer-to-float conversions took sixteen.
struct PairSigns {
  __nv_bfloat162 one, top, low;                            // +-1, -+128, -+192 per half
};
__device__ __forceinline__ __nv_bfloat162 as_bf162(unsigned int u) { return *reinterpret_cast<__nv_bfloat162*>(&u); }
__device__ __forceinline__ PairSigns pair_signs(bool neg_lo, bool neg_hi) {
  const unsigned int f = (neg_lo ? 0x8000u : 0u) | (neg_hi ? 0x80000000u : 0u);
  return {as_bf162(0x3F803F80u ^ f), as_bf162(0xC300C300u ^ f), as_bf162(0xC340C340u ^ f)};
}
template <int s>
__device__ __forceinline__ __nv_bfloat162 digit_pair(unsigned long long lo, unsigned long long hi, PairSigns g) {
  constexpr int sh = 7 * (S - s);
  constexpr unsigned int mask = s == 1 ? 0xFFu : 0x7Fu;
  const unsigned int j = ((unsigned int)(lo >> sh) & mask) | (((unsigned int)(hi >> sh) & mask) << 16);
  return __hfma2(as_bf162(j + 0x43004300u), g.one, s == 1 ? g.top : g.low);
}
template <int s = 1, class F>
__device__ __forceinline__ void each_digit(F&& f) {
  f(std::integral_constant<int, s>());
  if constexpr (s < S) each_digit<s + 1>(f);
}
__device__ __forceinline__ bool sign_of(double x) { return __double2hiint(x) < 0; }

// exponent e with |v| < 2^e for every v whose |high word| is at most mb; E_BAD for inf or NaN
__device__ __forceinline__ int scale_exponent(unsigned int mb) {
  const int E = (int)(mb >> 20);
  return E == 0x7FF ? E_BAD : (E == 0 ? 0 : E - 1022);
}

// One warp per (site i, contour row z): the two rows 2 z (Re, -Im) and 2 z + 1 (Im, Re) of the
// embedding share their digits and their scale.  Jrow (hopping equal on every bond): column z'
// also carries J(t(z')), so that X is the plain sum of the neighbours' columns.
__global__ void __launch_bounds__(256) k_oz64_aprep(const double2* __restrict__ lam, const double* __restrict__ Jrow,
                                                    int Nr, int Nt, int Nm, double dt, double beta, int Kp,
                                                    __nv_bfloat16* __restrict__ as, int* __restrict__ esig) {
  const int Nc = 2 * Nt + Nm, N2 = 2 * Nc;
  const size_t row = (size_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (row >= (size_t)Nr * Nc) return;
  const double2* lrow = lam + row * Nc;
  auto value = [&](int k) {
    double2 v = cmul(lrow[k], contour_weight(k, Nt, Nm, dt, beta));
    if (Jrow) {
      const double j = Jrow[contour_time_index(k, Nt)];
      v.x *= j;
      v.y *= j;
    }
    return v;
  };
  unsigned int mb = 0;
  for (int k = lane; k < Nc; k += 32) {
    const double2 v = value(k);
    mb = max(mb, max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu));
  }
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  const int e = scale_exponent(mb);
  const size_t r0 = 2 * row;                               // = i N2 + 2 z
  if (lane < 2) esig[r0 + lane] = e;
  const SliceRow dst(as, row / Nc, N2, BM, 2 * (int)(row % Nc), Kp);
  for (int k = lane; 2 * k < Kp; k += 32) {
    const double2 v = k < Nc ? value(k) : make_double2(0.0, 0.0);
    const unsigned long long Ar = biased_digits(v.x, e), Ai = biased_digits(v.y, e);
    const bool nr = sign_of(v.x), ni = sign_of(v.y);
    const PairSigns top = pair_signs(nr, !ni), bot = pair_signs(ni, nr);
    each_digit([&](auto sc) {
      constexpr int s = decltype(sc)::value;
      __nv_bfloat162* d = dst.at(k) + (s - 1) * dst.slice;
      d[0] = digit_pair<s>(Ar, Ai, top);
      d[BK / 2] = digit_pair<s>(Ai, Ar, bot);              // the next row: the same swizzle
    });
  }
}

// One warp per (site i, vector column n), sites fastest (the four reads of a neighbour's column
// meet in L2): X = sum_j J_ij G_j in FP64, column scale, digits.  UNIFORM: J sits in the Lambda
// slices.  PER_LANE contour points per lane in registers; PER_LANE = 0: any Nc, X summed twice.
// Bound by the FP64 pipe (83 % busy): 8x8, Nc = 64, 4096 columns 0.259 ms with four additions per part,
// 0.197 with the three it needs (floor of its bytes 0.118).
template <bool UNIFORM, int PER_LANE>
__global__ void __launch_bounds__(256) k_oz64_xprep(const double2* G, const double* __restrict__ Jtab,
                                                    const int* __restrict__ nbr, const int* __restrict__ nbond, int Nr,
                                                    int Nt, int Nc, int ncol, int Kp, __nv_bfloat16* __restrict__ xs,
                                                    int* __restrict__ etau, const int* __restrict__ run) {
  ptx::grid_launch_next();
  ptx::grid_wait();
  if (run && !*(volatile const int*)run) return;           // the series has stopped
  const size_t wi = (size_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (wi >= (size_t)Nr * ncol) return;
  const int i = (int)(wi % Nr), n = (int)(wi / Nr);
  const size_t w = (size_t)i * ncol + n;
  const double2* col[4];
  const double* jrow[4];
  bool has[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = nbr[i * 4 + q];
    has[q] = j >= 0;
    col[q] = G + ((size_t)(has[q] ? j : i) * ncol + n) * Nc;
    if (!UNIFORM) jrow[q] = Jtab + (size_t)(has[q] ? nbond[i * 4 + q] : 0) * Nt;
  }
  auto gather = [&](int z) {
    double2 x = make_double2(0.0, 0.0);
    const int tk = UNIFORM ? 0 : contour_time_index(z, Nt);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (!has[q]) continue;
      const double2 g = ptx::load_d2(col[q] + z);
      if (UNIFORM) {
        if (q == 0) {                                      // (x is still zero: one FP64 addition less)
          x = g;
        } else {
          x.x += g.x;
          x.y += g.y;
        }
      } else {
        const double j = jrow[q][tk];
        x.x = q == 0 ? j * g.x : fma(j, g.x, x.x);
        x.y = q == 0 ? j * g.y : fma(j, g.y, x.y);
      }
    }
    return x;
  };
  constexpr int NREG = PER_LANE > 0 ? PER_LANE : 1;
  double2 x[NREG];
  unsigned int mb = 0;
  auto fold = [&](double2 v) {
    mb = max(mb, max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu));
  };
  if (PER_LANE > 0) {
#pragma unroll
    for (int u = 0; u < NREG; ++u) {
      const int z = lane + 32 * u;
      x[u] = z < Nc ? gather(z) : make_double2(0.0, 0.0);
      fold(x[u]);
    }
  } else {
    for (int z = lane; z < Nc; z += 32) fold(gather(z));
  }
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  const int e = scale_exponent(mb);
  if (lane == 0) etau[w] = e;
  const SliceRow dst(xs, i, ncol, BN, n, Kp);
  auto put = [&](int z, double2 v) {
    const unsigned long long Ar = biased_digits(v.x, e), Ai = biased_digits(v.y, e);
    const PairSigns g = pair_signs(sign_of(v.x), sign_of(v.y));
    each_digit([&](auto sc) {
      constexpr int s = decltype(sc)::value;
      dst.at(z)[(s - 1) * dst.slice] = digit_pair<s>(Ar, Ai, g);
    });
  };
  if (PER_LANE > 0) {
#pragma unroll
    for (int u = 0; u < NREG; ++u) {
      const int z = lane + 32 * u;
      if (2 * z < Kp) put(z, x[u]);
    }
  } else {
    for (int z = lane; 2 * z < Kp; z += 32) put(z, z < Nc ? gather(z) : make_double2(0.0, 0.0));
  }
}

// Operands of a batched complex product C_b[u][t] = sum_i X_b[i][u] A_b[i][t] (b < batch, i < nk; A, X stored
// [b][i][t], t < Nc): the digits of A_b^T as the embedding's rows (AROWS: rows 2 t and 2 t + 1, esig) or
// of X_b^T as columns (etau), the summed index i running along the slices' rows.  One block per (b, 32
// values of t): the scale from one pass over i, the digits from a second one through shared memory, so
// that reads are coalesced in t and writes in i.
template <bool AROWS>
__global__ void __launch_bounds__(256) k_oz64_tslice(const double2* __restrict__ V, int nk, int Nc, int Kp, int batch,
                                                     __nv_bfloat16* __restrict__ sl, int* __restrict__ ex) {
  __shared__ double2 tile[32][33];
  __shared__ unsigned int smax[8][32];
  const int b = blockIdx.y, t0 = blockIdx.x * 32, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double2* Vb = V + (size_t)b * nk * Nc;
  unsigned int mb = 0;
  if (t0 + lane < Nc)
    for (int i = warp; i < nk; i += 8) {
      const double2 v = Vb[(size_t)i * Nc + t0 + lane];
      mb = max(mb, max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu));
    }
  smax[warp][lane] = mb;
  __syncthreads();
  if (warp == 0) {
    for (int q = 1; q < 8; ++q) mb = max(mb, smax[q][lane]);
    smax[0][lane] = (unsigned int)scale_exponent(mb);
  }
  __syncthreads();
  const int rows = AROWS ? 2 * Nc : Nc;                    // slice rows per batch entry
  if (threadIdx.x < 32 && t0 + lane < Nc) {
    const int e = (int)smax[0][lane];
    if (AROWS) ex[(size_t)b * rows + 2 * (t0 + lane)] = ex[(size_t)b * rows + 2 * (t0 + lane) + 1] = e;
    else ex[(size_t)b * rows + t0 + lane] = e;
  }
  for (int i0 = 0; 2 * i0 < Kp; i0 += 32) {
    for (int r = warp; r < 32; r += 8)
      tile[r][lane] = i0 + r < nk && t0 + lane < Nc ? Vb[(size_t)(i0 + r) * Nc + t0 + lane] : make_double2(0.0, 0.0);
    __syncthreads();
    if (2 * (i0 + lane) < Kp)
      for (int r = warp; r < 32 && t0 + r < Nc; r += 8) {
        const double2 v = tile[lane][r];
        const int e = (int)smax[0][r];
        const unsigned long long Ar = biased_digits(v.x, e), Ai = biased_digits(v.y, e);
        const bool nr = sign_of(v.x), ni = sign_of(v.y);
        const SliceRow dst(sl, b, rows, AROWS ? BM : BN, (AROWS ? 2 : 1) * (t0 + r), Kp);
        const PairSigns top = pair_signs(nr, AROWS ? !ni : ni), bot = pair_signs(ni, nr);
        each_digit([&](auto sc) {
          constexpr int s = decltype(sc)::value;
          __nv_bfloat162* d = dst.at(i0 + lane) + (s - 1) * dst.slice;
          d[0] = digit_pair<s>(Ar, Ai, top);
          if (AROWS) d[BK / 2] = digit_pair<s>(Ai, Ar, bot);
        });
      }
    __syncthreads();
  }
}

// V 2^e as FP64, rounded to nearest (halves away from zero); 0 below the normal range, inf above it
__device__ __forceinline__ double fixed_to_double(long long V, int e) {
  const unsigned long long a = (unsigned long long)(V < 0 ? -V : V);
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);              // leading bit at 63
  const unsigned long long q = (m >> 11) + ((m >> 10) & 1);  // 53 bits, the leading one adds 1 to the exponent
  const int ex = 1085 - lz + e;
  unsigned long long bits = ((unsigned long long)(unsigned)ex << 52) + q;
  if (ex >= 2045) bits = 0x7FF0000000000000ull;
  if (ex < 1 || a == 0) bits = 0;
  if (e >= E_BAD / 2) bits = 0x7FF8000000000000ull;
  return __longlong_as_double((long long)(bits | ((unsigned long long)V & 0x8000000000000000ull)));
}

// The same where every nonzero result is in the normal range (|e| < 900), in two thirds of the instructions
__device__ __forceinline__ double fixed_to_double_normal(long long V, int e) {
  const unsigned long long a = (unsigned long long)(V < 0 ? -V : V);
  const unsigned int ah = (unsigned int)(a >> 32), al = (unsigned int)a;
  const unsigned int hi = ah ? ah : al, lo = ah ? al : 0u;
  const int lz = __clz((int)hi);
  const unsigned int mh = __funnelshift_l(lo, hi, lz), ml = lo << (lz & 31);
  const unsigned long long q = (((unsigned long long)(mh >> 11) << 32) | __funnelshift_r(ml, mh, 11)) + ((ml >> 10) & 1);
  const unsigned int top = (unsigned int)((ah ? 1085 : 1053) - lz + e) << 20;
  const unsigned int h = (unsigned int)(q >> 32) + top;
  return __hiloint2double((int)(((a == 0 ? 0u : h)) | ((unsigned int)(V >> 32) & 0x80000000u)), (int)(unsigned int)q);
}

// The norms decide when an iteration stops, relative to a scale: they are held in FP32 in units of the power of two
// below that scale (24 bits, from 2^-74 to 2^63 of it; the FP64 pipe has no room for their squares).
struct NormUnit {
  unsigned int least;                                      // high word of 2^-126 units
  static constexpr unsigned int SPAN = (0x47E - 0x381) << 20;   // from there to 2^127 units
  __device__ __forceinline__ explicit NormUnit(unsigned long long scale)
      : least((unsigned int)(0x381 + (scale == 0ull ? 0 : max(-880, min(880, (int)(scale >> 52) - 1023)))) << 20) {}
  // |d| in units as FP32, from its bits (truncated; no conversion on the FP64 pipe): 0 outside the span; top keeps
  // the largest high word
  __device__ __forceinline__ float magnitude(double d, unsigned int& top) const {
    const unsigned int hi = (unsigned int)__double2hiint(d) & 0x7FFFFFFFu, lo = (unsigned int)__double2loint(d);
    const unsigned int t = hi - least;
    top = max(top, hi);
    return t < SPAN ? __uint_as_float(__funnelshift_l(lo, t, 3) + 0x00800000u) : 0.f;
  }
  // max of the word with the square root of a running maximum of squares (infinite where an entry lay above the
  // span, or was infinite or not a number)
  __device__ __forceinline__ void flush(float sq, unsigned int top, unsigned long long* norm, int lane) const {
    const float inf = __int_as_float(0x7f800000);
    if (top >= least + SPAN) sq = inf;
    for (int o = 16; o > 0; o >>= 1) sq = fmaxf(sq, __shfl_xor_sync(0xffffffffu, sq, o));
    // (an FP64 square root, even of one lane, holds the SM's FP64 pipe for hundreds of cycles a warp)
    if (lane != 0) return;
    const float m = sqrtf(sq);
    unsigned long long bits = (unsigned long long)__double_as_longlong((double)m);
    if (m > 0.f && m < inf) bits += ((unsigned long long)least << 32) - (0x381ull << 52);
    atomicMax(norm, bits);
  }
};

// Persistent: one CTA per SM walks 128 x 64 output tiles (row tile fastest, then column tile, then
// site).  A stage is a 32-deep k-block of all eight slices of both operands.  Per k16 step,
// slice s of A times slices 1..9-s of X (back to back in the stage) lands in the TMEM blocks of
// diagonals s+1..9: twelve MMAs of N <= 256 for the 36 products.
// The eight accumulators fill TMEM, in two groups with barriers of their own: a segment's last k-block
// finishes diagonals 2..5 first, which the epilogue reads into int64 registers under the products of
// diagonals 6..9, and the next tile's first k-block starts on each group as soon as it is read.  The
// rest of the epilogue overlaps the MMAs.  64 columns per tile, because at 32 (two sets) each A slice
// would be read from L2 twice as often.
// Measured per launch: 10x10, Nc = 128, 512 columns (6.7 GFLOP of FP64) 0.160 ms, 8x8, Nc = 64, 4096
// columns 0.244 ms; the FP64-pipe kernel took 6.33 and 8.04 ms.  On the way there (10x10 / 8x8, ms): one
// accumulator group and tensor-map copies 0.190 / 0.298; the epilogue's loop without branches - / 0.285;
// two groups 0.176 / 0.252; slices in tile order 0.160 / 0.244.  k-blocks of 16 in four stages: 0.173 /
// 0.256 (a k-block of 16 takes 1560 cycles, one of 32 2680; the tensor rate alone would be 2304).
// Nc = 128 is bound by the MMAs, Nc = 64 by the epilogue (about 13000 of a tile's 16500 cycles) and the
// 1.1 GB of DRAM traffic.
template <int MODE>
__global__ void __launch_bounds__(THREADS, 1)
    k_oz64_gemm(const __nv_bfloat16* __restrict__ as, const __nv_bfloat16* __restrict__ xs,
                const int* __restrict__ esig, const int* etau, const double* Gin,
                const double2* __restrict__ lam, const int* __restrict__ src_site, const int* __restrict__ src_time,
                int Nr, int Nc, int KB, int ncol, int gs, double* __restrict__ out, float* __restrict__ r32, int Ns,
                unsigned long long* __restrict__ norm, int* __restrict__ err, const int* __restrict__ run) {
  using namespace ptx;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], acc_full[2], acc_empty[2], drain;
  __shared__ uint32_t tmem_holder;
  __shared__ WaitCtl wctl;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N2 = 2 * Nc;
  const int MT = (N2 + BM - 1) / BM, NT = (ncol + BN - 1) / BN;
  int tiles = MT * NT * Nr;
  const int nseg = (KB + SEG_KB - 1) / SEG_KB;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&acc_full[h], 1);
      mbar_init(&acc_empty[h], 512);
    }
    mbar_init(&drain, 1);
    wait_ctl_init(&wctl);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_holder, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_holder;
  grid_launch_next();
  grid_wait();
  if (run && !*(volatile const int*)run) tiles = 0;        // the series has stopped
  volatile WaitCtl* abort_p = &wctl;
  auto stage_ptr = [&](int s) { return smem + (size_t)s * STAGE_BYTES; };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      int g = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const int mt = tile % MT, nt = (tile / MT) % NT, site = tile / (MT * NT);
        const uint32_t ra = min(BM, N2 - mt * BM) * ROW_BYTES, rx = min(BN, ncol - nt * BN) * ROW_BYTES;
        const uint8_t* pa = reinterpret_cast<const uint8_t*>(as) + ((size_t)site * N2 + mt * BM) * KB * (S * ROW_BYTES);
        const uint8_t* px = reinterpret_cast<const uint8_t*>(xs) + ((size_t)site * ncol + nt * BN) * KB * (S * ROW_BYTES);
        for (int kb = 0; kb < KB; ++kb, ++g) {
          const int s = g % STAGES;
          if (g >= STAGES && !mbar_wait(&empty[s], ((g / STAGES) - 1) & 1, abort_p)) {
            ok = false;
            break;
          }
          uint8_t* st = stage_ptr(s);
          mbar_expect_tx(&full[s], S * (ra + rx));
          // (rows of a tile's end that no copy writes hold what was there: only unused results see them)
          auto load = [&](uint8_t* to, uint32_t tile_bytes, const uint8_t* from, uint32_t bytes) {
            if (bytes == tile_bytes) bulk_load(to, from, S * tile_bytes, &full[s]);
            else
              for (int q = 0; q < S; ++q) bulk_load(to + q * tile_bytes, from + q * bytes, bytes, &full[s]);
          };
          load(st, A_TILE, pa + (size_t)kb * S * ra, ra);
          load(st + S * A_TILE, X_TILE, px + (size_t)kb * S * rx, rx);
        }
      }
      for (int q = g > STAGES ? g - STAGES : 0; q < g; ++q)
        mbar_wait(&full[q % STAGES], (q / STAGES) & 1, abort_p, false);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      int g = 0, t = 0;
      bool ok = true, any = false;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        for (int kb = 0; kb < KB && ok; ++kb, ++g) {
          const bool first = kb % SEG_KB == 0;              // a new segment overwrites the accumulators
          const bool last = kb + 1 == KB || (kb + 1) % SEG_KB == 0;
          const int s = g % STAGES;
          if (!mbar_wait(&full[s], (g / STAGES) & 1, abort_p)) {
            ok = false;
            break;
          }
          const uint32_t base = smem_u32(stage_ptr(s));
          // blocks 0..3 first, so that the epilogue empties them under the other blocks' products
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (first && t >= 1 && !mbar_wait(&acc_empty[h], (t - 1) & 1, abort_p)) {
              ok = false;
              break;
            }
            tc_fence_after();
#pragma unroll
            for (int k16 = 0; k16 < BK / 16; ++k16) {
#pragma unroll
              for (int sl = 0; sl < (h ? S : HALF); ++sl) {
                const int t0 = h && sl < HALF ? HALF - sl : 0;            // first X slice
                const int nblk = (h ? S : HALF) - (h && sl < HALF ? HALF : sl);   // <= 4: N <= 256
                const uint32_t idesc = IDESC0 | ((uint32_t)(nblk * BN >> 3) << 17);
                mma<0>(tmem + (uint32_t)((sl + t0) * BN), sdesc_sw64(base + sl * A_TILE + k16 * 32),
                       sdesc_sw64(base + S * A_TILE + t0 * X_TILE + k16 * 32), idesc,
                       (first && k16 == 0 && sl == 0) ? 0u : 1u);
              }
            }
            any = true;
            if (h) mma_commit(&empty[s]);
            if (last) mma_commit(&acc_full[h]);
          }
          if (last) ++t;
        }
      }
      if (any) {
        mma_commit(&drain);
        mbar_wait(&drain, 0, abort_p, false);
      }
    }
  } else if (warp >= 4) {
    // ---------------- epilogue: warps 4-19, four per TMEM lane quarter ----------------
    const int q4 = warp & 3, part = (warp - 4) >> 2;
    const uint32_t tacc = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(part * COLS_PER_WARP);
    // int64 unit 2^-53 of the scales' product, coarser by the bits that several segments add
    int extra = 0;
    while ((1 << extra) < nseg) ++extra;
    int t = 0;
    bool go = true;
    for (int tile = blockIdx.x; tile < tiles && go; tile += gridDim.x) {
      const int mt = tile % MT, nt = (tile / MT) % NT, site = tile / (MT * NT);
      const int m = mt * BM + q4 * 32 + lane;
      const int n_first = nt * BN + part * COLS_PER_WARP;
      const bool row_ok = m < N2;
      const int es = row_ok ? esig[(size_t)site * N2 + m] : 0;
      const int cols = max(0, min(COLS_PER_WARP, ncol - n_first));
      // lane j < 16: scale exponent and source of the warp's column j (read by shuffle below)
      static_assert(COLS_PER_WARP == 16, "one column per lane of a half warp");
      const int et_l = lane < cols ? load_i(etau + (size_t)site * ncol + n_first + lane) : 0;
      const unsigned src_here =
          __ballot_sync(0xffffffffu, MODE != 2 && lane < cols && __ldg(src_site + n_first + lane) == site);
      int qcur = n_first / gs;
      NormUnit unit(MODE != 2 && cols > 0 ? norm[ncol / gs + qcur] : 0ull);   // (the scales follow the norms)
      unsigned int top = 0;
      const size_t off0 = ((size_t)site * ncol + n_first) * N2 + (row_ok ? m : 0);
      // G of this lane's row, eight columns at a time (the first ones before the wait)
      double gin[2][8];
      auto load_g = [&](int h) {
        const int c = 8 * h;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          gin[h][j] = MODE != 2 && c + j < cols ? load_d(Gin + off0 + (size_t)(c + j) * N2) : 0.0;
      };
      load_g(0);
      long long V[COLS_PER_WARP];
      for (int seg = 0; seg < nseg; ++seg, ++t) {
#pragma unroll
        for (int h = 0; h < 2 && go; ++h) {
          go = mbar_wait(&acc_full[h], t & 1, abort_p);
          go = __all_sync(0xffffffffu, go);                 // tcgen05.ld below is warp-collective
          if (!go) break;
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < COLS_PER_WARP / 4; ++c) {
            uint32_t r[HALF][4];
#pragma unroll
            for (int d = 0; d < HALF; ++d) tmem_ld4(tacc + (uint32_t)((h * HALF + d) * BN + c * 4), r[d]);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              auto f = [&](int d) { return __uint_as_float(r[d][j]); };
              auto n = [&](int d) { return (long long)__float2int_rn(f(d)); };
              long long v;
              if (h == 0) {                                 // diagonals 2..5: a multiple of 2^18
                v = n(3) * (1ll << 18) + n(2) * (1ll << 25) + (n(1) + n(0) * (1ll << 7)) * (1ll << 32);
                if (extra) v >>= extra;
                V[c * 4 + j] = seg ? V[c * 4 + j] + v : v;
              } else {                                      // 6 and 7; 8 and 9 are below the unit's last bits
                v = (long long)__float2int_rn(fmaf(f(3), 0x1p-10f, f(2) * 0x1p-3f));
                v += n(1) * (1ll << 4) + n(0) * (1ll << 11);
                if (extra) v = (v + (1ll << (extra - 1))) >> extra;
                V[c * 4 + j] += v;
              }
            }
          }
          tc_fence_before();
          mbar_arrive(&acc_empty[h]);                       // the next segment's MMAs may start
        }
        if (!go) break;
      }
      if (!go) break;
      load_g(1);
      int left = min(COLS_PER_WARP, (qcur + 1) * gs - n_first);   // columns to the next norm group
      float sq = 0.f;                                       // running max |d|^2 of the group
      // A whole tile without sources, in one norm group and far from the ends of the exponent range takes
      // a loop without branches, whose columns overlap; two columns share a shuffle for their norms.
      if (MODE == 0 && cols == COLS_PER_WARP && left == COLS_PER_WARP && src_here == 0 &&
          __all_sync(0xffffffffu, row_ok && abs(es) < 400 && abs(et_l) < 400)) {
        const bool odd = lane & 1;
#pragma unroll
        for (int j = 0; j < COLS_PER_WARP; j += 2) {
          float a2[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int et = __shfl_sync(0xffffffffu, et_l, j + u);
            const double y = fixed_to_double_normal(V[j + u], es + et - 53 + extra);
            out[off0 + (size_t)(j + u) * N2] = y;
            const float a = unit.magnitude(y - gin[j / 8][(j + u) % 8], top);
            a2[u] = a * a;
          }
          const float other = __shfl_xor_sync(0xffffffffu, odd ? a2[0] : a2[1], 1);
          sq = fmaxf(sq, (odd ? a2[1] : a2[0]) + other);
        }
        unit.flush(sq, top, norm + qcur, lane);
        continue;
      }
#pragma unroll
      for (int j = 0; j < COLS_PER_WARP; ++j) {
        const int et = __shfl_sync(0xffffffffu, et_l, j);
        double y = fixed_to_double(V[j], es + et - 53 + extra);
        if (j >= cols) continue;                            // warp-uniform
        if (MODE == 2) {                                    // a plain product
          if (row_ok) out[off0 + (size_t)j * N2] = y;
          continue;
        }
        if (j == left) {
          unit.flush(sq, top, norm + qcur, lane);
          ++qcur;
          unit = NormUnit(norm[ncol / gs + qcur]);
          top = 0;
          left = j + gs;
          sq = 0.f;
        }
        if ((src_here >> j & 1) && row_ok) {                // B = Lambda_s e_{z'}
          const double2 b = lam[((size_t)site * Nc + (m >> 1)) * Nc + src_time[n_first + j]];
          y += (m & 1) ? b.y : b.x;
        }
        const double d = y - gin[j / 8][j % 8];
        const float a = row_ok ? unit.magnitude(d, top) : 0.f;
        if (row_ok) {
          if (MODE == 0) out[off0 + (size_t)j * N2] = y;
          else r32[((size_t)site * ncol + n_first + j) * 2 * Ns + (m >> 1) + ((m & 1) ? Ns : 0)] = (float)d;
        }
        const float a2 = a * a;
        sq = fmaxf(sq, a2 + __shfl_xor_sync(0xffffffffu, a2, 1));
      }
      if (MODE != 2 && cols > 0) unit.flush(sq, top, norm + qcur, lane);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
  // a wait that ran out raises the flag and makes the norm infinite, so that the host looks at the
  // flag only where a norm is not finite
  if (threadIdx.x == 0 && wctl.abort) {
    atomicExch(err, 1);
    if (MODE != 2) atomicMax(norm, 0x7FF0000000000000ull);
  }
}

Oz64State* state(dyson_ctx* c) {
  if (!c->oz64) c->oz64 = new Oz64State();
  return static_cast<Oz64State*>(c->oz64);
}

template <class T>
int grow(dyson_ctx* c, T** p, size_t* have, size_t bytes, const char* what) {
  if (*have >= bytes) return DYSON_OK;
  if (*p) cudaFree(*p);
  *p = nullptr;
  *have = 0;
  cudaError_t e = cudaMalloc((void**)p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return ctx_fail(c, DYSON_ERR_OOM, std::string(what) + ": " + cudaGetErrorString(e));
  }
  *have = bytes;
  return DYSON_OK;
}

size_t a_slice_bytes(const dyson_ctx* c) { return (size_t)S * c->Nr * 2 * c->Nc * k_pad(c->Nc) * 2; }

const double* uniform_hopping(const dyson_ctx* c) { return c->j_uniform && c->Nb > 0 ? c->dJ : nullptr; }

template <bool UNIFORM>
void launch_xprep(dyson_ctx* c, int ncol, const double2* G, Oz64State* st, const int* run) {
  const size_t warps = (size_t)c->Nr * ncol;
  const unsigned blocks = (unsigned)((warps + 7) / 8);
  const int Kp = k_pad(c->Nc), pts = Kp / 2;               // padded points per column
  auto go = [&](auto kernel) {
    launch_overlapped(run != nullptr, kernel, blocks, 256, 0, c->stream, G, c->dJ, c->d_nbr, c->d_nbond, c->Nr, c->Nt,
                      c->Nc, ncol, Kp, st->xs, st->etau, run);
  };
  if (pts <= 32) go(k_oz64_xprep<UNIFORM, 1>);
  else if (pts <= 64) go(k_oz64_xprep<UNIFORM, 2>);
  else if (pts <= 128) go(k_oz64_xprep<UNIFORM, 4>);
  else if (pts <= 256) go(k_oz64_xprep<UNIFORM, 8>);
  else go(k_oz64_xprep<UNIFORM, 0>);
}

}  // namespace

bool oz64_usable(dyson_ctx* c, size_t* more) {
  *more = 0;
  if (c->slice_memory >= 0 && (int64_t)a_slice_bytes(c) > c->slice_memory) return false;
  Oz64State* st = static_cast<Oz64State*>(c->oz64);
  if (st && st->a_bytes >= a_slice_bytes(c)) return true;
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return false;
  *more = a_slice_bytes(c);
  return c->slice_memory >= 0 || a_slice_bytes(c) <= (free_b + dyson_detail::scratch_bytes(c)) / 3;
}

int oz64_reserve(dyson_ctx* c, int ncol) {
  Oz64State* st = state(c);
  int rc;
  if ((rc = grow(c, &st->xs, &st->x_bytes, (size_t)S * c->Nr * ncol * k_pad(c->Nc) * 2, "FP64 slices of X"))) return rc;
  return grow(c, &st->etau, &st->tau_bytes, (size_t)c->Nr * ncol * sizeof(int), "FP64 column scales");
}

size_t oz64_x_bytes(const dyson_ctx* c) {
  const Oz64State* st = static_cast<const Oz64State*>(c->oz64);
  return st ? st->x_bytes + st->tau_bytes : 0;
}

void oz64_release_x(dyson_ctx* c) {
  Oz64State* st = static_cast<Oz64State*>(c->oz64);
  if (!st) return;
  cudaFree(st->xs);
  cudaFree(st->etau);
  st->xs = nullptr;
  st->etau = nullptr;
  st->x_bytes = st->tau_bytes = 0;
}

double oz64_bytes_per_element(const dyson_ctx* c) {
  return (double)S * 2 * k_pad(c->Nc) / c->Nc + 4.0 / c->Nc;
}

void oz64_invalidate(dyson_ctx* c) {
  if (c->oz64) static_cast<Oz64State*>(c->oz64)->a_ready = false;
}

namespace {
int prepare_common(dyson_ctx* c) {
  Oz64State* st = state(c);
  if (!st->d_err) {
    DY_CUDA(c, cudaMalloc(&st->d_err, sizeof(int)));
    DY_CUDA(c, cudaMemsetAsync(st->d_err, 0, sizeof(int), c->stream));
    DY_CUDA(c, cudaDeviceGetAttribute(&st->num_sms, cudaDevAttrMultiProcessorCount, c->device));
  }
  if (!st->smem_set) {
    DY_CUDA(c, cudaFuncSetAttribute(k_oz64_gemm<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    DY_CUDA(c, cudaFuncSetAttribute(k_oz64_gemm<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    DY_CUDA(c, cudaFuncSetAttribute(k_oz64_gemm<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    st->smem_set = true;
  }
  return DYSON_OK;
}
}  // namespace

int oz64_prepare(dyson_ctx* c) {
  Oz64State* st = state(c);
  const int Nr = c->Nr, Nc = c->Nc, N2 = 2 * Nc, Kp = k_pad(Nc);
  int rc = prepare_common(c);
  if (rc) return rc;
  if (!st->a_ready) {
    if ((rc = grow(c, &st->as, &st->a_bytes, a_slice_bytes(c), "FP64 slices of Lambda"))) return rc;
    if ((rc = grow(c, &st->esig, &st->sig_bytes, (size_t)Nr * N2 * sizeof(int), "FP64 row scales"))) return rc;
    const size_t rows = (size_t)Nr * Nc;
    k_oz64_aprep<<<(unsigned)((rows + 7) / 8), 256, 0, c->stream>>>(c->d_lam, uniform_hopping(c), Nr, c->Nt, c->Nm,
                                                                   c->dt, c->beta, Kp, st->as, st->esig);
    DY_CUDA(c, cudaGetLastError());
    c->launches += 1;
    st->a_ready = true;
  }
  return DYSON_OK;
}

int oz64_sweep(dyson_ctx* c, int ncol, int gs, const double2* Gin, double2* out, float* r32, int mode,
               const int* run) {
  int rc = oz64_prepare(c);
  if (rc) return rc;
  Oz64State* st = state(c);
  const int Nr = c->Nr, Nc = c->Nc, N2 = 2 * Nc, Kp = k_pad(Nc);
  if ((rc = oz64_reserve(c, ncol))) return rc;
  if (uniform_hopping(c)) launch_xprep<true>(c, ncol, Gin, st, run);
  else launch_xprep<false>(c, ncol, Gin, st, run);
  DY_CUDA(c, cudaGetLastError());
  const long long tiles = (long long)((N2 + BM - 1) / BM) * ((ncol + BN - 1) / BN) * Nr;
  const int grid = (int)std::min<long long>(tiles, st->num_sms);
  auto go = [&](auto kernel) {
    launch_overlapped(run != nullptr, kernel, (unsigned)grid, THREADS, SMEM_BYTES, c->stream, st->as, st->xs, st->esig,
                      st->etau, reinterpret_cast<const double*>(Gin), c->d_lam, c->d_src_site, c->d_src_time, Nr, Nc,
                      Kp / BK, ncol, gs, reinterpret_cast<double*>(out), r32, c->Ns, c->d_norm, st->d_err, run);
  };
  if (mode == 0) go(k_oz64_gemm<0>);
  else go(k_oz64_gemm<1>);
  DY_CUDA(c, cudaGetLastError());
  c->launches += 2;
  return DYSON_OK;
}

int oz64_batched_product(dyson_ctx* c, int batch, int nk, int Nc, const double2* A, const double2* X, double2* out) {
  int rc = prepare_common(c);
  if (rc) return rc;
  Oz64State* st = state(c);
  const int Kp = (2 * nk + BK - 1) / BK * BK, N2 = 2 * Nc;
  // scratch for as many entries at a time as fit in a sixteenth of the free memory, or in what the caller allows
  const size_t per_a = (size_t)S * N2 * Kp * 2, per_x = per_a / 2, per_e = (size_t)3 * Nc * sizeof(int);
  size_t free_b = 0, total_b = 0;
  DY_CUDA(c, cudaMemGetInfo(&free_b, &total_b));
  const size_t per = per_a + per_x + per_e;
  const int step = (int)std::min<size_t>(batch, (c->slice_memory >= 0 ? (size_t)c->slice_memory : free_b / 16) / per);
  if (step < 1) return DYSON_ERR_OOM;
  char* buf = nullptr;
  if (cudaMalloc((void**)&buf, step * per) != cudaSuccess) {
    cudaGetLastError();
    return DYSON_ERR_OOM;
  }
  auto* as = reinterpret_cast<__nv_bfloat16*>(buf);
  auto* xs = reinterpret_cast<__nv_bfloat16*>(buf + step * per_a);
  int* esig = reinterpret_cast<int*>(buf + step * (per_a + per_x));
  int* etau = esig + (size_t)step * N2;
  rc = DYSON_OK;
  cudaError_t e = cudaSuccess;
  for (int b0 = 0; b0 < batch && rc == DYSON_OK && e == cudaSuccess; b0 += step) {
    const int nb = std::min(step, batch - b0);
    const dim3 grid((Nc + 31) / 32, nb);
    const size_t o = (size_t)b0 * nk * Nc;
    k_oz64_tslice<true><<<grid, 256, 0, c->stream>>>(A + o, nk, Nc, Kp, nb, as, esig);
    k_oz64_tslice<false><<<grid, 256, 0, c->stream>>>(X + o, nk, Nc, Kp, nb, xs, etau);
    const long long tiles = (long long)((N2 + BM - 1) / BM) * ((Nc + BN - 1) / BN) * nb;
    k_oz64_gemm<2><<<(int)std::min<long long>(tiles, st->num_sms), THREADS, SMEM_BYTES, c->stream>>>(
        as, xs, esig, etau, nullptr, nullptr, nullptr, nullptr, nb, Nc, Kp / BK, Nc, Nc,
        reinterpret_cast<double*>(out + (size_t)b0 * Nc * Nc), nullptr, Nc, nullptr, st->d_err, nullptr);
    c->launches += 3;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && rc == DYSON_OK) rc = oz64_check_error(c);   // (waits for the stream: the scratch goes now)
  else cudaStreamSynchronize(c->stream);
  cudaFree(buf);
  if (e != cudaSuccess) return ctx_fail(c, DYSON_ERR_CUDA, std::string("batched product: ") + cudaGetErrorString(e));
  return rc;
}

int oz64_set_wait_limit(dyson_ctx* c, unsigned long long ns) {
  DY_CUDA(c, cudaMemcpyToSymbolAsync(ptx::g_wait_limit_ns, &ns, sizeof ns, 0, cudaMemcpyHostToDevice, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  return DYSON_OK;
}

int oz64_check_error(dyson_ctx* c) {
  Oz64State* st = static_cast<Oz64State*>(c->oz64);
  if (!st || !st->d_err) return DYSON_OK;
  int flag = 0;
  DY_CUDA(c, cudaMemcpyAsync(&flag, st->d_err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  if (!flag) return DYSON_OK;
  DY_CUDA(c, cudaMemsetAsync(st->d_err, 0, sizeof(int), c->stream));
  return ctx_fail(c, DYSON_ERR_TIMEOUT, "an FP64 sweep pipeline wait exceeded its time limit");
}

void oz64_release(dyson_ctx* c) {
  Oz64State* st = static_cast<Oz64State*>(c->oz64);
  if (!st) return;
  void* ptrs[] = {st->as, st->esig, st->xs, st->etau, st->d_err};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete st;
  c->oz64 = nullptr;
}
