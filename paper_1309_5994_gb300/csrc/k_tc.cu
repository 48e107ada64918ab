// K2: one series sweep of App. C on the 5th-generation tensor cores,
//     d_out = r + (Lambda W) X,   X_i(n, k) = sum_{j in NN(i)} J_ij(k) d_in_j(n, k),
// over the FP32 planar chunk state (per vector column: Ns real parts, then Ns
// imaginary parts; Ns is Nc rounded up to a multiple of 64, the padding zeros).
//
//   k_tc_fused   the general form: one persistent launch per sweep on CTA pairs
//                (tcgen05 cta_group::2), the gather X = sum_j J_ij d_j computed by the
//                GEMM's own producer warps, Lambda W and X as FP16 hi + lo halves under
//                power-of-two scales, three products
//                A_hi X_hi + A_hi X_lo + A_lo X_hi accumulated in FP32 in tensor
//                memory (its own comment below has the tiles and the measurements).
// The explicitly selected unfused forms (dyson_set_sweep_variant; Nc % 64 == 0) run 3xTF32 products of
// the real embedding [[Re, -Im], [Im, Re]] (M = K = 2Nc) in two launches per sweep:
//   k_tc_gather  X = sum_j J_ij d_j (FP32, coalesced float4, columns of all
//                sites visited block by block so neighbour rows hit in L2);
//   k_tc_gemm    persistent: one CTA per SM walks 128 x 256 output tiles (row
//                tile fastest, then column tile, then site, so X tiles and the
//                site's Lambda are shared through L2).  Warp roles:
//                  warp 0       TMA loads of A_hi, A_lo, X (128-byte swizzle, 2 stages)
//                  warps 4-7    split X into TF32 hi/lo in place in shared memory
//                  warp 1       one thread issues tcgen05.mma into one of two
//                               256-column TMEM accumulators
//                  warps 8-11   epilogue: tcgen05.ld, + r, store d_out, update norm
//                so the epilogue of one tile overlaps the MMAs of the next.
//   k_tc_gemm_pair  the same GEMM on clusters of two CTAs (256 x 256 tiles, three 64 KB
//                stages).
// Every mbarrier wait is bounded (2 s of %globaltimer); on expiry the CTA
// raises an error flag, lets in-flight copies and MMAs land, frees TMEM and
// exits, and the host returns DYSON_ERR_TIMEOUT.
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "ptx.cuh"
#include "tc.cuh"

namespace {

constexpr int BM = 128, BN = 256, BK = 32, STAGES = 2;
static_assert(BN == TC_TILE_COLS, "support-truncation tables are laid out per GEMM column tile");
constexpr int PREFETCH = 4;                            // k-blocks of L2 prefetch ahead of the loads
constexpr int A_TILE = BM * BK * 4;                    // 16 KB
constexpr int X_TILE = BN * BK * 4;                    // 32 KB
constexpr int STAGE_BYTES = 2 * A_TILE + 2 * X_TILE;   // A_hi, A_lo, X (-> X_hi), X_lo
constexpr int TMA_BYTES = 2 * A_TILE + X_TILE;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
constexpr int THREADS = 384;
constexpr uint32_t ACC_COLS = BN;                      // one accumulator: 128 lanes x 256 fp32
constexpr uint32_t TMEM_COLS = 2 * ACC_COLS;           // double-buffered

// kind::tf32, D = F32, A = B = TF32, both K-major, M = 128, N = 256
constexpr uint32_t IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(BM >> 4) << 24);

struct TcState {
  CUtensorMap a_hi, a_lo, x;
  const float* a_hi_ptr = nullptr;
  const float* a_lo_ptr = nullptr;
  const float* x_ptr = nullptr;
  int x_ncol = -1;
  float* xbuf = nullptr;
  size_t xbuf_bytes = 0;
  int* d_err = nullptr;
  int* h_err = nullptr;              // pinned copy of d_err (tc_error_enqueue / tc_error_status)
  bool smem_set = false;
  int num_sms = 0;
  // CTA-pair kernel: X map with half-width boxes, co-resident clusters (0 = unused)
  CUtensorMap xh;
  int xh_ncol = -1;
  const float* xh_ptr = nullptr;
  int pair_clusters = -1;
  // fused gather + GEMM (k_tc_fused<GT>): maps of the FP16 Lambda halves, co-resident clusters
  // (-1: not yet asked)
  CUtensorMap h_hi, h_lo;
  const void* h_hi_ptr = nullptr;
  const void* h_lo_ptr = nullptr;
  int fused_clusters = -1;
};

// Round to TF32 (10 explicit mantissa bits), to nearest with ties away from zero,
// by integer arithmetic on the bit pattern: adding half of the 13 dropped bits
// then clearing them rounds the magnitude (sign-magnitude encoding).  Two
// full-rate integer instructions instead of a conversion instruction.
__device__ __forceinline__ float to_tf32(float v) {
  return __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xFFFFE000u);
}

__device__ __forceinline__ unsigned long long nonneg_bits(float v) {
  double d = (v == v) ? (double)v : __longlong_as_double(0x7ff0000000000000ULL);
  return (unsigned long long)__double_as_longlong(d);
}

// ---------------------------------------------------------------------------
// gather: X[i][n][k] = sum_j J_ij(k mod Nc) d_j[n][k]
// grid: one CTA per (block of 16 vector columns, site), column block outermost
// ---------------------------------------------------------------------------
constexpr int GATHER_COLS = 16;

// act (optional, [Nr][column tiles of BN]): the first sweep at which the tile can
// be non-zero; blocks of later tiles are skipped (support truncation)
__global__ __launch_bounds__(256) void k_tc_gather(const float* __restrict__ din, const float* __restrict__ Jz,
                                                       const int* __restrict__ nbr, const int* __restrict__ nbond,
                                                       float* __restrict__ X, int Nr, int Nc, int ncol,
                                                       const int* __restrict__ act, int sweep) {
  const int i = blockIdx.x % Nr;
  const int nblk = blockIdx.x / Nr;
  if (act && act[i * ((ncol + BN - 1) / BN) + (nblk * GATHER_COLS) / BN] > sweep) return;
  const int N2 = 2 * Nc;
  int nb[4], bd[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    nb[s] = nbr[i * 4 + s];
    bd[s] = nbond[i * 4 + s];
  }
  const int per_col4 = N2 / 4;
  const int total4 = GATHER_COLS * per_col4;
  for (int e = threadIdx.x; e < total4; e += blockDim.x) {
    int c = e / per_col4, k = (e - c * per_col4) * 4;
    int n = nblk * GATHER_COLS + c;
    if (n >= ncol) break;
    int kz = k < Nc ? k : k - Nc;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (nb[s] < 0) continue;
      float4 j = *reinterpret_cast<const float4*>(Jz + (size_t)bd[s] * Nc + kz);
      float4 g = *reinterpret_cast<const float4*>(din + ((size_t)nb[s] * ncol + n) * N2 + k);
      acc.x = fmaf(j.x, g.x, acc.x);
      acc.y = fmaf(j.y, g.y, acc.y);
      acc.z = fmaf(j.z, g.z, acc.z);
      acc.w = fmaf(j.w, g.w, acc.w);
    }
    *reinterpret_cast<float4*>(X + ((size_t)i * ncol + n) * N2 + k) = acc;
  }
}

// (a, b) = hi + lo in FP16, packed with a in the low halves; the difference a - hi is exact in FP32
__device__ __forceinline__ void split_f16(float a, float b, unsigned int& hi, unsigned int& lo) {
  const __half2 h = __floats2half2_rn(a, b);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
  hi = *reinterpret_cast<const unsigned int*>(&h);
  lo = *reinterpret_cast<const unsigned int*>(&l);
}

// split an fp32 tile (float4 granules e = tt, tt + 128, ...) into TF32 hi in place and lo at x + bytes
template <int BYTES>
__device__ __forceinline__ void split_tile(uint8_t* x, int tt) {
  float4* xh = reinterpret_cast<float4*>(x);
  float4* xl = reinterpret_cast<float4*>(x + BYTES);
#pragma unroll 4
  for (int e = tt; e < BYTES / 16; e += 128) {
    float4 v = xh[e], h, l;
    h.x = to_tf32(v.x); l.x = to_tf32(v.x - h.x);
    h.y = to_tf32(v.y); l.y = to_tf32(v.y - h.y);
    h.z = to_tf32(v.z); l.z = to_tf32(v.z - h.z);
    h.w = to_tf32(v.w); l.w = to_tf32(v.w - h.w);
    xh[e] = h;
    xl[e] = l;
  }
}

__device__ __forceinline__ void fold_ymax(TcScale* s, float y, int lane) {
  unsigned int u = __float_as_uint(y);                    // y >= 0 (fmaxf drops NaN: the norm reports it)
  u = __reduce_max_sync(0xffffffffu, u);
  if (lane == 0) atomicMax(&s->ymax, u);
}

// scale of the next sweep from the maxima that the last one (or a seed) left
__global__ void k_tc_scale(TcScale* __restrict__ sc, int ng, float jbound) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < ng) set_scale(sc + q, __uint_as_float(sc[q].ymax), jbound);
}
// seeds of the maxima: a bound common to all groups, or a bound per group
__global__ void k_tc_seed(TcScale* __restrict__ sc, int ng, const double* __restrict__ ref, float bound) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  // (1 + 1e-6: an FP32 state may exceed an FP64 bound by its rounding)
  if (q < ng) sc[q].ymax = __float_as_uint(ref ? (float)(ref[q] * 1.000001) : bound);
}
// seed by reading the state: one warp per (site, vector column)
__global__ void __launch_bounds__(256) k_tc_seed_scan(const float* __restrict__ d, int Nr, int Nc, int ncol, int gs,
                                                      TcScale* __restrict__ sc) {
  const size_t w = (size_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (w >= (size_t)Nr * ncol) return;
  const int n = (int)(w % ncol);
  const float4* p = reinterpret_cast<const float4*>(d + w * 2 * Nc);
  float m = 0.f;
  for (int k = lane; k < Nc / 2; k += 32) {
    const float4 v = p[k];
    m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
  }
  const unsigned int u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if (lane == 0 && u > sc[n / gs].ymax) atomicMax(&sc[n / gs].ymax, u);
}

// epilogue of one warp's 32 accumulator lanes x BN columns (TMEM address tacc):
// y = r + acc at planar row mg, columns n_first.., store y, and fold max|y - d_in|
// into norm[] per group of gs columns (gs a multiple of 32)
__device__ __forceinline__ void epilogue_rows(uint32_t tacc, int mg, int n_first, int site, int ncol, int gs,
                                              size_t N2, const float* __restrict__ r, const float* __restrict__ din,
                                              float* __restrict__ dout, unsigned long long* __restrict__ norm,
                                              int lane) {
  using namespace ptx;
  constexpr int CH = 32;                            // columns per tcgen05.ld
  int qcur = n_first / gs;
  float runmax = 0.f;
  for (int c = 0; c < BN / CH; ++c) {
    const int n0 = n_first + c * CH;
    if (n0 >= ncol) break;                          // uniform across the warp
    const int q = n0 / gs;
    if (q != qcur) {
      float m = runmax;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) atomicMax(norm + qcur, nonneg_bits(m));
      qcur = q;
      runmax = 0.f;
    }
    float rv[CH], dv[CH];
    uint32_t v[CH];
    const size_t base = ((size_t)site * ncol + n0) * N2 + mg;
#pragma unroll
    for (int j = 0; j < CH; ++j) {
      rv[j] = __ldcs(r + base + (size_t)j * N2);
      dv[j] = __ldcs(din + base + (size_t)j * N2);
    }
    tmem_ld32(tacc + (uint32_t)(c * CH), v);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < CH; ++j) {
      const float y = rv[j] + __uint_as_float(v[j]);
      float d = fabsf(y - dv[j]);
      d = (d == d) ? d : __int_as_float(0x7f800000);
      __stcs(dout + base + (size_t)j * N2, y);
      runmax = fmaxf(runmax, d);
    }
  }
  float m = runmax;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) atomicMax(norm + qcur, nonneg_bits(m));
}

// ---------------------------------------------------------------------------
// persistent GEMM + epilogue of the single-CTA form
// ---------------------------------------------------------------------------
// One 128 x 256 output tile, as every warp role decodes it.
struct TileRef {
  int mt, nt, site;
  bool active;
};

// act/sweep: support truncation (tiles whose act entry exceeds the sweep hold zeros and are
// skipped), act == nullptr: none
__device__ __forceinline__ TileRef decode_tile(int tile, int MT, int NT, const int* __restrict__ act, int sweep) {
  TileRef T;
  T.mt = tile % MT;
  T.nt = (tile / MT) % NT;
  T.site = tile / (MT * NT);
  T.active = !(act && act[T.site * NT + T.nt] > sweep);
  return T;
}

__global__ void __launch_bounds__(THREADS, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap map_ahi, const __grid_constant__ CUtensorMap map_alo,
              const __grid_constant__ CUtensorMap map_x, const float* __restrict__ r, const float* __restrict__ din,
              float* __restrict__ dout, int Nr, int Nc, int ncol, int gs, unsigned long long* __restrict__ norm,
              int* __restrict__ err, const int* __restrict__ act, int sweep) {
  using namespace ptx;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_tma[STAGES], full_split[STAGES], empty[STAGES];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], drain;
  __shared__ uint32_t tmem_holder;
  __shared__ WaitCtl wctl;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KB = (2 * Nc) / BK, MT = (2 * Nc) / BM, NT = (ncol + BN - 1) / BN;
  const int tiles = MT * NT * Nr;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_tma[s], 1);
      mbar_init(&full_split[s], 128);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 128);
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
  volatile WaitCtl* abort_p = &wctl;
  auto stage_ptr = [&](int s) { return smem + (size_t)s * STAGE_BYTES; };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      int g = 0;                                        // k-blocks issued by this CTA
      bool ok = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const TileRef T = decode_tile(tile, MT, NT, act, sweep);
        if (!T.active) continue;
        // the next active tile of this CTA, for the L2 prefetch that runs ahead of the loads
        int t2 = tile + (int)gridDim.x;
        TileRef N;
        N.active = false;
        for (; t2 < tiles; t2 += gridDim.x) {
          N = decode_tile(t2, MT, NT, act, sweep);
          if (N.active) break;
        }
        for (int kb = 0; kb < KB; ++kb, ++g) {
          const int s = g % STAGES;
          if (g >= STAGES && !mbar_wait(&empty[s], ((g / STAGES) - 1) & 1, abort_p)) {
            ok = false;
            break;
          }
          uint8_t* st = stage_ptr(s);
          mbar_expect_tx(&full_tma[s], TMA_BYTES);
          tma_load_3d(st, &map_ahi, &full_tma[s], kb * BK, T.mt * BM, T.site);
          tma_load_3d(st + A_TILE, &map_alo, &full_tma[s], kb * BK, T.mt * BM, T.site);
          tma_load_3d(st + 2 * A_TILE, &map_x, &full_tma[s], kb * BK, T.nt * BN, T.site);
          // warm L2 with the tiles of the k-block PREFETCH steps ahead: the stage
          // loads then see L2 latency instead of DRAM latency
          const int ahead = kb + PREFETCH;
          if (ahead < KB) {
            tma_prefetch_3d(&map_ahi, ahead * BK, T.mt * BM, T.site);
            tma_prefetch_3d(&map_alo, ahead * BK, T.mt * BM, T.site);
            tma_prefetch_3d(&map_x, ahead * BK, T.nt * BN, T.site);
          } else if (N.active && ahead - KB < KB) {
            const int k2 = ahead - KB;
            tma_prefetch_3d(&map_ahi, k2 * BK, N.mt * BM, N.site);
            tma_prefetch_3d(&map_alo, k2 * BK, N.mt * BM, N.site);
            tma_prefetch_3d(&map_x, k2 * BK, N.nt * BN, N.site);
          }
        }
      }
      // let every copy this thread issued land before the CTA can exit
      for (int q = g > STAGES ? g - STAGES : 0; q < g; ++q)
        mbar_wait(&full_tma[q % STAGES], (q / STAGES) & 1, abort_p, false);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      int g = 0, t = 0;
      bool ok = true, any = false;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const TileRef T = decode_tile(tile, MT, NT, act, sweep);
        if (!T.active) continue;
        const int buf = t & 1;
        if (t >= 2 && !mbar_wait(&acc_empty[buf], ((t >> 1) - 1) & 1, abort_p)) break;
        ++t;
        tc_fence_after();
        const uint32_t dacc = tmem + (uint32_t)(buf * ACC_COLS);
        for (int kb = 0; kb < KB; ++kb, ++g) {
          const int s = g % STAGES;
          if (!mbar_wait(&full_split[s], (g / STAGES) & 1, abort_p)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_hi = smem_u32(stage_ptr(s));
          const uint32_t a_lo = a_hi + A_TILE;
          const uint32_t x_hi = a_hi + 2 * A_TILE;
          const uint32_t x_lo = x_hi + X_TILE;
#pragma unroll
          for (int k8 = 0; k8 < BK / 8; ++k8) {
            const uint32_t off = k8 * 32;   // 8 TF32 values inside the 128-byte swizzle row
            const uint64_t dah = sdesc_sw128(a_hi + off), dal = sdesc_sw128(a_lo + off);
            const uint64_t dxh = sdesc_sw128(x_hi + off), dxl = sdesc_sw128(x_lo + off);
            mma<1>(dacc, dah, dxh, IDESC, (kb | k8) ? 1u : 0u);
            mma<1>(dacc, dah, dxl, IDESC, 1u);
            mma<1>(dacc, dal, dxh, IDESC, 1u);
          }
          mma_commit(&empty[s]);
          any = true;
        }
        if (ok) mma_commit(&acc_full[buf]);
      }
      if (any) {
        mma_commit(&drain);                               // all MMAs of this thread completed
        mbar_wait(&drain, 0, abort_p, false);
      }
    }
  } else if (warp >= 4 && warp < 8) {
    // ---------------- split X into TF32 hi / lo ----------------
    const int tt = threadIdx.x - 128;
    int g = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      const TileRef T = decode_tile(tile, MT, NT, act, sweep);
      if (!T.active) continue;
      for (int kb = 0; kb < KB; ++kb, ++g) {
        const int s = g % STAGES;
        if (!mbar_wait(&full_tma[s], (g / STAGES) & 1, abort_p)) {
          ok = false;
          break;
        }
        split_tile<X_TILE>(stage_ptr(s) + 2 * A_TILE, tt);
        fence_async_smem();
        mbar_arrive(&full_split[s]);
      }
    }
  } else if (warp >= 8) {
    // ---------------- epilogue ----------------
    const int q4 = warp - 8;                            // TMEM lane quarter (warp % 4)
    int t = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      const TileRef T = decode_tile(tile, MT, NT, act, sweep);
      if (!T.active) continue;
      const int buf = t & 1;
      bool go = mbar_wait(&acc_full[buf], (t >> 1) & 1, abort_p);
      ++t;
      go = __all_sync(0xffffffffu, go);                 // tcgen05.ld below is warp-collective
      if (!go) break;
      tc_fence_after();
      epilogue_rows(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(buf * ACC_COLS), T.mt * BM + q4 * 32 + lane,
                    T.nt * BN, T.site, ncol, gs, 2 * (size_t)Nc, r, din, dout, norm, lane);
      // this accumulator may be overwritten by the MMAs of tile t + 2
      tc_fence_before();
      mbar_arrive(&acc_empty[buf]);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
  if (threadIdx.x == 0 && wctl.abort) atomicExch(err, 1);
}

// ---------------------------------------------------------------------------
// CTA-pair form (cluster of 2, tcgen05 cta_group::2): the pair computes a
// 256 x 256 tile with M = 256 MMAs.  CTA r of the pair loads Lambda rows
// 128 r .. 128 r + 127 of the tile and X columns 128 r .. 128 r + 127, splits only
// its half of X, and holds rows 128 r .. of the accumulator in its own TMEM.
// The even CTA's MMA thread reads both CTAs' shared memory, so per SM the TMA,
// split and MMA operand traffic through shared memory drop by a third, and
// three 64 KB stages fit.  Pipeline:
//   TMA (each CTA, own barrier) -> split (each CTA) -> arrive on the even CTA's
//   full_split -> MMAs -> commit multicast to both CTAs' empty / acc_full ->
//   epilogue (each CTA) -> arrive on the even CTA's acc_empty.
// ---------------------------------------------------------------------------
constexpr int PM = 256;                                 // tile rows per pair
constexpr int PX_TILE = (BN / 2) * BK * 4;              // 16 KB: one CTA's half of the X tile
constexpr int P_STAGES = 3;
constexpr int P_STAGE_BYTES = 2 * A_TILE + 2 * PX_TILE;  // A_hi, A_lo, X (-> X_hi), X_lo
constexpr int P_TMA_BYTES = 2 * A_TILE + PX_TILE;
constexpr int P_SMEM_BYTES = P_STAGES * P_STAGE_BYTES + 1024;
constexpr uint32_t P_IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(BN >> 3) << 17) |
                             ((uint32_t)(PM >> 4) << 24);

__global__ void __launch_bounds__(THREADS, 1)
    k_tc_gemm_pair(const __grid_constant__ CUtensorMap map_ahi, const __grid_constant__ CUtensorMap map_alo,
                   const __grid_constant__ CUtensorMap map_xh, const float* __restrict__ r,
                   const float* __restrict__ din, float* __restrict__ dout, int Nr, int Nc, int ncol, int gs,
                   unsigned long long* __restrict__ norm, int* __restrict__ err) {
  using namespace ptx;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_tma[P_STAGES], full_split[P_STAGES], empty[P_STAGES];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], drain;
  __shared__ uint32_t tmem_holder;
  __shared__ WaitCtl wctl;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int KB = (2 * Nc) / BK;
  const int MT = (2 * Nc) / PM, NT = (ncol + BN - 1) / BN;
  const int tiles = MT * NT * Nr;

  if (threadIdx.x == 0) {
    for (int s = 0; s < P_STAGES; ++s) {
      mbar_init(&full_tma[s], 1);
      mbar_init(&full_split[s], 256);                   // 128 split threads of each CTA (even CTA's copy is used)
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 256);                    // 128 epilogue threads of each CTA
    }
    mbar_init(&drain, 1);
    wait_ctl_init(&wctl);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(&tmem_holder, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_sync();                                       // the peer's barriers exist before any remote arrive
  tc_fence_after();
  const uint32_t tmem = tmem_holder;
  volatile WaitCtl* abort_p = &wctl;
  auto stage_ptr = [&](int s) { return smem + (size_t)s * P_STAGE_BYTES; };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer (both CTAs) ----------------
      int g = 0;
      bool ok = true;
      for (int tile = pair; tile < tiles && ok; tile += npairs) {
        const int mt = tile % MT, nt = (tile / MT) % NT, site = tile / (MT * NT);
        const int row0 = mt * PM + (int)rank * BM;
        // a half tile wholly past the last column loads columns 0.. instead (its
        // products land in accumulator columns the epilogue never reads), so no
        // box lies entirely outside the tensor
        int col0 = nt * BN + (int)rank * (BN / 2);
        col0 = col0 < ncol ? col0 : 0;
        for (int kb = 0; kb < KB; ++kb, ++g) {
          const int s = g % P_STAGES;
          if (g >= P_STAGES && !mbar_wait(&empty[s], ((g / P_STAGES) - 1) & 1, abort_p)) {
            ok = false;
            break;
          }
          uint8_t* st = stage_ptr(s);
          mbar_expect_tx(&full_tma[s], P_TMA_BYTES);
          tma_load_3d(st, &map_ahi, &full_tma[s], kb * BK, row0, site);
          tma_load_3d(st + A_TILE, &map_alo, &full_tma[s], kb * BK, row0, site);
          tma_load_3d(st + 2 * A_TILE, &map_xh, &full_tma[s], kb * BK, col0, site);
          {
            const int ahead = kb + PREFETCH;
            const int t2 = ahead < KB ? tile : tile + npairs;
            if (t2 < tiles && (ahead < KB || ahead - KB < KB)) {
              const int k2 = ahead < KB ? ahead : ahead - KB;
              const int m2 = t2 % MT, n2 = (t2 / MT) % NT, s2 = t2 / (MT * NT);
              tma_prefetch_3d(&map_ahi, k2 * BK, m2 * PM + (int)rank * BM, s2);
              tma_prefetch_3d(&map_alo, k2 * BK, m2 * PM + (int)rank * BM, s2);
              const int c2 = n2 * BN + (int)rank * (BN / 2);
              tma_prefetch_3d(&map_xh, k2 * BK, c2 < ncol ? c2 : 0, s2);
            }
          }
        }
      }
      for (int q = g > P_STAGES ? g - P_STAGES : 0; q < g; ++q)
        mbar_wait(&full_tma[q % P_STAGES], (q / P_STAGES) & 1, abort_p, false);
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // ---------------- MMA issuer (even CTA only) ----------------
      int g = 0, t = 0;
      bool ok = true, any = false;
      for (int tile = pair; tile < tiles && ok; tile += npairs, ++t) {
        const int buf = t & 1;
        if (t >= 2 && !mbar_wait_cluster(&acc_empty[buf], ((t >> 1) - 1) & 1, abort_p)) break;
        tc_fence_after();
        const uint32_t dacc = tmem + (uint32_t)(buf * ACC_COLS);
        for (int kb = 0; kb < KB; ++kb, ++g) {
          const int s = g % P_STAGES;
          if (!mbar_wait_cluster(&full_split[s], (g / P_STAGES) & 1, abort_p)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_hi = smem_u32(stage_ptr(s));
          const uint32_t a_lo = a_hi + A_TILE;
          const uint32_t x_hi = a_hi + 2 * A_TILE;
          const uint32_t x_lo = x_hi + PX_TILE;
#pragma unroll
          for (int k8 = 0; k8 < BK / 8; ++k8) {
            const uint32_t off = k8 * 32;
            const uint64_t dah = sdesc_sw128(a_hi + off), dal = sdesc_sw128(a_lo + off);
            const uint64_t dxh = sdesc_sw128(x_hi + off), dxl = sdesc_sw128(x_lo + off);
            mma_pair_tf32(dacc, dah, dxh, P_IDESC, (kb | k8) ? 1u : 0u);
            mma_pair_tf32(dacc, dah, dxl, P_IDESC, 1u);
            mma_pair_tf32(dacc, dal, dxh, P_IDESC, 1u);
          }
          mma_commit_pair_mc(&empty[s], 0x3);
          any = true;
        }
        if (ok) mma_commit_pair_mc(&acc_full[buf], 0x3);
      }
      if (any) {
        mma_commit_pair_mc(&drain, 0x1);
        mbar_wait(&drain, 0, abort_p, false);
      }
    }
  } else if (warp >= 4 && warp < 8) {
    // ---------------- split own half of X (both CTAs) ----------------
    const int tt = threadIdx.x - 128;
    const uint32_t split_bar0 = mapa(smem_u32(&full_split[0]), 0);
    int g = 0;
    bool ok = true;
    for (int tile = pair; tile < tiles && ok; tile += npairs) {
      for (int kb = 0; kb < KB; ++kb, ++g) {
        const int s = g % P_STAGES;
        if (!mbar_wait(&full_tma[s], (g / P_STAGES) & 1, abort_p)) {
          ok = false;
          break;
        }
        split_tile<PX_TILE>(stage_ptr(s) + 2 * A_TILE, tt);
        fence_async_smem();
        mbar_arrive_remote(split_bar0 + (uint32_t)(s * sizeof(uint64_t)));
      }
    }
  } else if (warp >= 8) {
    // ---------------- epilogue (both CTAs, own 128 rows) ----------------
    const int q4 = warp - 8;
    const size_t N2 = 2 * (size_t)Nc;
    const uint32_t empty_bar0 = mapa(smem_u32(&acc_empty[0]), 0);
    int t = 0;
    for (int tile = pair; tile < tiles; tile += npairs, ++t) {
      const int mt = tile % MT, nt = (tile / MT) % NT, site = tile / (MT * NT);
      const int buf = t & 1;
      bool go = mbar_wait(&acc_full[buf], (t >> 1) & 1, abort_p);
      go = __all_sync(0xffffffffu, go);
      if (!go) break;
      tc_fence_after();
      epilogue_rows(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(buf * ACC_COLS),
                    mt * PM + (int)rank * BM + q4 * 32 + lane, nt * BN, site, ncol, gs, N2, r, din, dout, norm, lane);
      tc_fence_before();
      mbar_arrive_remote(empty_bar0 + (uint32_t)(buf * sizeof(uint64_t)));
    }
  }

  // both CTAs stay resident until the even CTA's MMAs (which read the odd CTA's
  // shared memory and write its TMEM) have drained and every remote arrive landed
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
  if (threadIdx.x == 0 && wctl.abort) atomicExch(err, 1);
}

// ---------------------------------------------------------------------------
// Fused sweep on CTA pairs: the neighbour gather is the producer of the MMA's
// B operand.  Eight warps per CTA read the four neighbour rows of d_in
// (coalesced float4 loads, sixteen issued back to back and half a k-block
// ahead of their sums), scale them by J(k), sum, split the sum into FP16
// hi + lo and write both straight into the 128-byte-swizzled stage, so X never
// exists in global memory and only Lambda hi/lo travel by TMA.  The epilogue
// forms d_out = r + K d_in and the update norm max|d_out - d_in| as the unfused
// sweeps do (GMRES matvecs use it with r = 0).
// Operands: FP16 has the 11 significant bits of TF32 at half the bytes and twice the MMA
// rate; its range is made up by powers of two, one per row of Lambda W (2^14 <= max < 2^15)
// and one per column group of X (set_scale), taken out again in the epilogue.  hi + lo keeps
// 22 bits of every entry down to 2^-16 of the row's (group's) largest and 2^-39 of the
// largest below that, under the FP32 accumulation's own rounding.
// The kernel is bound by the latency of the loads through L2 at what an SM keeps in flight (10.4 TB/s of
// L2 traffic; tensor pipe 29 %, L2 33 %, DRAM 50 % busy), so the two forms differ in what they read.  Both have two
// accumulator sets of 256 TMEM columns, so that a tile's epilogue overlaps the next tile's MMAs:
//   <2>  a tile is (site, 128 vector columns, 256 contour points z): its two accumulators are the
//        real and the imaginary rows of those points.  A k-block is 64 complex points; the tiles
//        Re and Im of Lambda are loaded once and serve both halves of the embedding
//        [[Re, -Im], [Im, Re]] (the minus sign is the MMA's negate bit), and X is gathered once
//        per ceil(Ns / 256) tiles.  Two stages of 96 KB.  Ns >= 192.
//   <1>  a tile is (site, 256 vector columns, 256 rows of the embedding); a k-block is 64 real
//        values, three stages of 64 KB.  Ns = 64 and 128, where <2> would fill half of its rows at most.
// Bytes from L2 per sweep at 16x16, Nc = 256, 4096 columns, by count: X 8.6 GB, Lambda 4.3, epilogue 4.3
// and 2.1 written (<1>: X 17.2, Lambda 4.3; with the embedding in 512-row tiles: X 8.6, Lambda 8.6); the counters
// say 25 GB in all.  Measured there, in the mean over a solve's launches, truncated ones among them:
// 2.05 ms (2.15 per sweep that does work, with its check); 2.67 ms as <1> and 2.37 with the embedding in
// 512-row tiles; 2.66 ms in 3xTF32 with the traffic of <1>.  Each gather step waits for one loaded
// memory latency (about 2.3 us, 64 KB in flight per SM); fetching the next tile's neighbour rows
// into L2 ahead adds requests and cost 25 %.
// FP64 residual of one inner solve, 57 drawn problems on contours of 64 to 256 points: 0.39 to 1.21 of the 3xTF32
// form's, 0.63 in the mean (fewer roundings: twice the products per MMA).  With the lo halves scaled by 2^11, 22 bits
// down to 2^-29, it is the same: the range is no limit.
// SPLIT: contours that are no multiple of 64, whose other form is the FP32 CUDA-core sweep (every product and
// sum rounded to nearest).  The tensor memory accumulation truncates once per MMA, and with all three products in
// one accumulator the residual of an inner solve was 1.1 to 2.8 times that sweep's (Nc 33 to 151; 0.4 to 1.2 from
// 160 on).  So the small products get an accumulator of their own, and in <1> the large ones two that they take in
// turn: 0.26 to 1.02 times, 0.6 in the mean of 92 problems, Nc 26 to 250.  That fills the tensor memory with one set of
// accumulators and <1> takes 128 columns a tile (four stages of 48 KB).  A solve at 1e-10, one accumulator and
// SPLIT: 9x7, Nc = 100, 6 block columns 4.4 and 4.2 ms; 10x9, Nc = 105, 8 columns 7.1 and 6.8; 7x7, Nc = 151, 3
// columns 6.0 and 7.3; 9x8, Nc = 223, 6 columns 32.4 and 29.5 (with fewer sweeps); the CUDA-core sweep 21, 39, 27, 305.
// (13x15, Nc = 180, one column, 1e-6: 14.0 and 18.8; the CUDA-core sweep 70.)
// Sites are visited in bands of two lattice rows, column by column, so that
// a site's neighbours are read while they are still in L2.
// Warp roles (512 threads per CTA, both CTAs of the pair):
//   warp 0        TMA of this CTA's 128 rows of Lambda hi/lo per group (+ L2 prefetch)
//   warp 1        (even CTA) one thread issues the cta_group::2 MMAs
//   warp 2        one thread waits until this CTA's Lambda tiles of a stage have landed
//                 and its producer warps have written X, then arrives once on the even
//                 CTA's stage barrier (the only cluster-scope release per CTA and stage;
//                 producers arrive on a CTA-local barrier and never wait for TMA)
//   warps 4-11    gather producers: X columns 128 r .. 128 r + 127 of the tile
//   warps 12-15   epilogue: tcgen05.ld, + r, store, update norm
// Every wait is bounded like those of the other tcgen05 kernels.
// ---------------------------------------------------------------------------
constexpr int F_THREADS = 512;
constexpr int F_PROD_W0 = 4, F_PROD_WARPS = 8;
constexpr int F_EPI_W0 = 12;
constexpr int F_BK = 64;                                // k-block: 64 FP16 = one 128-byte swizzle row
static_assert(A_TILE == BM * F_BK * 2 && PX_TILE == (BN / 2) * F_BK * 2, "FP16 tiles of 64 fill the TF32 tiles of 32");
constexpr int F_A_GROUP = 2 * A_TILE;                   // Lambda hi + lo, this CTA's 128 rows of one accumulator
constexpr uint32_t F_NEGATE_A = 1u << 13;               // instruction descriptor: D += (-A) B
constexpr int F_SITE_BAND = 2;                          // lattice rows per band of the site order
constexpr int F_RELAY_W = 2;                            // warp 2: relays "Lambda landed" to the even CTA
// registers per thread of each warpgroup once the roles split: the producers keep sixteen
// neighbour loads in flight one k-block ahead, more than the 128 a thread of a 512-thread
// block gets at launch; the TMA / MMA / relay warpgroup needs few
constexpr int F_REG_CTRL = 56, F_REG_PROD = 168, F_REG_EPI = 120;
constexpr int F_REGS_AT_LAUNCH = 65536 / F_THREADS;
static_assert(F_REG_CTRL + 2 * F_REG_PROD + F_REG_EPI <= 4 * F_REGS_AT_LAUNCH,
              "the warpgroups' register shares exceed the block's registers at launch");
static_assert(F_PROD_W0 == 4 && F_PROD_WARPS == 8 && F_EPI_W0 == 12 && F_THREADS == 512,
              "the register split assumes warpgroups {0-3: control, 4-11: producers, 12-15: epilogue}");
template <int GT_, bool SPLIT>
struct FusedCfg {
  static constexpr int GT = GT_;
  static constexpr int NB = GT == 1 && !SPLIT ? 256 : 128;   // vector columns of a tile
  static constexpr int STEPS = GT * NB / 128;           // gather steps of a k-block
  static constexpr int X_TILE = (NB / 2) * F_BK * 2;    // one CTA's half of X hi (or lo)
  // GT = 2: Re hi, Re lo, Im hi, Im lo | Xr hi, Xr lo, Xi hi, Xi lo;  GT = 1: hi, lo | X hi, X lo
  static constexpr int STAGE = GT * F_A_GROUP + GT * 2 * X_TILE;
  static constexpr int STAGES = GT == 2 ? 2 : SPLIT ? 4 : 3;
  static constexpr int SMEM = STAGES * STAGE + 1024;
  // accumulators of one output (the first LARGE take hi x hi in turn, the last the small products) and
  // sets of them
  static constexpr int ACCS = !SPLIT ? 1 : GT == 1 ? 3 : 2, LARGE = ACCS == 3 ? 2 : 1;
  static constexpr int NBUF = SPLIT ? 1 : 2;
  static constexpr uint32_t ACC_STRIDE = GT * NB;       // TMEM columns from one accumulator to the next
  // kind::f16, D = F32, A = B = F16, K-major, M = 256, N = NB
  static constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(PM >> 4) << 24);
  static_assert(NBUF * ACCS * GT * NB <= 512, "TMEM holds 512 columns");
  static_assert(SMEM <= 227 * 1024, "shared memory of one CTA");
  static_assert(TC_TILE_COLS % NB == 0, "a tile lies in one column tile of the support table");
};

// site of visit index v: bands of F_SITE_BAND lattice rows, walked column by column
__device__ __forceinline__ int band_site(int v, int Lx, int Ly) {
  const int band = v / (F_SITE_BAND * Lx);
  const int y0 = band * F_SITE_BAND;
  const int h = min(F_SITE_BAND, Ly - y0);
  const int w = v - band * F_SITE_BAND * Lx;
  return (y0 + w % h) * Lx + w / h;
}

// A tile as every warp role decodes it.
struct FTile {
  int site, nt, gt;
  bool active;
};

// 256-row tiles of one accumulator
template <int GT>
__host__ __device__ __forceinline__ int fused_row_tiles(int Ns) {
  return ((GT == 2 ? Ns : 2 * Ns) + PM - 1) / PM;
}

// (act has one entry per site and TC_TILE_COLS columns)
template <class Cfg>
__device__ __forceinline__ FTile fused_tile(const FusedInst& I, int tile, int sweep) {
  constexpr int NB = Cfg::NB;
  FTile T;
  const int NGT = fused_row_tiles<Cfg::GT>(I.Ns), NT = (I.ncol + NB - 1) / NB;
  T.gt = tile % NGT;
  T.nt = (tile / NGT) % NT;
  T.site = band_site(tile / (NGT * NT), I.Lx, I.Ly);
  T.active = true;
  if (I.act) {
    const int nact = (I.ncol + TC_TILE_COLS - 1) / TC_TILE_COLS;
    T.active = I.act[T.site * nact + T.nt / (TC_TILE_COLS / NB)] <= sweep;
  }
  return T;
}

// Epilogue of one warp's 32 accumulator lanes: GT accumulators x NB columns in chunks of 16 columns.  The
// accumulators hold 2^(a + x) times the product, the row's and the column group's powers of two:
// y = r + acc adown sc[q].down; y is stored, max|y - d_in| folded into norm[] and max|y| into
// sc[].ymax (for the next sweep's scale) per group of gs columns.  The loads of r and d_in run one
// chunk ahead, the first ones before the accumulators are complete.  (Three chunks of 8 columns ahead,
// or a ring of four 8-column slots in shared memory filled by bulk copies, took 2.5-2.7 ms per sweep
// where this takes 2.1: 16x16, Nc = 256, 4096 columns.)  RZERO: r is zero on this tile.
template <class Cfg, bool RZERO>
struct FusedEpilogue {
  static constexpr int NB = Cfg::NB, CH = 16, PER = NB / CH, CHUNKS = Cfg::GT * PER;
  const float* __restrict__ r;
  const float* din;
  float* __restrict__ dout;
  int n_first, ncol, N2, row_gap;
  size_t base0;                                          // element of (site, column n_first, this lane's first row)
  float rv[2][CH], dv[2][CH];

  __device__ __forceinline__ size_t at(int e) const {
    return base0 + (size_t)(e % PER) * CH * N2 + (size_t)(e / PER) * row_gap;
  }
  template <int B>
  __device__ __forceinline__ void load(int e) {
    const int left = ncol - n_first - (e % PER) * CH;    // warp-uniform
    if (left <= 0) return;
    const size_t o = at(e);
    if (left >= CH) {
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        if (!RZERO) rv[B][j] = __ldcs(r + o + (size_t)j * N2);
        dv[B][j] = ptx::load_cs(din + o + (size_t)j * N2);
      }
    } else {
#pragma unroll
      for (int j = 0; j < CH; ++j)
        if (j < left) {
          if (!RZERO) rv[B][j] = __ldcs(r + o + (size_t)j * N2);
          dv[B][j] = ptx::load_cs(din + o + (size_t)j * N2);
        }
    }
  }
  float runmax = 0.f, ymax = 0.f, down = 0.f;
  int qcur = -1, qbeg = 0, qend = 0;                     // current norm group and its columns
  __device__ __forceinline__ void flush(unsigned long long* norm, TcScale* sc, int lane) {
    const unsigned int m = __reduce_max_sync(0xffffffffu, __float_as_uint(runmax));
    if (lane == 0) atomicMax(norm + qcur, nonneg_bits(__uint_as_float(m)));
    fold_ymax(sc + qcur, ymax, lane);
    runmax = ymax = 0.f;
  }
  template <int B>
  __device__ __forceinline__ void chunk(int e, uint32_t tacc, float adown, int gs, unsigned long long* norm,
                                        TcScale* sc, int lane) {
    const int n0 = n_first + (e % PER) * CH;
    if (n0 >= ncol) return;
    auto enter = [&](int n) {                            // warp-uniform
      if (n >= qbeg && n < qend) return;
      if (qcur >= 0) flush(norm, sc, lane);
      qcur = n / gs;
      qbeg = qcur * gs;
      qend = qbeg + gs;
      down = adown * ptx::load_f(&sc[qcur].down);
    };
    enter(n0);
    uint32_t v[CH];
    ptx::tmem_ld16(tacc + (uint32_t)(e * CH), v);
    ptx::tmem_wait_ld();
#pragma unroll
    for (int a = 1; a < Cfg::ACCS; ++a) {
      uint32_t w[CH];
      ptx::tmem_ld16(tacc + a * Cfg::ACC_STRIDE + (uint32_t)(e * CH), w);
      ptx::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < CH; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(w[j]));
    }
    const size_t o = at(e);
    auto column = [&](int j) {
      const float y = RZERO ? __uint_as_float(v[j]) * down : fmaf(__uint_as_float(v[j]), down, rv[B][j]);
      float d = fabsf(y - dv[B][j]);
      d = (d == d) ? d : __int_as_float(0x7f800000);
      __stcs(dout + o + (size_t)j * N2, y);
      runmax = fmaxf(runmax, d);
      ymax = fmaxf(ymax, fabsf(y));
    };
    if (n0 + CH <= ncol && n0 + CH <= qend) {
#pragma unroll
      for (int j = 0; j < CH; ++j) column(j);
    } else {                                             // the last columns, or a group ends inside the chunk
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        if (n0 + j >= ncol) break;
        enter(n0 + j);
        column(j);
      }
    }
  }
};

// r = 0 (a matvec), or r non-zero only on the rows of each column's source site (the first right-hand
// side Lambda delta_s) and no column of the tile has its source here
__device__ __forceinline__ bool r_is_zero(const FusedInst& I, int site, int n_first, int NB, int lane) {
  if (I.r == nullptr) return true;
  if (!I.rsrc) return false;
  bool here = false;
  for (int n = n_first + lane; n < min(I.ncol, n_first + NB); n += 32) here |= __ldg(I.rsrc + n) == site;
  return !__any_sync(0xffffffffu, here);
}

template <int GT, bool SPLIT>
__global__ void __launch_bounds__(F_THREADS, 1)
    k_tc_fused(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
               const __grid_constant__ FusedInst I, int* __restrict__ err, int sweep, const int* __restrict__ run,
               const int* __restrict__ sweeps_done) {
  using namespace ptx;
  using Cfg = FusedCfg<GT, SPLIT>;
  constexpr int STAGES = Cfg::STAGES, NBUF = Cfg::NBUF, STAGE = Cfg::STAGE, NB = Cfg::NB, X_TILE = Cfg::X_TILE;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_a[STAGES], xready[STAGES], full[STAGES], empty[STAGES];
  __shared__ __align__(8) uint64_t acc_full[NBUF], acc_empty[NBUF], drain;
  __shared__ uint32_t tmem_holder;
  __shared__ WaitCtl wctl;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int KB = (GT == 2 ? I.Ns : 2 * I.Ns) / F_BK;    // k-blocks of 64 complex points, or 64 real values
  const int row_gap = GT == 2 ? I.Ns : 0;               // rows of the two accumulators: z and Ns + z
  int tiles = I.Lx * I.Ly * ((I.ncol + NB - 1) / NB) * fused_row_tiles<GT>(I.Ns);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_a[s], 1);
      mbar_init(&xready[s], F_PROD_WARPS);              // this CTA's producer warps wrote X
      mbar_init(&full[s], 2);                           // each CTA's relay (even CTA's copy)
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 256);                    // 128 epilogue threads of each CTA
    }
    mbar_init(&drain, 1);
    wait_ctl_init(&wctl);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(&tmem_holder, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = tmem_holder;
  volatile WaitCtl* abort_p = &wctl;
  auto stage_ptr = [&](int s) { return smem + (size_t)s * STAGE; };
  // Everything above runs under the end of the kernel before (launch_overlapped).  A sweep enqueued behind
  // the end of its series has no tiles (every CTA reads the same flag); in a batch the sweep number (for the
  // support table) is the device count of sweeps done, plus one.
  grid_launch_next();
  grid_wait();
  if (run && *(volatile const int*)run == 0) tiles = 0;
  if (sweeps_done) sweep = *(volatile const int*)sweeps_done + 1;

  // each warpgroup sets its register budget first, in its own branch, so that the code of
  // each role is compiled against that budget
  if (warp < F_PROD_W0) {
    reg_budget<F_REG_CTRL, F_REGS_AT_LAUNCH>();
    if (warp == 0) {
      if (lane == 0) {
        // ---------------- TMA: Lambda hi / lo (each CTA its own rows) ----------------
        int g = 0;
        bool ok = true;
        for (int tile = pair; tile < tiles && ok; tile += npairs) {
          const FTile T = fused_tile<Cfg>(I, tile, sweep);
          if (!T.active) continue;
          for (int kb = 0; kb < KB; ++kb, ++g) {
            const int s = g % STAGES;
            if (g >= STAGES && !mbar_wait(&empty[s], ((g / STAGES) - 1) & 1, abort_p)) {
              ok = false;
              break;
            }
            uint8_t* st = stage_ptr(s);
            mbar_expect_tx(&full_a[s], GT * F_A_GROUP);
#pragma unroll
            for (int gi = 0; gi < GT; ++gi) {
              const int row0 = T.gt * PM + (int)rank * BM + gi * row_gap;
              tma_load_3d(st + gi * F_A_GROUP, &map_hi, &full_a[s], kb * F_BK, row0, T.site);
              tma_load_3d(st + gi * F_A_GROUP + A_TILE, &map_lo, &full_a[s], kb * F_BK, row0, T.site);
            }
          }
        }
        for (int q = g > STAGES ? g - STAGES : 0; q < g; ++q)
          mbar_wait(&full_a[q % STAGES], (q / STAGES) & 1, abort_p, false);
      }
    } else if (warp == 1) {
      if (lane == 0 && rank == 0) {
        // ---------------- MMA issuer (even CTA) ----------------
        int g = 0, t = 0;
        bool ok = true, any = false;
        for (int tile = pair; tile < tiles && ok; tile += npairs) {
          const FTile T = fused_tile<Cfg>(I, tile, sweep);
          if (!T.active) continue;
          const int buf = t % NBUF;
          if (t >= NBUF && !mbar_wait_cluster(&acc_empty[buf], ((t / NBUF) - 1) & 1, abort_p)) break;
          ++t;
          tc_fence_after();
          for (int kb = 0; kb < KB; ++kb, ++g) {
            const int s = g % STAGES;
            if (!mbar_wait_cluster(&full[s], (g / STAGES) & 1, abort_p)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t st = smem_u32(stage_ptr(s));
            const uint32_t xb = st + GT * F_A_GROUP;
            // The small products first, since the accumulators round relative to what they hold: the final residual fell
            // on 28 of 30 drawn problems, by 19 % in the median; 16x16, Nc = 256, 1.8 % faster, 8x8, Nc = 128, 1.2 %
            // slower.
#pragma unroll
            for (int hi = 0; hi < 2; ++hi) {
#pragma unroll
              for (int k16 = 0; k16 < F_BK / 16; ++k16) {
                const uint32_t off = k16 * 32;
                // (fresh: the first products of an output overwrite what its accumulators held)
                auto products = [&](uint32_t dacc, uint32_t a, uint32_t x, uint32_t idesc, bool fresh) {
                  const uint64_t ah = sdesc_sw128(a + off), al = sdesc_sw128(a + A_TILE + off);
                  const uint64_t xh = sdesc_sw128(x + off), xl = sdesc_sw128(x + X_TILE + off);
                  if (hi) {
                    mma_pair_f16(dacc + (uint32_t)(k16 % Cfg::LARGE) * Cfg::ACC_STRIDE, ah, xh, idesc,
                                 SPLIT && fresh && kb == 0 && k16 < Cfg::LARGE ? 0u : 1u);
                  } else {
                    const uint32_t small = dacc + (uint32_t)(Cfg::ACCS - 1) * Cfg::ACC_STRIDE;
                    mma_pair_f16(small, ah, xl, idesc, fresh && (kb | k16) == 0 ? 0u : 1u);
                    mma_pair_f16(small, al, xh, idesc, 1u);
                  }
                };
                const uint32_t d0 = tmem + (uint32_t)(buf * GT * NB);
                products(d0, st, xb, Cfg::IDESC, true);                                   // Re Xr (or A X)
                if constexpr (GT == 2) {
                  const uint32_t im = st + F_A_GROUP, xi = xb + 2 * X_TILE, d1 = d0 + NB;
                  products(d0, im, xi, Cfg::IDESC | F_NEGATE_A, false);                     // - Im Xi
                  products(d1, im, xb, Cfg::IDESC, true);                                 // Im Xr
                  products(d1, st, xi, Cfg::IDESC, false);                                // Re Xi
                }
              }
            }
            mma_commit_pair_mc(&empty[s], 0x3);
            any = true;
          }
          if (ok) mma_commit_pair_mc(&acc_full[buf], 0x3);
        }
        if (any) {
          mma_commit_pair_mc(&drain, 0x1);
          mbar_wait(&drain, 0, abort_p, false);
        }
      }
    } else if (warp == F_RELAY_W) {
      if (lane == 0) {
        // ---------------- relay: this CTA's stage complete -> even CTA's stage barrier ----------------
        const uint32_t full_bar0 = mapa(smem_u32(&full[0]), 0);
        int g = 0;
        bool ok = true;
        for (int tile = pair; tile < tiles && ok; tile += npairs) {
          const FTile T = fused_tile<Cfg>(I, tile, sweep);
          if (!T.active) continue;
          for (int kb = 0; kb < KB; ++kb, ++g) {
            const int s = g % STAGES;
            if (!mbar_wait(&full_a[s], (g / STAGES) & 1, abort_p) || !mbar_wait(&xready[s], (g / STAGES) & 1, abort_p)) {
              ok = false;
              break;
            }
            mbar_arrive_remote(full_bar0 + (uint32_t)(s * 8));
          }
        }
      }
    }
  } else if (warp < F_EPI_W0) {
    reg_budget<F_REG_PROD, F_REGS_AT_LAUNCH>();
    // ---------------- gather producers (both CTAs) ----------------
    // thread pt: the float4 groups k = 4 j .. + 3 and 32 + 4 j .. + 3 of 64 values (so that eight
    // lanes read 128 contiguous bytes) for the tile columns c0 + 32 i, i < NB / 64, of this CTA's half.
    // c0: the two columns of a half warp differ in bit 2, so that their 8-byte stores, which the
    // 128-byte swizzle places in one 64-byte half of a row each, meet in different banks.
    const int pt = threadIdx.x - F_PROD_W0 * 32;
    const int j = pt & 7, r4 = (pt >> 3) & 3, wv = pt >> 5;
    const int c0 = (wv >> 1) * 8 + (wv & 1) * 2 + (r4 >> 1) + (r4 & 1) * 4;
    int g = 0;
    int ok = 1;
    for (int tile = pair; tile < tiles && ok; tile += npairs) {
      const FTile T = fused_tile<Cfg>(I, tile, sweep);
      if (!T.active) continue;
      const int Ns = I.Ns, N2 = 2 * Ns, ncol = I.ncol, gs = I.gs;
      const float* din = I.din;
      const float* __restrict__ Jz = I.Jz;
      const TcScale* sc = I.sc;
      int nb[4], bd[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        nb[q] = __ldg(I.nbr + T.site * 4 + q);
        bd[q] = nb[q] >= 0 ? __ldg(I.nbond + T.site * 4 + q) : 0;
      }
      const int col0 = T.nt * NB + (int)rank * (NB / 2);
      // this thread's columns col0 + c0 + 32 i, i < ni, lie before the end
      const int ni = max(0, min(NB / 64, (ncol - col0 - c0 + 31) / 32));
      float up[NB / 64];
#pragma unroll
      for (int i = 0; i < NB / 64; ++i) up[i] = i < ni ? load_f(&sc[(col0 + c0 + 32 * i) / gs].up) : 0.f;
      // row of neighbour q at the first column (a valid address also where the neighbour is missing)
      const float* nbp[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        nbp[q] = din + (nb[q] >= 0 && ni > 0 ? ((size_t)nb[q] * ncol + col0 + c0) * N2 : 0) + 4 * j;
      const size_t cstride = (size_t)32 * N2;            // 32 columns further
      // A k-block is gathered in two steps of two columns: GT = 2, the real, then the imaginary parts
      // of both columns; GT = 1, two columns after the other two.  The sixteen neighbour loads of a
      // step are issued back to back (no load behind a branch) one step ahead of their sums, so that
      // their latency overlaps the previous step's sums, stores and stage wait.
      float4 v[4][2][2], jv[4][2];
      auto issue = [&](int kb, int h) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int ci = GT == 2 ? i : 2 * h + i;
            const bool ok_qi = nb[q] >= 0 && ci < ni;
            const float* p = ok_qi ? nbp[q] + ci * cstride + kb * F_BK + (GT == 2 ? h * Ns : 0) : nbp[q];
            v[q][i][0] = load_f4(p);
            v[q][i][1] = load_f4(p + 32);
          }
      };
      auto issue_j = [&](int kb) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = kb * F_BK + 32 * u + 4 * j;
          const int kz = k < Ns ? k : k - Ns;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            jv[q][u] = __ldg(reinterpret_cast<const float4*>(Jz + (size_t)bd[q] * Ns + kz));
            if (nb[q] < 0) jv[q][u] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
      };
      issue(0, 0);
      issue_j(0);
      for (int kb = 0; kb < KB; ++kb, ++g) {
        const int s = g % STAGES;
        uint8_t* xs = stage_ptr(s) + GT * F_A_GROUP;
#pragma unroll
        for (int h = 0; h < Cfg::STEPS; ++h) {
          float4 acc[2][2];
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                if (nb[q] >= 0 && (GT == 2 ? i : 2 * h + i) < ni) {
                  a.x = fmaf(jv[q][u].x, v[q][i][u].x, a.x);
                  a.y = fmaf(jv[q][u].y, v[q][i][u].y, a.y);
                  a.z = fmaf(jv[q][u].z, v[q][i][u].z, a.z);
                  a.w = fmaf(jv[q][u].w, v[q][i][u].w, a.w);
                }
              }
              acc[i][u] = a;
            }
          if (h + 1 < Cfg::STEPS) issue(kb, h + 1);
          else if (kb + 1 < KB) {
            issue(kb + 1, 0);
            issue_j(kb + 1);
          }
          if (h == 0) {
            if (g >= STAGES && !mbar_wait(&empty[s], ((g / STAGES) - 1) & 1, abort_p)) ok = 0;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int ci = GT == 2 ? i : 2 * h + i, c = c0 + 32 * ci;
            uint8_t* xd = xs + (GT == 2 ? h * 2 * X_TILE : 0);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const float f = up[ci];
              const int off = c * 128 + (((4 * u + (j >> 1)) ^ (c & 7)) << 4) + (j & 1) * 8;
              uint2 hi, lo;
              split_f16(acc[i][u].x * f, acc[i][u].y * f, hi.x, lo.x);
              split_f16(acc[i][u].z * f, acc[i][u].w * f, hi.y, lo.y);
              *reinterpret_cast<uint2*>(xd + off) = hi;
              *reinterpret_cast<uint2*>(xd + X_TILE + off) = lo;
            }
          }
        }
        if (!ok) break;
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&xready[s]);
      }
    }
  } else {
    reg_budget<F_REG_EPI, F_REGS_AT_LAUNCH>();
    // ---------------- epilogue (both CTAs, own 128 rows of each accumulator) ----------------
    const int q4 = warp - F_EPI_W0;
    const uint32_t empty_bar0 = mapa(smem_u32(&acc_empty[0]), 0);
    int t = 0;
    bool go = true;
    for (int tile = pair; tile < tiles && go; tile += npairs) {
      const FTile T = fused_tile<Cfg>(I, tile, sweep);
      if (!T.active) continue;
      const int buf = t % NBUF;
      const int N2 = 2 * I.Ns, gs = I.gs, n_first = T.nt * NB;
      const int m0 = T.gt * PM + (int)rank * BM + q4 * 32;
      const bool rows = m0 < (GT == 2 ? I.Ns : N2);       // a last row tile may be short (warp-uniform)
      const float ad = rows ? __ldg(I.adown + (size_t)T.site * N2 + m0 + lane) : 0.f;   // one scale for rows z and Ns + z
      unsigned long long* norm = I.norm;
      TcScale* sc = I.sc;
      const uint32_t tacc = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(buf * GT * NB);
      auto body = [&](auto E) {
        E.r = I.r;
        E.din = I.din;
        E.dout = I.dout;
        E.n_first = n_first;
        E.ncol = rows ? I.ncol : 0;
        E.N2 = N2;
        E.row_gap = row_gap;
        E.base0 = ((size_t)T.site * I.ncol + n_first) * N2 + m0 + lane;
        E.template load<0>(0);
        go = mbar_wait(&acc_full[buf], (t / NBUF) & 1, abort_p);
        go = __all_sync(0xffffffffu, go);                 // tcgen05.ld below is warp-collective
        if (!go) return;
        tc_fence_after();
        constexpr int CHUNKS = decltype(E)::CHUNKS;
        for (int e = 0; e < CHUNKS; e += 2) {
          E.template load<1>(e + 1);
          E.template chunk<0>(e, tacc, ad, gs, norm, sc, lane);
          if (e + 2 < CHUNKS) E.template load<0>(e + 2);
          E.template chunk<1>(e + 1, tacc, ad, gs, norm, sc, lane);
        }
        if (E.qcur >= 0) E.flush(norm, sc, lane);
      };
      if (r_is_zero(I, T.site, n_first, NB, lane)) body(FusedEpilogue<Cfg, true>{});
      else body(FusedEpilogue<Cfg, false>{});
      ++t;
      if (!go) break;
      tc_fence_before();
      mbar_arrive_remote(empty_bar0 + (uint32_t)(buf * sizeof(uint64_t)));
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
  if (threadIdx.x == 0 && wctl.abort) atomicExch(err, 1);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 3D map over an fp32 array [d2][d1][d0] with a (32 x box1 x 1) box, 128-byte swizzle
bool make_map(CUtensorMap* m, const float* base, uint64_t d0, uint64_t d1, uint64_t d2, uint32_t box1) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {d0 * 4, d0 * d1 * 4};
  cuuint32_t box[3] = {(cuuint32_t)BK, box1, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void*)base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3D map over an fp16 array [d2][d1][d0] with a (64 x box1 x 1) box, 128-byte swizzle
bool make_map16(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint32_t box1) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {d0 * 2, d0 * d1 * 2};
  cuuint32_t box[3] = {(cuuint32_t)F_BK, box1, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

TcState* state(dyson_ctx* c) {
  if (!c->tc) c->tc = new TcState();
  return static_cast<TcState*>(c->tc);
}

cudaLaunchConfig_t pair_config(cudaLaunchAttribute* at, unsigned pairs, int threads, size_t smem, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// co-resident CTA pairs of k_tc_gemm_pair on this device (0: the pair kernel cannot run)
int pair_clusters(dyson_ctx* c, TcState* st) {
  if (st->pair_clusters >= 0) return st->pair_clusters;
  st->pair_clusters = 0;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) sms = 0;
  if (sms >= 2 &&
      cudaFuncSetAttribute(k_tc_gemm_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, P_SMEM_BYTES) == cudaSuccess) {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = pair_config(at, (unsigned)(sms / 2), THREADS, P_SMEM_BYTES, c->stream);
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, k_tc_gemm_pair, &cfg) == cudaSuccess) st->pair_clusters = ncl;
  }
  cudaGetLastError();
  return st->pair_clusters;
}

// co-resident CTA pairs of k_tc_fused<GT, SPLIT> on this device (0: it cannot run)
template <int GT, bool SPLIT>
int fused_clusters_of(dyson_ctx* c) {
  const auto kernel = k_tc_fused<GT, SPLIT>;
  constexpr int smem = FusedCfg<GT, SPLIT>::SMEM;
  int sms = 0, n = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) sms = 0;
  // the warpgroups' register shares add up to exactly F_REGS_AT_LAUNCH per thread: with
  // any other count at launch the producers' increase could not be met, so the kernel is
  // not offered
  cudaFuncAttributes fa = {};
  if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess || fa.numRegs != F_REGS_AT_LAUNCH) sms = 0;
  if (sms >= 2 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess) {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = pair_config(at, (unsigned)(sms / 2), F_THREADS, smem, c->stream);
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, kernel, &cfg) == cudaSuccess) n = ncl;
  }
  cudaGetLastError();
  return n;
}

// pairs for every form of the fused kernel (0 where one of them cannot run)
int fused_clusters(dyson_ctx* c) {
  TcState* st = state(c);
  if (st->fused_clusters < 0)
    st->fused_clusters = std::min({fused_clusters_of<1, false>(c), fused_clusters_of<2, false>(c),
                                   fused_clusters_of<1, true>(c), fused_clusters_of<2, true>(c)});
  return st->fused_clusters;
}

// Several accumulators per output where the sweep takes the place of full FP32 products (k_tc_fused's comment).
bool fused_split(const dyson_ctx* c) { return c->Nc % 64 != 0; }
// Complex tiles wherever their 256 points are at least five eighths full: X is then gathered once per
// (site, column tile) and Lambda read once.  Shorter contours would fill a half at most; up to 128 points their
// embedding has a single tile of 256 rows.
// (SPLIT <2> has no room for two large accumulators: up to 191 points its residual is as large as the FP32 sweep's.)
int fused_gt_of(const dyson_ctx* c) { return contour_stride(c) >= (fused_split(c) ? 256 : 192) ? 2 : 1; }

// form of the fused kernel that serves the context's variant (0: none).  The unfused forms serve
// only contours that fill their tiles; every other contour takes the fused kernel.
int fused_gt(dyson_ctx* c) {
  const bool unfused = (c->tc_variant == DYSON_SWEEP_SINGLE_CTA || c->tc_variant == DYSON_SWEEP_CTA_PAIR ||
                        c->many_of_64) &&
                       c->Nc % 64 == 0;
  if (unfused || !encode_fn()) return 0;
  return fused_clusters(c) > 0 ? fused_gt_of(c) : 0;
}

}  // namespace

int contour_stride(const dyson_ctx* c) { return (c->Nc + 63) / 64 * 64; }

bool tc_uses_fused(dyson_ctx* c) { return fused_gt(c) > 0; }

bool tc_uses_pair(dyson_ctx* c) {
  return c->tc_variant == DYSON_SWEEP_CTA_PAIR && c->Nc % 128 == 0 && pair_clusters(c, state(c)) > 0;
}

// (below 24 points more than five eighths of a padded column would be zeros)
bool tc_supported(dyson_ctx* c) {
  return c->Nc >= 24 && encode_fn() != nullptr && (c->Nc % 64 == 0 || fused_gt(c) > 0);
}

namespace {

int tc_prepare_common(dyson_ctx* c) {
  TcState* st = state(c);
  if (!st->d_err) {
    DY_CUDA(c, cudaMalloc(&st->d_err, sizeof(int)));
    DY_CUDA(c, cudaMemsetAsync(st->d_err, 0, sizeof(int), c->stream));
    DY_CUDA(c, cudaDeviceGetAttribute(&st->num_sms, cudaDevAttrMultiProcessorCount, c->device));
  }
  return DYSON_OK;
}

// tensor maps of the FP16 Lambda
int tc_prepare_fused(dyson_ctx* c) {
  int rc = tc_prepare_common(c);
  if (rc) return rc;
  TcState* st = state(c);
  const int N2 = 2 * contour_stride(c);
  if (st->h_hi_ptr != c->d_lam16_hi || st->h_lo_ptr != c->d_lam16_lo) {
    if (!make_map16(&st->h_hi, c->d_lam16_hi, N2, N2, c->Nr, BM) || !make_map16(&st->h_lo, c->d_lam16_lo, N2, N2, c->Nr, BM))
      return ctx_fail(c, DYSON_ERR_CUDA, "cuTensorMapEncodeTiled failed for the FP16 Lambda");
    st->h_hi_ptr = c->d_lam16_hi;
    st->h_lo_ptr = c->d_lam16_lo;
  }
  return DYSON_OK;
}

// tensor maps of the TF32 Lambda and the gather buffer of the unfused forms, for ncol columns
int tc_prepare(dyson_ctx* c, int ncol) {
  int rc = tc_prepare_common(c);
  if (rc) return rc;
  TcState* st = state(c);
  const int Nc = c->Nc, N2 = 2 * Nc, Nr = c->Nr;
  if (st->a_hi_ptr != c->d_lam_hi || st->a_lo_ptr != c->d_lam_lo) {
    if (!make_map(&st->a_hi, c->d_lam_hi, N2, N2, Nr, BM) || !make_map(&st->a_lo, c->d_lam_lo, N2, N2, Nr, BM))
      return ctx_fail(c, DYSON_ERR_CUDA, "cuTensorMapEncodeTiled failed for Lambda");
    st->a_hi_ptr = c->d_lam_hi;
    st->a_lo_ptr = c->d_lam_lo;
  }
  if (!st->smem_set) {
    DY_CUDA(c, cudaFuncSetAttribute(k_tc_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    st->smem_set = true;
  }
  size_t xbytes = (size_t)Nr * ncol * N2 * sizeof(float);
  if (st->xbuf_bytes < xbytes) {
    if (st->xbuf) cudaFree(st->xbuf);
    st->xbuf = nullptr;
    st->xbuf_bytes = 0;
    cudaError_t e = cudaMalloc(&st->xbuf, xbytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return ctx_fail(c, DYSON_ERR_OOM, "tensor-core gather buffer");
    }
    st->xbuf_bytes = xbytes;
    st->x_ptr = nullptr;
  }
  if (st->x_ptr != st->xbuf || st->x_ncol != ncol) {
    if (!make_map(&st->x, st->xbuf, N2, ncol, Nr, BN))
      return ctx_fail(c, DYSON_ERR_CUDA, "cuTensorMapEncodeTiled failed for X");
    st->x_ptr = st->xbuf;
    st->x_ncol = ncol;
  }
  return DYSON_OK;
}

template <int GT, bool SPLIT>
int launch_fused(dyson_ctx* c, const FusedInst& e, int sweep, const int* run, const int* sweeps_done,
                 cudaStream_t stream) {
  TcState* st = state(c);
  const int NB = FusedCfg<GT, SPLIT>::NB;
  const long long tiles = (long long)e.Lx * e.Ly * ((e.ncol + NB - 1) / NB) * fused_row_tiles<GT>(e.Ns);
  cudaLaunchAttribute at[2];
  cudaLaunchConfig_t cfg = pair_config(at, (unsigned)std::min<long long>(tiles, fused_clusters(c)), F_THREADS,
                                       FusedCfg<GT, SPLIT>::SMEM, stream);
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  if (c->overlap) cfg.numAttrs = 2;
  DY_CUDA(c, cudaLaunchKernelEx(&cfg, k_tc_fused<GT, SPLIT>, st->h_hi, st->h_lo, e, st->d_err, sweep, run, sweeps_done));
  DY_CUDA(c, cudaGetLastError());
  c->launches += 1;
  return DYSON_OK;
}

}  // namespace

float tc_jbound(const dyson_ctx* c) { return 4.f * c->j_max; }

int tc_seed_scale(dyson_ctx* c, int ng, const double* ref, double bound) {
  k_tc_seed<<<(ng + 127) / 128, 128, 0, c->stream>>>(c->d_xscale, ng, ref, (float)bound);
  c->launches += 1;
  DY_CUDA(c, cudaGetLastError());
  return DYSON_OK;
}

int tc_seed_scale_scan(dyson_ctx* c, int ncol, int gs, const float* d) {
  int rc = tc_seed_scale(c, (ncol + gs - 1) / gs, nullptr, 0.0);
  if (rc) return rc;
  const size_t warps = (size_t)c->Nr * ncol;
  k_tc_seed_scan<<<(unsigned)((warps + 7) / 8), 256, 0, c->stream>>>(d, c->Nr, contour_stride(c), ncol, gs,
                                                                     c->d_xscale);
  c->launches += 1;
  DY_CUDA(c, cudaGetLastError());
  return DYSON_OK;
}

int tc_set_scale(dyson_ctx* c, int ng) {
  k_tc_scale<<<(ng + 127) / 128, 128, 0, c->stream>>>(c->d_xscale, ng, tc_jbound(c));
  c->launches += 1;
  DY_CUDA(c, cudaGetLastError());
  return DYSON_OK;
}

int tc_prepare_sweep(dyson_ctx* c, int ncol, bool fused) {
  return fused || fused_gt(c) > 0 ? tc_prepare_fused(c) : tc_prepare(c, ncol);
}

bool tc_fused_runs(dyson_ctx* c) { return encode_fn() && fused_clusters(c) > 0; }

int tc_fused_sweep(dyson_ctx* c, int ncol, int gs, const float* r, const float* din, float* dout, const int* act,
                   int sweep, int rform, const int* run, const int* sweeps_done, cudaStream_t stream) {
  int rc = tc_prepare_fused(c);
  if (rc) return rc;
  FusedInst e = {};
  e.r = rform == TC_R_ZERO ? nullptr : r;
  e.din = din;
  e.dout = dout;
  e.Jz = c->d_Jz;
  e.nbr = c->d_nbr;
  e.nbond = c->d_nbond;
  e.norm = c->d_norm;
  e.adown = c->d_a_down;
  e.sc = c->d_xscale;
  e.rsrc = rform == TC_R_ON_SOURCES ? c->d_src_site : nullptr;
  e.act = act;
  e.Lx = c->Lx;
  e.Ly = c->Ly;
  e.Ns = contour_stride(c);
  e.ncol = ncol;
  e.gs = gs;
  const auto launch = fused_gt_of(c) == 1 ? (fused_split(c) ? launch_fused<1, true> : launch_fused<1, false>)
                                          : (fused_split(c) ? launch_fused<2, true> : launch_fused<2, false>);
  return launch(c, e, sweep, run, sweeps_done, stream);
}

int tc_sweep(dyson_ctx* c, int ncol, int gs, const float* r, const float* din, float* dout, int phases,
             const int* act, int sweep, int rform) {
  const int gt = fused_gt(c);
  int rc;
  if (gt > 0) {
    // one launch gathers and multiplies: the gather phase alone launches nothing
    if (!(phases & TC_GEMM)) return tc_prepare_fused(c);
    if ((rc = tc_set_scale(c, (ncol + gs - 1) / gs))) return rc;
    return tc_fused_sweep(c, ncol, gs, r, din, dout, act, sweep, rform, nullptr, nullptr, c->stream);
  }
  if ((rc = tc_prepare(c, ncol))) return rc;
  TcState* st = state(c);
  const int Nc = c->Nc, N2 = 2 * Nc, Nr = c->Nr;
  if (phases & TC_GATHER) {
    k_tc_gather<<<Nr * ((ncol + GATHER_COLS - 1) / GATHER_COLS), 256, 0, c->stream>>>(
        din, c->d_Jz, c->d_nbr, c->d_nbond, st->xbuf, Nr, Nc, ncol, act, sweep);
    DY_CUDA(c, cudaGetLastError());
    c->launches += 1;
  }
  if (!(phases & TC_GEMM)) return DYSON_OK;
  // truncated sweeps run on the single-CTA kernel, which skips tiles
  if (!act && tc_uses_pair(c)) {
    if (st->xh_ptr != st->xbuf || st->xh_ncol != ncol) {
      if (!make_map(&st->xh, st->xbuf, N2, ncol, Nr, BN / 2))
        return ctx_fail(c, DYSON_ERR_CUDA, "cuTensorMapEncodeTiled failed for X halves");
      st->xh_ptr = st->xbuf;
      st->xh_ncol = ncol;
    }
    const long long tiles = (long long)(N2 / PM) * ((ncol + BN - 1) / BN) * Nr;
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = pair_config(at, (unsigned)std::min<long long>(tiles, st->pair_clusters), THREADS,
                                         P_SMEM_BYTES, c->stream);
    DY_CUDA(c, cudaLaunchKernelEx(&cfg, k_tc_gemm_pair, st->a_hi, st->a_lo, st->xh, r, din, dout, Nr, Nc, ncol, gs,
                                  c->d_norm, st->d_err));
  } else {
    const long long tiles = (long long)(N2 / BM) * ((ncol + BN - 1) / BN) * Nr;
    const int grid = (int)std::min<long long>(tiles, st->num_sms);
    k_tc_gemm<<<grid, THREADS, SMEM_BYTES, c->stream>>>(st->a_hi, st->a_lo, st->x, r, din, dout, Nr, Nc, ncol, gs,
                                                        c->d_norm, st->d_err, act, sweep);
  }
  DY_CUDA(c, cudaGetLastError());
  c->launches += 1;
  return DYSON_OK;
}

int tc_set_wait_limit(dyson_ctx* c, unsigned long long ns) {
  DY_CUDA(c, cudaMemcpyToSymbolAsync(ptx::g_wait_limit_ns, &ns, sizeof ns, 0, cudaMemcpyHostToDevice, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  return DYSON_OK;
}

int tc_error_enqueue(dyson_ctx* c) {
  TcState* st = static_cast<TcState*>(c->tc);
  if (!st || !st->d_err) return DYSON_OK;
  if (!st->h_err) {
    DY_CUDA(c, cudaMallocHost((void**)&st->h_err, sizeof(int)));
    *st->h_err = 0;
  }
  DY_CUDA(c, cudaMemcpyAsync(st->h_err, st->d_err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  return DYSON_OK;
}

int tc_error_status(dyson_ctx* c) {
  TcState* st = static_cast<TcState*>(c->tc);
  if (!st || !st->h_err || !*st->h_err) return DYSON_OK;
  *st->h_err = 0;
  cudaMemsetAsync(st->d_err, 0, sizeof(int), c->stream);
  return ctx_fail(c, DYSON_ERR_TIMEOUT, "a tensor-core pipeline wait exceeded its time limit");
}

int tc_check_error(dyson_ctx* c) {
  int rc = tc_error_enqueue(c);
  if (rc) return rc;
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  return tc_error_status(c);
}

size_t tc_x_bytes(const dyson_ctx* c) {
  const TcState* st = static_cast<const TcState*>(c->tc);
  return st ? st->xbuf_bytes : 0;
}

void tc_release_x(dyson_ctx* c) {
  TcState* st = static_cast<TcState*>(c->tc);
  if (!st) return;
  cudaFree(st->xbuf);
  st->xbuf = nullptr;
  st->xbuf_bytes = 0;
  st->x_ptr = st->xh_ptr = nullptr;
}

void tc_release(dyson_ctx* c) {
  TcState* st = static_cast<TcState*>(c->tc);
  if (!st) return;
  if (st->xbuf) cudaFree(st->xbuf);
  if (st->d_err) cudaFree(st->d_err);
  if (st->h_err) cudaFreeHost(st->h_err);
  delete st;
  c->tc = nullptr;
}
