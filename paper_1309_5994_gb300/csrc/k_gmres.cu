// Preconditioned GMRES of App. C as the inner solver of the mixed-precision path.
//
// The refinement needs d with (I - K) d = r (r: the FP64-accurate residual,
// rounded to the FP32 planar state).  With the block-diagonal preconditioner
// P = B^{-1} of App. C the preconditioned operator is I - K, the initial guess
// is u0 = P b (here r itself) and the first residue is z0 = r - (I - K) r = K r.
// Per column (vector column n of the chunk, its own Krylov space):
//   q_0 = z0 / |z0|;  for j = 0, 1, ...:
//     w = (I - K) q_j                      (K: the 3xTF32 tensor-core sweep with a zero r)
//     two passes of classical Gram-Schmidt: h_ij += <q_i, w>, w -= h_ij q_i (i <= j)
//     h_{j+1,j} = |w|,  q_{j+1} = w / h_{j+1,j}
//     complex Givens rotations reduce the Hessenberg column; |g_{j+1}| is the
//     preconditioned residual of the current iterate
//   until max_n |g_{j+1}| / |r_n| <= tol or j + 1 = m (restart from the iterate);
//   then y = R^{-1} g and d = u0 + sum_i y_i q_i.
// Vectors are FP32 planar states [Nr][ncol][2Nc]; reductions, rotations and the
// small triangular solves are FP64.  The series stalls where the FP32 rounding of
// its transient partial sums is amplified beyond 1 (long contours) or diverges
// (spectral radius of K above 1); GMRES converges in both cases because each
// Krylov vector is normalised and the residual is minimised.
#include <cmath>
#include <vector>

#include "common.cuh"
#include "detail.cuh"
#include "gmres.cuh"
#include "sumsq.cuh"
#include "tc.cuh"

using namespace dyson_detail;

namespace {

constexpr int GM_THREADS = 256;

struct GmState {
  float* Q = nullptr;                 // m + 1 Krylov vectors
  float* zero = nullptr;              // zero right-hand side of the matvec
  float* u = nullptr;                 // K q_j
  float* w = nullptr;                 // the vector being orthogonalised
  double2* h = nullptr;               // [ncol][m + 1] first-pass projections of the current column
  double2* h2 = nullptr;              // [ncol][m + 1] second-pass projections
  double* nrm = nullptr;              // [ncol] |w|^2 after orthogonalisation
  double* nrm0 = nullptr;             // [ncol] |(I - K) q_j|^2 before it
  double* nrm1 = nullptr;             // [ncol] |w|^2 after the first pass
  double* bnorm = nullptr;            // [ncol] |r|
  double* beta = nullptr;             // [ncol] |z0| of the current cycle
  double* cs = nullptr;               // [ncol][m] Givens cosines
  double2* sn = nullptr;              // [ncol][m] Givens sines
  double2* g = nullptr;               // [ncol][m + 1] rotated right-hand side
  double2* R = nullptr;               // [ncol][m][m] rotated Hessenberg (column j at R[n][.][j])
  double2* y = nullptr;               // [ncol][m]
  unsigned long long* res = nullptr;  // max over columns of |g_{j+1}| / |r| (bits of a double)
  unsigned long long* h_res = nullptr;
  size_t vsz = 0;
  int m = 0, ncol = 0;
};

GmState* gstate(dyson_ctx* c) {
  if (!c->gm) c->gm = new GmState();
  return static_cast<GmState*>(c->gm);
}

__device__ __forceinline__ double2 gm_mul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 gm_conj(double2 a) { return make_double2(a.x, -a.y); }

// Second Gram-Schmidt pass only where the first lost most of the vector: the
// test of Daniel, Gragg, Kaufman and Stewart, |w| < 0.7 |(I - K) q_j|.
__device__ __forceinline__ bool reorth_needed(const double* after, const double* before, int n) {
  return after[n] < 0.49 * before[n];
}

// The vector kernels work on items: one warp, one column n, VEC 32 T contour points of one site, real
// and imaginary parts in registers (VEC = 4 where the stride allows float4 loads).  Items of a column
// are numbered site-major; a block takes a range of one column's items, its warps every eighth of them.
// They are bound by HBM: per Arnoldi step the basis is read once for the projections and once for
// the update.  12x12, Nc = 384, 384 columns (170 MB a vector): see the rates at k_gm_dots.
template <int VEC, int T>
struct Slab {
  float re[T][VEC], im[T][VEC];
};
struct ItemPos {
  size_t base;                                          // first element of (site, column)
  int z0;                                               // first contour point of this lane
};
template <int VEC, int T>
__device__ __forceinline__ ItemPos item_pos(int item, int nz, int n, int ncol, int Ns, int lane) {
  const int s = item / nz, zc = item - s * nz;
  return {((size_t)s * ncol + n) * 2 * Ns, (zc * 32 * T + lane) * VEC};
}
template <int VEC, int T>
__device__ __forceinline__ void load_slab(Slab<VEC, T>& x, const float* __restrict__ p, ItemPos at, int Ns) {
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int z = at.z0 + 32 * VEC * t;
    const bool in = z < Ns;
    if (VEC == 4) {
      const float4 r = in ? *reinterpret_cast<const float4*>(p + at.base + z) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 i = in ? *reinterpret_cast<const float4*>(p + at.base + Ns + z) : make_float4(0.f, 0.f, 0.f, 0.f);
      x.re[t][0] = r.x; x.re[t][1 % VEC] = r.y; x.re[t][2 % VEC] = r.z; x.re[t][3 % VEC] = r.w;
      x.im[t][0] = i.x; x.im[t][1 % VEC] = i.y; x.im[t][2 % VEC] = i.z; x.im[t][3 % VEC] = i.w;
    } else {
      x.re[t][0] = in ? p[at.base + z] : 0.f;
      x.im[t][0] = in ? p[at.base + Ns + z] : 0.f;
    }
  }
}
template <int VEC, int T>
__device__ __forceinline__ void store_slab(const Slab<VEC, T>& x, float* __restrict__ p, ItemPos at, int Ns) {
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int z = at.z0 + 32 * VEC * t;
    if (z >= Ns) continue;
    if (VEC == 4) {
      *reinterpret_cast<float4*>(p + at.base + z) =
          make_float4(x.re[t][0], x.re[t][1 % VEC], x.re[t][2 % VEC], x.re[t][3 % VEC]);
      *reinterpret_cast<float4*>(p + at.base + Ns + z) =
          make_float4(x.im[t][0], x.im[t][1 % VEC], x.im[t][2 % VEC], x.im[t][3 % VEC]);
    } else {
      p[at.base + z] = x.re[t][0];
      p[at.base + Ns + z] = x.im[t][0];
    }
  }
}
template <int VEC, int T>
__device__ __forceinline__ double slab_norm2(const Slab<VEC, T>& x) {
  SumSq q;
#pragma unroll
  for (int t = 0; t < T; ++t)
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      q.add(x.re[t][v]);
      q.add(x.im[t][v]);
    }
  return q.value();
}

// Sum of eight FP64 values over a warp: halving exchanges (nine additions; the FP64 pipe takes 16 cycles
// for each); lanes 4 i .. 4 i + 3 return value i.
__device__ __forceinline__ double reduce8(double (&v)[8], int lane) {
#pragma unroll
  for (int o = 16, half = 4; o >= 4; o >>= 1, half >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const double send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// h[n][i] += <Q_i[n], a[n] - b[n]>  (b may be null) over a range of items; nrm0 (given): += |a - b|^2.
// With a gate (after, before), columns that need no second pass are skipped.  Grid (ncol, ranges).
// w = a - b of an item stays in registers while the whole basis passes by it; FP32 products are summed in
// FP32 within a lane's part of an item and in FP64 across lanes and items (GB300's FP64 pipe is too slow
// for a product per element); a warp adds up its items in shared memory.  12x12, Nc = 384, 384 columns
// (170 MB a vector), 20 basis vectors on average: 0.78 ms with groups of four basis vectors per pass over
// the items, which read a and b again for every group (not from L2: 60 MB of them are in use at a time),
// 0.44 ms with the whole basis (both Gram-Schmidt passes averaged; 6.9 TB/s).
constexpr int GM_GROUP = 4;
constexpr int GM_MAX_VEC = 64;                          // basis vectors (the restart length is at most 60)
template <int VEC, int T>
__global__ void __launch_bounds__(GM_THREADS, 2) k_gm_dots(const float* __restrict__ Q, size_t vsz, int nvec,
                                                           const float* __restrict__ a, const float* __restrict__ b,
                                                           int items, int nz, int Ns, int ncol, int items_per_blk,
                                                           double2* __restrict__ h, int hstride,
                                                           double* __restrict__ nrm0, const double* __restrict__ after,
                                                           const double* __restrict__ before) {
  __shared__ double sh[GM_THREADS / 32][2 * GM_MAX_VEC];
  __shared__ double sh_sq[GM_THREADS / 32];
  const int n = blockIdx.x;
  if (after && !reorth_needed(after, before, n)) return;
  const int i0 = blockIdx.y * items_per_blk, i1 = min(items, i0 + items_per_blk);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* mine = sh[warp];
  for (int e = lane; e < 2 * GM_MAX_VEC; e += 32) mine[e] = 0.0;
  __syncwarp();
  double sq = 0.0;
  for (int item = i0 + warp; item < i1; item += GM_THREADS / 32) {
    const ItemPos at = item_pos<VEC, T>(item, nz, n, ncol, Ns, lane);
    Slab<VEC, T> w, q[2];
    // the next basis vector's loads are in flight while one is multiplied (a vector past the last
    // reads the last one again; its sums are dropped)
    auto fetch = [&](int k, Slab<VEC, T>& y) { load_slab(y, Q + (size_t)min(k, nvec - 1) * vsz, at, Ns); };
    fetch(0, q[0]);
    load_slab(w, a, at, Ns);
    if (b) {
      load_slab(q[1], b, at, Ns);
#pragma unroll
      for (int t = 0; t < T; ++t)
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          w.re[t][v] -= q[1].re[t][v];
          w.im[t][v] -= q[1].im[t][v];
        }
    }
    if (nrm0) sq += slab_norm2(w);
    for (int g0 = 0; g0 < nvec; g0 += GM_GROUP) {
      double v8[2 * GM_GROUP];
#pragma unroll
      for (int k = 0; k < GM_GROUP; ++k) {
        fetch(g0 + k + 1, q[(k + 1) & 1]);
        const Slab<VEC, T>& y = q[k & 1];
        float sr = 0.f, si = 0.f;
#pragma unroll
        for (int t = 0; t < T; ++t)
#pragma unroll
          for (int v = 0; v < VEC; ++v) {                // conj(q) w
            sr = fmaf(y.re[t][v], w.re[t][v], fmaf(y.im[t][v], w.im[t][v], sr));
            si = fmaf(y.re[t][v], w.im[t][v], fmaf(-y.im[t][v], w.re[t][v], si));
          }
        v8[2 * k] = (double)sr;
        v8[2 * k + 1] = (double)si;
      }
      const double sum = reduce8(v8, lane);
      if ((lane & 3) == 0) mine[2 * g0 + (lane >> 2)] += sum;
    }
  }
  if (nrm0) {
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) sh_sq[warp] = sq;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 2 * nvec + (nrm0 ? 1 : 0); e += blockDim.x) {
    double v = 0.0;
    for (int q = 0; q < GM_THREADS / 32; ++q) v += e < 2 * nvec ? sh[q][e] : sh_sq[q];
    double2* hp = &h[(size_t)n * hstride + e / 2];
    atomicAdd(e == 2 * nvec ? &nrm0[n] : (e & 1 ? &hp->y : &hp->x), v);
  }
}

// sum over the block's warps of one FP64 value per lane, added to *out by one thread
__device__ __forceinline__ void block_add(double v, double* out) {
  __shared__ double sh[GM_THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < GM_THREADS / 32; ++q) t += sh[q];
    atomicAdd(out, t);
  }
}

// nrm[n] += |a[n]|^2; grid (ncol, ranges)
template <int VEC, int T>
__global__ void __launch_bounds__(GM_THREADS) k_gm_norm2(const float* __restrict__ a, int items, int nz, int Ns,
                                                         int ncol, int items_per_blk, double* __restrict__ nrm) {
  const int n = blockIdx.x, i0 = blockIdx.y * items_per_blk, i1 = min(items, i0 + items_per_blk);
  double acc = 0.0;
  for (int item = i0 + (int)(threadIdx.x >> 5); item < i1; item += GM_THREADS / 32) {
    Slab<VEC, T> x;
    load_slab(x, a, item_pos<VEC, T>(item, nz, n, ncol, Ns, threadIdx.x & 31), Ns);
    acc += slab_norm2(x);
  }
  block_add(acc, &nrm[n]);
}

// out = a - b + c elementwise over the whole chunk state
__global__ void k_gm_lin3(const float* __restrict__ a, const float* __restrict__ b, const float* __restrict__ c,
                          float* __restrict__ out, size_t n) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
    out[e] = a[e] - b[e] + c[e];
}

// v <- sqrt(v)
__global__ void k_gm_sqrt(double* __restrict__ v, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = sqrt(fmax(v[i], 0.0));
}

// w[n] = (a[n] - b[n]) + sign sum_{i < nvec} h[n][i] Q_i[n]  (b may be null), nrm[n] (given) += |w[n]|^2.
// With a gate (after, before): columns that need no second pass keep w and
// take nrm[n] = after[n].  Grid (ncol, ranges).
// (a and w may be the same array: each element is read, then written, by one thread)
template <int VEC, int T>
__global__ void __launch_bounds__(GM_THREADS) k_gm_update(const float* __restrict__ Q, size_t vsz, int nvec,
                                                          const double2* __restrict__ h, int hstride, float sign,
                                                          const float* a, const float* __restrict__ b, float* w,
                                                          int items, int nz, int Ns, int ncol, int items_per_blk,
                                                          double* __restrict__ nrm, const double* __restrict__ after,
                                                          const double* __restrict__ before) {
  __shared__ float2 hs[64];
  const int n = blockIdx.x;
  if (after && !reorth_needed(after, before, n)) {
    if (blockIdx.y == 0 && threadIdx.x == 0) atomicAdd(&nrm[n], after[n]);
    return;
  }
  for (int i = threadIdx.x; i < nvec; i += blockDim.x) {
    const double2 v = h[(size_t)n * hstride + i];
    hs[i] = make_float2(sign * (float)v.x, sign * (float)v.y);
  }
  __syncthreads();
  const int i0 = blockIdx.y * items_per_blk, i1 = min(items, i0 + items_per_blk);
  double acc = 0.0;
  for (int item = i0 + (int)(threadIdx.x >> 5); item < i1; item += GM_THREADS / 32) {
    const ItemPos at = item_pos<VEC, T>(item, nz, n, ncol, Ns, threadIdx.x & 31);
    Slab<VEC, T> x, q[3];
    load_slab(x, a, at, Ns);
    if (b) {
      load_slab(q[0], b, at, Ns);
#pragma unroll
      for (int t = 0; t < T; ++t)
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          x.re[t][v] -= q[0].re[t][v];
          x.im[t][v] -= q[0].im[t][v];
        }
    }
    auto fold = [&](const Slab<VEC, T>& y, float2 c) {
#pragma unroll
      for (int t = 0; t < T; ++t)
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          x.re[t][v] += c.x * y.re[t][v] - c.y * y.im[t][v];
          x.im[t][v] += c.x * y.im[t][v] + c.y * y.re[t][v];
        }
    };
    // three vectors' loads in flight: two ahead of the one that is added
    auto fetch = [&](Slab<VEC, T>& y, int i) {
      if (i < nvec) load_slab(y, Q + (size_t)i * vsz, at, Ns);
    };
    fetch(q[0], 0);
    fetch(q[1], 1);
    for (int i = 0; i < nvec; i += 3) {
      fetch(q[2], i + 2);
      fold(q[0], hs[i]);
      if (i + 1 >= nvec) break;
      fetch(q[0], i + 3);
      fold(q[1], hs[i + 1]);
      if (i + 2 >= nvec) break;
      fetch(q[1], i + 4);
      fold(q[2], hs[i + 2]);
    }
    store_slab(x, w, at, Ns);
    acc += slab_norm2(x);
  }
  if (nrm) block_add(acc, &nrm[n]);
}

// out[n] = x[n] / sqrt(nrm[n]) (0 where nrm = 0); grid (ncol, ranges)
template <int VEC, int T>
__global__ void __launch_bounds__(GM_THREADS) k_gm_scale(const float* __restrict__ x, const double* __restrict__ nrm,
                                                         float* __restrict__ out, int items, int nz, int Ns, int ncol,
                                                         int items_per_blk) {
  const int n = blockIdx.x, i0 = blockIdx.y * items_per_blk, i1 = min(items, i0 + items_per_blk);
  __shared__ float f_sh;
  if (threadIdx.x == 0) f_sh = nrm[n] > 0.0 ? (float)(1.0 / sqrt(nrm[n])) : 0.f;
  __syncthreads();
  const float f = f_sh;
  for (int item = i0 + (int)(threadIdx.x >> 5); item < i1; item += GM_THREADS / 32) {
    const ItemPos at = item_pos<VEC, T>(item, nz, n, ncol, Ns, threadIdx.x & 31);
    Slab<VEC, T> v;
    load_slab(v, x, at, Ns);
#pragma unroll
    for (int t = 0; t < T; ++t)
#pragma unroll
      for (int k = 0; k < VEC; ++k) {
        v.re[t][k] *= f;
        v.im[t][k] *= f;
      }
    store_slab(v, out, at, Ns);
  }
}

// Start of a cycle, per column: beta = sqrt(nrm), g = (beta, 0, ...).
__global__ void k_gm_start(int ncol, int m, const double* __restrict__ nrm, double* __restrict__ beta,
                           double2* __restrict__ g) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncol) return;
  const double b = sqrt(fmax(nrm[n], 0.0));
  beta[n] = b;
  for (int i = 0; i <= m; ++i) g[(size_t)n * (m + 1) + i] = make_double2(i == 0 ? b : 0.0, 0.0);
}

// Column j of the Hessenberg matrix, per column n: apply the earlier rotations,
// make rotation j, rotate g, keep the reduced column in R, and fold the new
// residual |g_{j+1}| / |r| into res (max over columns).
__global__ void k_gm_givens(int j, int ncol, int m, const double2* __restrict__ h, const double2* __restrict__ h2,
                            const double* __restrict__ nrm,
                            const double* __restrict__ bnorm, double* __restrict__ cs, double2* __restrict__ sn,
                            double2* __restrict__ g, double2* __restrict__ R, unsigned long long* __restrict__ res) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncol) return;
  const double2* h1c = h + (size_t)n * (m + 1);
  const double2* h2c = h2 + (size_t)n * (m + 1);
  auto hc = [&](int i) { return make_double2(h1c[i].x + h2c[i].x, h1c[i].y + h2c[i].y); };
  double* c_ = cs + (size_t)n * m;
  double2* s_ = sn + (size_t)n * m;
  double2* gn = g + (size_t)n * (m + 1);
  double2* Rn = R + (size_t)n * m * m;
  double2 col_i = hc(0);
  for (int i = 0; i < j; ++i) {
    const double2 next = hc(i + 1);
    // [a; b] <- [c a + s b; -conj(s) a + c b]
    const double2 a = col_i;
    const double2 top = make_double2(c_[i] * a.x + gm_mul(s_[i], next).x, c_[i] * a.y + gm_mul(s_[i], next).y);
    const double2 sa = gm_mul(gm_conj(s_[i]), a);
    col_i = make_double2(-sa.x + c_[i] * next.x, -sa.y + c_[i] * next.y);
    Rn[(size_t)i * m + j] = top;
  }
  const double2 a = col_i;                           // entry j after the earlier rotations
  const double bsub = sqrt(fmax(nrm[n], 0.0));       // h_{j+1,j}, real and non-negative
  const double aa = sqrt(a.x * a.x + a.y * a.y);
  double c, rr;
  double2 s, r;
  if (aa == 0.0) {
    c = 0.0;
    s = make_double2(1.0, 0.0);
    r = make_double2(bsub, 0.0);
  } else {
    rr = sqrt(aa * aa + bsub * bsub);
    c = aa / rr;
    s = make_double2(bsub * a.x / (rr * aa), bsub * a.y / (rr * aa));
    r = make_double2(a.x / aa * rr, a.y / aa * rr);
  }
  c_[j] = c;
  s_[j] = s;
  Rn[(size_t)j * m + j] = r;
  const double2 gj = gn[j];
  gn[j] = make_double2(c * gj.x, c * gj.y);
  const double2 t = gm_mul(gm_conj(s), gj);
  gn[j + 1] = make_double2(-t.x, -t.y);
  const double bn = bnorm[n];
  const double rel = bn > 0.0 ? sqrt(t.x * t.x + t.y * t.y) / bn : 0.0;
  atomicMax(res, (unsigned long long)__double_as_longlong(rel == rel ? rel : 1e300));
}

// y = R^{-1} g over the first d rows, per column
__global__ void k_gm_backsolve(int d, int ncol, int m, const double2* __restrict__ R, const double2* __restrict__ g,
                               double2* __restrict__ y) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncol) return;
  const double2* Rn = R + (size_t)n * m * m;
  const double2* gn = g + (size_t)n * (m + 1);
  double2* yn = y + (size_t)n * m;
  for (int i = d - 1; i >= 0; --i) {
    double2 acc = gn[i];
    for (int k = i + 1; k < d; ++k) {
      const double2 p = gm_mul(Rn[(size_t)i * m + k], yn[k]);
      acc.x -= p.x;
      acc.y -= p.y;
    }
    const double2 di = Rn[(size_t)i * m + i];
    const double den = di.x * di.x + di.y * di.y;
    yn[i] = den > 0.0 ? make_double2((acc.x * di.x + acc.y * di.y) / den, (acc.y * di.x - acc.x * di.y) / den)
                      : make_double2(0.0, 0.0);
  }
}

template <class T>
int gm_alloc(dyson_ctx* c, T** p, size_t count) {
  if (*p) cudaFree(*p);
  *p = nullptr;
  cudaError_t e = cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return ctx_fail(c, DYSON_ERR_OOM, std::string("GMRES buffers: ") + cudaGetErrorString(e));
  }
  return DYSON_OK;
}

// buffers for ncol columns of vsz floats and restart length m
int gm_prepare(dyson_ctx* c, size_t vsz, int ncol, int m) {
  GmState* st = gstate(c);
  if (st->vsz == vsz && st->ncol == ncol && st->m == m) return DYSON_OK;
  int rc;
  if ((rc = gm_alloc(c, &st->Q, (size_t)(m + 1) * vsz)) || (rc = gm_alloc(c, &st->zero, vsz)) ||
      (rc = gm_alloc(c, &st->u, vsz)) || (rc = gm_alloc(c, &st->w, vsz)) ||
      (rc = gm_alloc(c, &st->h, (size_t)ncol * (m + 1))) || (rc = gm_alloc(c, &st->h2, (size_t)ncol * (m + 1))) ||
      (rc = gm_alloc(c, &st->nrm, ncol)) || (rc = gm_alloc(c, &st->nrm0, ncol)) ||
      (rc = gm_alloc(c, &st->nrm1, ncol)) ||
      (rc = gm_alloc(c, &st->bnorm, ncol)) || (rc = gm_alloc(c, &st->beta, ncol)) ||
      (rc = gm_alloc(c, &st->cs, (size_t)ncol * m)) || (rc = gm_alloc(c, &st->sn, (size_t)ncol * m)) ||
      (rc = gm_alloc(c, &st->g, (size_t)ncol * (m + 1))) || (rc = gm_alloc(c, &st->R, (size_t)ncol * m * m)) ||
      (rc = gm_alloc(c, &st->y, (size_t)ncol * m)) || (rc = gm_alloc(c, &st->res, 1))) {
    st->vsz = 0;
    return rc;
  }
  if (!st->h_res) DY_CUDA(c, cudaMallocHost((void**)&st->h_res, sizeof(unsigned long long)));
  DY_CUDA(c, cudaMemsetAsync(st->zero, 0, vsz * sizeof(float), c->stream));
  st->vsz = vsz;
  st->ncol = ncol;
  st->m = m;
  return DYSON_OK;
}

}  // namespace

size_t gmres_bytes(const dyson_ctx* c) {
  const GmState* st = static_cast<const GmState*>(c->gm);
  return st ? (size_t)(st->m + 4) * st->vsz * sizeof(float) : 0;
}

int gmres_restart_length(dyson_ctx* c, int ncol) {
  const size_t vbytes = (size_t)c->Nr * ncol * 2 * c->Ns * sizeof(float);
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return 0;
  const double budget = 0.8 * (double)(free_b + gmres_bytes(c));
  const int fit = (int)(budget / (double)vbytes) - 4;
  return std::max(0, std::min(c->gmres_restart > 0 ? c->gmres_restart : 40, std::min(fit, 60)));
}

namespace {

// the vector kernels for one item shape
template <int VEC, int T>
int gmres_run(dyson_ctx* c, int ncol, const float* r, float* x, int max_iters, double tol, dyson_report* rep,
              const MatvecFn& matvec, int m) {
  GmState* st = gstate(c);
  cudaStream_t s = c->stream;
  const int Ns = c->Ns;                                  // (padding points are zeros)
  const size_t vsz = (size_t)c->Nr * ncol * 2 * Ns;
  int rc;
  // ranges of items per column: enough blocks for every SM, and at least two items per warp
  const int nz = (Ns + 32 * VEC * T - 1) / (32 * VEC * T), items = c->Nr * nz;
  const int want = std::max(1, std::min((items + 15) / 16, (152 * 16 + ncol - 1) / ncol));
  const int per = ((items + want - 1) / want + 7) / 8 * 8;   // (a block's eight warps take equally many)
  const dim3 grid(ncol, (items + per - 1) / per);
  const int cb = (ncol + 127) / 128;
  const int lin_grid = (int)std::min<size_t>((vsz + 255) / 256, 152 * 16);
  const size_t hbytes = (size_t)ncol * (m + 1) * sizeof(double2);

  // |r| per column, and the iterate starts at u0 = r
  DY_CUDA(c, cudaMemsetAsync(st->bnorm, 0, ncol * sizeof(double), s));
  k_gm_norm2<VEC, T><<<grid, GM_THREADS, 0, s>>>(r, items, nz, Ns, ncol, per, st->bnorm);
  k_gm_sqrt<<<cb, 128, 0, s>>>(st->bnorm, ncol);
  DY_CUDA(c, cudaMemcpyAsync(x, r, vsz * sizeof(float), cudaMemcpyDeviceToDevice, s));
  c->launches += 2;
  int its = 0;
  double rel = INFINITY;
  while (its < max_iters) {
    // residue of the iterate: z0 = r - (I - K) x = r - x + K x
    if ((rc = matvec(st->zero, x, st->u, 0.0))) return rc;
    rep->sweeps += 1;
    rep->gemm_flops += sweep_flops(c, ncol);
    k_gm_lin3<<<lin_grid, 256, 0, s>>>(r, x, st->u, st->w, vsz);
    DY_CUDA(c, cudaMemsetAsync(st->nrm, 0, ncol * sizeof(double), s));
    k_gm_norm2<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->w, items, nz, Ns, ncol, per, st->nrm);
    k_gm_start<<<cb, 128, 0, s>>>(ncol, m, st->nrm, st->beta, st->g);
    k_gm_scale<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->w, st->nrm, st->Q, items, nz, Ns, ncol, per);
    c->launches += 4;
    int d = 0;
    for (int j = 0; j < m && its < max_iters; ++j) {
      ++its;
      float* qj = st->Q + (size_t)j * vsz;
      // u = K q_j, so w = (I - K) q_j = q_j - u (|q_j| <= 1: every column has unit length)
      if ((rc = matvec(st->zero, qj, st->u, 1.0001))) return rc;
      rep->sweeps += 1;
      rep->gemm_flops += sweep_flops(c, ncol);
      // classical Gram-Schmidt: h = <Q, q_j - u>, w = q_j - u - Q h; then, for the
      // columns that lost most of their length, a second pass h2 = <Q, w>, w -= Q h2
      DY_CUDA(c, cudaMemsetAsync(st->h, 0, hbytes, s));
      DY_CUDA(c, cudaMemsetAsync(st->h2, 0, hbytes, s));
      DY_CUDA(c, cudaMemsetAsync(st->nrm0, 0, ncol * sizeof(double), s));
      DY_CUDA(c, cudaMemsetAsync(st->nrm1, 0, ncol * sizeof(double), s));
      DY_CUDA(c, cudaMemsetAsync(st->nrm, 0, ncol * sizeof(double), s));
      k_gm_dots<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->Q, vsz, j + 1, qj, st->u, items, nz, Ns, ncol, per, st->h,
                                                    m + 1, st->nrm0, nullptr, nullptr);
      k_gm_update<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->Q, vsz, j + 1, st->h, m + 1, -1.f, qj, st->u, st->w, items,
                                                      nz, Ns, ncol, per, st->nrm1, nullptr, nullptr);
      k_gm_dots<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->Q, vsz, j + 1, st->w, nullptr, items, nz, Ns, ncol, per,
                                                    st->h2, m + 1, nullptr, st->nrm1, st->nrm0);
      k_gm_update<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->Q, vsz, j + 1, st->h2, m + 1, -1.f, st->w, nullptr, st->w,
                                                      items, nz, Ns, ncol, per, st->nrm, st->nrm1, st->nrm0);
      k_gm_scale<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->w, st->nrm, st->Q + (size_t)(j + 1) * vsz, items, nz, Ns,
                                                     ncol, per);
      DY_CUDA(c, cudaMemsetAsync(st->res, 0, sizeof(unsigned long long), s));
      k_gm_givens<<<cb, 128, 0, s>>>(j, ncol, m, st->h, st->h2, st->nrm, st->bnorm, st->cs, st->sn, st->g, st->R,
                                     st->res);
      DY_CUDA(c, cudaMemcpyAsync(st->h_res, st->res, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
      DY_CUDA(c, cudaGetLastError());
      DY_CUDA(c, cudaStreamSynchronize(s));
      c->host_syncs += 1;
      flush_timers(c);
      c->launches += 6;
      d = j + 1;
      rel = bits_to_double(*st->h_res);
      rep->update = rel;
      if (!(rel < kDivergedGrowth)) return ctx_fail(c, DYSON_ERR_DIVERGED, "GMRES residual not finite");
      if (rel <= tol) break;
    }
    // x += Q_d y,  y = R^{-1} g
    k_gm_backsolve<<<cb, 128, 0, s>>>(d, ncol, m, st->R, st->g, st->y);
    k_gm_update<VEC, T><<<grid, GM_THREADS, 0, s>>>(st->Q, vsz, d, st->y, m, 1.f, x, nullptr, x, items, nz, Ns, ncol,
                                                    per, nullptr, nullptr, nullptr);
    c->launches += 2;
    DY_CUDA(c, cudaGetLastError());
    if (rel <= tol) break;
  }
  return DYSON_OK;
}

}  // namespace

int gmres_inner_solve(dyson_ctx* c, int ncol, const float* r, float* x, int max_iters, double tol,
                      dyson_report* rep, const MatvecFn& matvec) {
  if (ncol > 65535 || c->Nr > 65535) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "GMRES chunks hold <= 65535 columns");
  const int m = gmres_restart_length(c, ncol);
  if (m < 2) return ctx_fail(c, DYSON_ERR_OOM, "GMRES needs room for at least 3 Krylov vectors");
  const size_t vsz = (size_t)c->Nr * ncol * 2 * c->Ns;
  int rc = gm_prepare(c, vsz, ncol, m);
  if (rc) return rc;
  // float4 items where every column's halves are 16-byte aligned (the tensor-core sweeps' stride is a
  // multiple of 64; the CUDA-core sweep's is Nc)
  if (c->Ns % 4 != 0) return gmres_run<1, 1>(c, ncol, r, x, max_iters, tol, rep, matvec, m);
  const int t = (c->Ns + 127) / 128;                     // float4 per lane and part that cover a column
  if (t == 1) return gmres_run<4, 1>(c, ncol, r, x, max_iters, tol, rep, matvec, m);
  if (t % 3 == 0) return gmres_run<4, 3>(c, ncol, r, x, max_iters, tol, rep, matvec, m);
  return gmres_run<4, 2>(c, ncol, r, x, max_iters, tol, rep, matvec, m);
}

void gmres_release(dyson_ctx* c) {
  GmState* st = static_cast<GmState*>(c->gm);
  if (!st) return;
  void* ptrs[] = {st->Q, st->zero, st->u, st->w, st->h, st->h2, st->nrm, st->nrm0, st->nrm1, st->bnorm, st->beta,
                  st->cs, st->sn, st->g, st->R, st->y, st->res};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (st->h_res) cudaFreeHost(st->h_res);
  delete st;
  c->gm = nullptr;
}
