// Entry points of the C ABI declared in include/dyson.h.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <limits>

#include "common.cuh"
#include "detail.cuh"
#include "gmres.cuh"
#include "oz.cuh"
#include "oz64.cuh"
#include "ptx.cuh"
#include "symmetry.cuh"
#include "tc.cuh"

namespace dyson_detail {

thread_local std::string g_noctx_err;

int fail_noctx(int code, const std::string& m) {
  g_noctx_err = m;
  return code;
}

template <class T>
cudaError_t dalloc(T** p, size_t count) {
  return cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T));
}

double bits_to_double(unsigned long long b) {
  double d;
  std::memcpy(&d, &b, sizeof d);
  return d;
}

// -------------------------------------------------------------------------
void flush_timers(dyson_ctx* c) {
  for (auto& p : c->pending) {
    float ms = 0.f;
    if (cudaEventSynchronize(p.b) == cudaSuccess && cudaEventElapsedTime(&ms, p.a, p.b) == cudaSuccess) {
      c->prof_ms[p.kind] += ms;
      c->prof_launches[p.kind] += 1;
    }
    cudaEventDestroy(p.a);
    cudaEventDestroy(p.b);
  }
  c->pending.clear();
}

int ensure_work(dyson_ctx* c, size_t bytes) {
  if (c->work_bytes >= bytes) return DYSON_OK;
  if (c->work) cudaFree(c->work);
  c->work = nullptr;
  c->work_bytes = 0;
  cudaError_t e = cudaMalloc(&c->work, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return ctx_fail(c, DYSON_ERR_OOM, "work buffer of " + std::to_string(bytes) + " bytes: " + cudaGetErrorString(e));
  }
  c->work_bytes = bytes;
  return DYSON_OK;
}

// per-vector-column source arrays (ncol entries) and per-group norm/scale words (ng groups)
int ensure_cols(dyson_ctx* c, int ncol, int ng) {
  if (c->src_cap < ncol) {
    if (c->d_src_site) cudaFree(c->d_src_site);
    if (c->d_src_time) cudaFree(c->d_src_time);
    c->d_src_site = c->d_src_time = nullptr;
    c->src_cap = 0;
    DY_CUDA(c, dalloc(&c->d_src_site, ncol));
    DY_CUDA(c, dalloc(&c->d_src_time, ncol));
    c->src_cap = ncol;
  }
  if (c->norm_cap < ng) {
    if (c->d_norm) cudaFree(c->d_norm);
    if (c->h_norm) cudaFreeHost(c->h_norm);
    c->d_norm = nullptr;
    c->h_norm = nullptr;
    c->norm_cap = 0;
    if (c->d_xscale) cudaFree(c->d_xscale);
    if (c->d_rref) cudaFree(c->d_rref);
    c->d_xscale = nullptr;
    c->d_rref = nullptr;
    DY_CUDA(c, dalloc(&c->d_norm, 2 * (size_t)ng));
    DY_CUDA(c, dalloc(&c->d_xscale, ng));
    DY_CUDA(c, dalloc(&c->d_rref, ng));
    DY_CUDA(c, cudaMallocHost((void**)&c->h_norm, 2 * (size_t)ng * sizeof(unsigned long long)));
    c->norm_cap = ng;
  }
  return DYSON_OK;
}

// copy the host source arrays of the current chunk to the device
int upload_sources(dyson_ctx* c, int ncol) {
  DY_CUDA(c, cudaMemcpyAsync(c->d_src_site, c->h_src_site.data(), ncol * sizeof(int), cudaMemcpyHostToDevice,
                             c->stream));
  DY_CUDA(c, cudaMemcpyAsync(c->d_src_time, c->h_src_time.data(), ncol * sizeof(int), cudaMemcpyHostToDevice,
                             c->stream));
  return DYSON_OK;
}

// read norm[0..ng) (and scale[ng..2ng) when with_scale) to the host
int read_norms(dyson_ctx* c, int ng, bool with_scale) {
  DY_CUDA(c, cudaMemcpyAsync(c->h_norm, c->d_norm, (with_scale ? 2 : 1) * (size_t)ng * sizeof(unsigned long long),
                             cudaMemcpyDeviceToHost, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  c->host_syncs += 1;
  flush_timers(c);
  return DYSON_OK;
}

// max over groups of norm[q] / ref[q] (groups with ref = 0 hold only padding columns)
double rel_max(const unsigned long long* norm, const double* ref, int ng) {
  double m = 0.0;
  for (int q = 0; q < ng; ++q) {
    double v = bits_to_double(norm[q]) / std::max(ref[q], 1e-300);
    if (!(v == v)) return std::numeric_limits<double>::infinity();
    m = std::max(m, v);
  }
  return m;
}


// algorithmic contour-GEMM flops of one sweep over ncol vector columns
double sweep_flops(const dyson_ctx* c, int ncol) { return 8.0 * c->Nc * (double)c->Nc * c->Nr * ncol; }

// After one FP64 sweep: the update max_q norm_q / scale_q to the host, and whether the series goes on, with
// the host loop's rule; norm words cleared for the next sweep.  One warp.
__global__ void k_f64_check(unsigned long long* __restrict__ norm, const unsigned long long* __restrict__ scale, int ng,
                            double tol, double* __restrict__ upd, int* __restrict__ run) {
  ptx::grid_launch_next();
  ptx::grid_wait();
  if (!*(volatile int*)run) return;
  double m = 0.0;
  int bad = 0;
  for (int q = threadIdx.x; q < ng; q += 32) {
    const double v = __longlong_as_double((long long)norm[q]) / fmax(__longlong_as_double((long long)scale[q]), 1e-300);
    if (!(v == v)) bad = 1;
    else m = fmax(m, v);
    norm[q] = 0ull;
  }
  for (int o = 16; o > 0; o >>= 1) {
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (threadIdx.x != 0) return;
  if (bad) m = __longlong_as_double(0x7ff0000000000000ll);
  *upd = m;
  if (!(m < kDivergedF64) || m <= tol) *run = 0;
}

int prepare_f64_series(dyson_ctx* c) {
  if (!c->d_f64_run) DY_CUDA(c, cudaMalloc((void**)&c->d_f64_run, sizeof(int)));
  if (!c->h_f64_upd) DY_CUDA(c, cudaMallocHost((void**)&c->h_f64_upd, kF64Ahead * sizeof(double)));
  for (cudaEvent_t& e : c->f64_ev)
    if (!e) DY_CUDA(c, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  return DYSON_OK;
}

// Plain FP64 series over the chunk (ncol vector columns, norm groups of gs columns):
// G <- B + K G until the relative update <= tol.
// Up to kF64Ahead sweeps are enqueued before the first one's update has reached the host; those behind
// the last one find the series stopped and return at once (its result is in the other buffer).  Their
// launches overlap (launch_overlapped).  4x4, Nc = 64, 29 sweeps of 49 us: 2.07 ms with a synchronisation after
// each sweep (20 us of idle GPU), 1.79 enqueued ahead, 1.60 overlapped; 3x3, Nc = 26: 1.33, 1.04, 0.85.
// A profiled series and the FP64-pipe sweep, which does not read the flag, wait for each sweep.
int solve_f64(dyson_ctx* c, int ncol, int gs, double tol, int max_sweeps, double2** result, dyson_report* r) {
  const int ng = ncol / gs;
  const size_t n_el = (size_t)c->Nr * ncol * c->Nc;
  double2* Ga = (double2*)c->work;
  double2* Gb = Ga + n_el;
  DY_CUDA(c, cudaMemsetAsync(Ga, 0, n_el * sizeof(double2), c->stream));
  DY_CUDA(c, cudaMemsetAsync(c->d_norm, 0, 2 * (size_t)ng * sizeof(unsigned long long), c->stream));
  launch_init_rhs(c->d_lam, c->d_src_site, c->d_src_time, c->Nr, c->Nc, ncol, gs, Ga, c->d_norm + ng, c->stream);
  c->launches += 1;
  int rc = prepare_f64_series(c);
  if (rc) return rc;
  DY_CUDA(c, cudaMemsetAsync(c->d_f64_run, 1, sizeof(int), c->stream));   // (any non-zero value)
  *result = Ga;
  const int ahead = c->use_oz64 && !c->profiling ? kF64Ahead : 1;
  int enqueued = 0;
  auto enqueue = [&]() -> int {
    {
      KernelTimer t(c, DYSON_KERNEL_SWEEP_F64);
      if (c->use_oz64) {
        if ((rc = oz64_sweep(c, ncol, gs, Ga, Gb, nullptr, 0, c->d_f64_run))) return rc;
      } else {
        launch_sweep_f64(c->d_lam, c->d_JW, c->d_nbr, c->d_nbond, Ga, Gb, nullptr, c->Nc, c->d_src_site, c->d_src_time,
                         c->Nr, c->Nc, ncol, gs, 0, c->d_norm, c->stream);
        c->launches += 1;
      }
    }
    DY_CUDA(c, launch_overlapped(true, k_f64_check, 1, 32, 0, c->stream, c->d_norm, c->d_norm + ng, ng, tol,
                                 c->h_f64_upd + enqueued % kF64Ahead, c->d_f64_run));
    c->launches += 1;
    DY_CUDA(c, cudaEventRecord(c->f64_ev[enqueued % kF64Ahead], c->stream));
    std::swap(Ga, Gb);
    ++enqueued;
    return DYSON_OK;
  };
  int status = DYSON_ERR_NOT_CONVERGED;
  for (int done = 0; done < max_sweeps; ++done) {
    while (enqueued < max_sweeps && enqueued - done < ahead)
      if ((rc = enqueue())) return rc;
    DY_CUDA(c, cudaEventSynchronize(c->f64_ev[done % kF64Ahead]));
    c->host_syncs += 1;
    flush_timers(c);
    const double upd = *static_cast<volatile double*>(c->h_f64_upd + done % kF64Ahead);
    *result = (enqueued - done) % 2 ? Ga : Gb;             // the output of sweep done + 1
    r->sweeps += 1;
    r->gemm_flops += sweep_flops(c, ncol);
    r->update = upd;
    if (!(upd < kDivergedF64)) {
      if (c->use_oz64 && (rc = oz64_check_error(c))) return rc;
      status = DYSON_ERR_DIVERGED;
      break;
    }
    if (upd <= tol) {
      status = DYSON_OK;
      break;
    }
  }
  return status;
}

// After one sweep of a batch: the update max_q norm_q / rref_q (norm words
// cleared for the next sweep), the next sweep's FP16 scales, and the stopping rule (series_step).
// One warp; returns at once once the series has stopped.
__global__ void k_series_check(unsigned long long* __restrict__ norm, const double* __restrict__ rref, int ng,
                               int max_sweeps, double target, double abort_peak, SeriesState* __restrict__ S,
                               TcScale* __restrict__ xscale, float jbound) {
  ptx::grid_launch_next();
  ptx::grid_wait();
  if (!*(volatile int*)&S->run) return;
  for (int q = threadIdx.x; q < ng; q += 32) set_scale(xscale + q, __uint_as_float(xscale[q].ymax), jbound);
  double m = 0.0;
  int bad = 0;
  for (int q = threadIdx.x; q < ng; q += 32) {
    const double v = __longlong_as_double((long long)norm[q]) / fmax(rref[q], 1e-300);
    if (!(v == v)) bad = 1;
    else m = fmax(m, v);
    norm[q] = 0ull;
  }
  for (int o = 16; o > 0; o >>= 1) {
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (threadIdx.x != 0) return;
  series_step(*S, bad ? __longlong_as_double(0x7ff0000000000000ll) : m, max_sweeps, target, abort_peak);
}

// kind that the fused sweep is timed as: its own where the context selected it, the general
// tensor-core sweep where it runs as the default
int fused_kind(const dyson_ctx* c) {
  return c->tc_variant == DYSON_SWEEP_FUSED_PAIR || c->tc_variant == DYSON_SWEEP_FUSED_PAIR_WIDE
             ? DYSON_KERNEL_SWEEP_TC_FUSED
             : DYSON_KERNEL_SWEEP_TC;
}

// one tensor-core sweep dout = r + K din with per-kind event timing: the
// fused gather + GEMM launch, or the gather launch and the GEMM launch
int tc_timed_sweep(dyson_ctx* c, int ncol, int gs, const float* r, const float* din, float* dout, const int* act,
                   int sweep, int rform = TC_R_DENSE) {
  if (tc_uses_fused(c)) {
    KernelTimer t(c, fused_kind(c));
    return tc_sweep(c, ncol, gs, r, din, dout, TC_GATHER | TC_GEMM, act, sweep, rform);
  }
  int rc;
  {
    KernelTimer t(c, DYSON_KERNEL_GATHER_TC);
    if ((rc = tc_sweep(c, ncol, gs, r, din, dout, TC_GATHER, act, sweep))) return rc;
  }
  KernelTimer t(c, tc_uses_pair(c) && !act ? DYSON_KERNEL_SWEEP_TC_PAIR : DYSON_KERNEL_SWEEP_TC);
  return tc_sweep(c, ncol, gs, r, din, dout, TC_GEMM, act, sweep);
}

// the series starts from d = r: its scales come from the reference norms max|r| (c->d_rref)
int seed_series(dyson_ctx* c, const std::vector<double>& rref) {
  DY_CUDA(c, cudaMemcpyAsync(c->d_rref, rref.data(), rref.size() * sizeof(double), cudaMemcpyHostToDevice,
                             c->stream));                  // pageable: complete when the call returns
  return tc_seed_scale(c, (int)rref.size(), c->d_rref, 0.0);
}

// Start of a series on the fused sweep, da already holding r and the scales seeded.
int SeriesRun::begin(bool plateau) {
  if (!c->d_series) {
    DY_CUDA(c, cudaMalloc(&c->d_series, sizeof(SeriesState)));
    DY_CUDA(c, cudaMallocHost(&c->h_series, sizeof(SeriesState)));
  }
  SeriesState* hS = static_cast<SeriesState*>(c->h_series);
  *hS = series_start(plateau);
  int rc;
  if ((rc = tc_prepare_sweep(c, ncol, true)) || (rc = tc_set_scale(c, ncol / gs))) return rc;
  DY_CUDA(c, cudaMemcpyAsync(c->d_series, hS, sizeof(SeriesState), cudaMemcpyHostToDevice, c->stream));
  DY_CUDA(c, cudaMemsetAsync(c->d_norm, 0, (size_t)(ncol / gs) * sizeof(unsigned long long), c->stream));
  return DYSON_OK;
}

const SeriesState* SeriesRun::state() const { return static_cast<const SeriesState*>(c->h_series); }
bool SeriesRun::running() const { return state()->run != 0; }

// `sweeps` sweeps (even, so that every batch starts from da), each followed by its check, on the context's
// stream, and the copies of the series' state and of the error flag behind them.
int SeriesRun::enqueue(bool overlap) {
  SeriesState* dS = static_cast<SeriesState*>(c->d_series);
  int rc;
  for (int k = 0; k < sweeps; ++k) {
    c->overlap = overlap && k > 0;
    rc = tc_fused_sweep(c, ncol, gs, r32, k % 2 ? db : da, k % 2 ? da : db, act, 0, rform, &dS->run, &dS->sweeps, c->stream);
    c->overlap = false;
    if (rc) return rc;
    DY_CUDA(c, launch_overlapped(overlap, k_series_check, 1, 32, 0, c->stream, c->d_norm, c->d_rref, ncol / gs, max_sweeps,
                                 target, abort_peak, dS, c->d_xscale, tc_jbound(c)));
    c->launches += 1;
  }
  before = state()->sweeps;
  if ((rc = tc_error_enqueue(c))) return rc;
  DY_CUDA(c, cudaMemcpyAsync(c->h_series, dS, sizeof(SeriesState), cudaMemcpyDeviceToHost, c->stream));
  return DYSON_OK;
}

// After the stream has been waited for: sweeps that ran; da: the state that the last one left.
int SeriesRun::collect(int* rc) {
  if ((*rc = tc_error_status(c))) return 0;
  const int n_run = state()->sweeps - before;
  rep->sweeps += n_run;
  rep->gemm_flops += n_run * sweep_flops(c, ncol);
  rep->update = state()->last;
  if (!running() && n_run % 2) std::swap(da, db);          // the last sweep wrote db
  return n_run;
}

// inner solve d <- r + K d in FP32 (SIMT or 3xTF32 tensor cores)
// act (optional): support truncation of the tensor-core sweeps (tc_sweep), valid
// while every column of r32 is zero off its source site
// r_on_sources: r32 is non-zero only on each column's source site (the first right-hand side)
// With the fused sweep, c->graph_sweeps sweeps at a time are enqueued, each followed by k_series_check: one
// host synchronisation per batch instead of one per sweep.  These sweeps take their sweep number (for the
// support table) from the device count of sweeps done.  The launches overlap (launch_overlapped): a
// sweep's CTAs set up under the check before it.  As replays of a captured graph, whose capture and
// instantiation every inner solve paid for: 8x8, Nc = 128, 6.58 ms a solve, 9x7, Nc = 100, 4.46; so 6.52 and
// 4.33 (enqueued without the overlap 6.88 and 4.56).
int inner_solve(dyson_ctx* c, int ncol, int gs, int precision, float* r32, float* da, float* db, int max_sweeps,
                const std::vector<double>& rref, float** dres, dyson_report* rep, double abort_peak, const int* act,
                int* outcome, double target, bool r_on_sources, bool plateau) {
  const int ng = ncol / gs;
  const size_t n32 = (size_t)c->Nr * ncol * 2 * c->Ns;
  DY_CUDA(c, cudaMemcpyAsync(da, r32, n32 * sizeof(float), cudaMemcpyDeviceToDevice, c->stream));
  if (act) DY_CUDA(c, cudaMemsetAsync(db, 0, n32 * sizeof(float), c->stream));   // skipped tiles stay 0
  const int rform = r_on_sources ? TC_R_ON_SOURCES : TC_R_DENSE;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  // (not inside a caller's own capture of the stream)
  const bool batches = c->graph_sweeps > 0 && precision == DYSON_PREC_TF32X3_F64REF && c->use_tc &&
                     tc_uses_fused(c) && cudaStreamIsCapturing(c->stream, &cap) == cudaSuccess &&
                     cap == cudaStreamCaptureStatusNone;
  const int eager_until = batches ? 0 : max_sweeps;
  SeriesState S = series_start(plateau);
  int rc;
  if (precision == DYSON_PREC_TF32X3_F64REF && c->use_tc && tc_uses_fused(c) && (rc = seed_series(c, rref))) return rc;
  while (S.run && S.sweeps < std::min(max_sweeps, eager_until)) {
    const int sweep = S.sweeps + 1;
    DY_CUDA(c, cudaMemsetAsync(c->d_norm, 0, (size_t)ng * sizeof(unsigned long long), c->stream));
    if (precision == DYSON_PREC_TF32X3_F64REF && c->use_tc) {
      if ((rc = tc_timed_sweep(c, ncol, gs, r32, da, db, act, sweep, rform))) return rc;
    } else {
      KernelTimer t(c, DYSON_KERNEL_SWEEP_F32);
      launch_sweep_f32_simt(c->d_lam32, c->d_Jz, contour_stride(c), c->d_nbr, c->d_nbond, r32, da, db, c->Nr, c->Nc, ncol, gs,
                            c->d_norm, c->stream);
      c->launches += 1;
    }
    DY_CUDA(c, cudaGetLastError());
    // one synchronisation per sweep: the norms and the pipeline's error flag come back together
    if (c->use_tc && (rc = tc_error_enqueue(c))) return rc;
    if ((rc = read_norms(c, ng, false))) return rc;
    if (c->use_tc && (rc = tc_error_status(c))) return rc;
    std::swap(da, db);
    const double upd = rel_max(c->h_norm, rref.data(), ng);
    rep->sweeps += 1;
    rep->gemm_flops += sweep_flops(c, ncol);
    rep->update = upd;
    series_step(S, upd, max_sweeps, target, abort_peak);
  }
  if (S.run && batches) {
    SeriesRun run{c, ncol, gs, max_sweeps, c->graph_sweeps, r32, da, db, act, rform, target, abort_peak, rep};
    if ((rc = run.begin(plateau))) return rc;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (c->profiling) {
      cudaEventCreate(&e0);
      cudaEventCreate(&e1);
    }
    while (rc == DYSON_OK && run.running()) {
      if (e0) cudaEventRecord(e0, c->stream);
      rc = run.enqueue(true);
      if (e1) cudaEventRecord(e1, c->stream);
      if (rc) break;
      const cudaError_t e = cudaStreamSynchronize(c->stream);
      if (e != cudaSuccess) rc = ctx_fail(c, DYSON_ERR_CUDA, std::string("inner series: ") + cudaGetErrorString(e));
      c->host_syncs += 1;
      const int n_run = rc ? 0 : run.collect(&rc);
      float ms = 0.f;
      if (e0 && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess) {
        c->prof_ms[fused_kind(c)] += ms;                   // the batch, its checks included
        c->prof_launches[fused_kind(c)] += n_run;
      }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (rc) return rc;
    S = *run.state();
    da = run.da;
  }
  if (outcome) *outcome = S.outcome;
  if (S.outcome == SERIES_NOT_FINITE) return ctx_fail(c, DYSON_ERR_DIVERGED, "FP32 series update not finite");
  if (S.outcome == SERIES_ABORTED) return DYSON_ERR_DIVERGED;   // the caller switches to GMRES
  *dres = da;
  return DYSON_OK;
}

// out = zero + K in: one FP32 sweep with a zero right-hand side (the GMRES matvec);
// bound: an upper bound of |in|, or 0 to read it from the state
int matvec_f32(dyson_ctx* c, int ncol, int gs, int precision, const float* zero, const float* in, float* out,
               double bound) {
  int rc;
  if (precision == DYSON_PREC_TF32X3_F64REF && c->use_tc) {
    if (tc_uses_fused(c) &&
        (rc = bound > 0.0 ? tc_seed_scale(c, ncol / gs, nullptr, bound) : tc_seed_scale_scan(c, ncol, gs, in)))
      return rc;
    if ((rc = tc_timed_sweep(c, ncol, gs, zero, in, out, nullptr, 0, TC_R_ZERO))) return rc;
  } else {
    KernelTimer t(c, DYSON_KERNEL_SWEEP_F32);
    launch_sweep_f32_simt(c->d_lam32, c->d_Jz, contour_stride(c), c->d_nbr, c->d_nbond, zero, in, out, c->Nr, c->Nc, ncol, gs,
                          c->d_norm, c->stream);
    c->launches += 1;
  }
  DY_CUDA(c, cudaGetLastError());
  return DYSON_OK;
}

// Support truncation (Sec. IV.D): the first right-hand
// side Lambda delta_s is non-zero only on the source site of each column, and a
// sweep spreads an iterate by one hop, so after n sweeps a column is zero beyond
// lattice distance n of its source.  act[i][t] = min over the columns of 256-column
// tile t of the distance from site i to the column's source: the first sweep at
// which the tile can be non-zero.  Uploaded to c->d_act; nullptr when it cannot help.
const int* support_table(dyson_ctx* c, int ncol) {
  const int NT = (ncol + TC_TILE_COLS - 1) / TC_TILE_COLS;
  std::vector<int> act((size_t)c->Nr * NT, std::numeric_limits<int>::max());
  int far = 0;
  for (int t = 0; t < NT; ++t) {
    const int v1 = std::min(ncol, (t + 1) * TC_TILE_COLS);
    int last = -1;
    for (int v = t * TC_TILE_COLS; v < v1; ++v) {
      const int s = c->h_src_site[v];
      if (s == last || s < 0) continue;                  // padding columns (site -1) stay zero
      last = s;
      const int sx = s % c->Lx, sy = s / c->Lx;
      for (int i = 0; i < c->Nr; ++i) {
        const int d = std::abs(i % c->Lx - sx) + std::abs(i / c->Lx - sy);
        int& a = act[(size_t)i * NT + t];
        a = std::min(a, d);
      }
    }
  }
  for (int a : act) far = std::max(far, a);
  if (far < 2) return nullptr;                           // every tile is live from the first sweeps
  const size_t bytes = act.size() * sizeof(int);
  if (c->act_bytes < bytes) {
    if (c->d_act) cudaFree(c->d_act);
    c->d_act = nullptr;
    c->act_bytes = 0;
    if (cudaMalloc(&c->d_act, bytes) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;                                    // optional: run untruncated
    }
    c->act_bytes = bytes;
  }
  // pageable source: the copy completes before the call returns
  if (cudaMemcpyAsync(c->d_act, act.data(), bytes, cudaMemcpyHostToDevice, c->stream) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return c->d_act;
}

// complex FP32 series refined by FP64 residuals: G += solve(r), r = B + K G - G
int solve_mixed(dyson_ctx* c, int ncol, int gs, int precision, double tol, int max_sweeps, double2** result,
                dyson_report* rep) {
  const int ng = ncol / gs;
  const size_t n_el = (size_t)c->Nr * ncol * c->Nc, n32 = (size_t)c->Nr * ncol * 2 * c->Ns;
  double2* G = (double2*)c->work;
  float* r32 = (float*)(G + n_el);
  float* da = r32 + n32;
  float* db = da + n32;
  int rc;
  // r = B (FP32), scale = max |B| per group; G = 0
  DY_CUDA(c, cudaMemsetAsync(G, 0, n_el * sizeof(double2), c->stream));
  DY_CUDA(c, cudaMemsetAsync(c->d_norm, 0, 2 * (size_t)ng * sizeof(unsigned long long), c->stream));
  launch_init_rhs(c->d_lam, c->d_src_site, c->d_src_time, c->Nr, c->Nc, ncol, gs, G, c->d_norm + ng, c->stream);
  launch_to_planar32(G, r32, (size_t)c->Nr * ncol, c->Nc, c->Ns, c->stream);
  c->launches += 2;
  DY_CUDA(c, cudaMemsetAsync(G, 0, n_el * sizeof(double2), c->stream));
  if ((rc = read_norms(c, ng, true))) return rc;
  std::vector<double> scale(ng), rref(ng);
  for (int q = 0; q < ng; ++q) rref[q] = scale[q] = bits_to_double(c->h_norm[ng + q]);
  // the caller reads the chunk state (observables, export) whatever the status
  *result = G;
  int status = DYSON_ERR_NOT_CONVERGED;
  double prev_res = std::numeric_limits<double>::infinity();
  int strikes = 0;
  // inner solver: the series of App. C, or its GMRES.  AUTO starts with the series
  // and switches to GMRES for the rest of the chunk when the series cannot serve:
  // it diverges, its transient peak times the FP32 rounding leaves no correct
  // digit, it uses its whole sweep budget, it ends on a plateau without gaining a digit, or the refined
  // residual grows.
  bool gmres = c->inner_solver == DYSON_INNER_GMRES, plateau = true;
  const bool may_switch = c->inner_solver == DYSON_INNER_AUTO;
  const MatvecFn mv = [&](const float* zero, const float* in, float* out, double bound) {
    return matvec_f32(c, ncol, gs, precision, zero, in, out, bound);
  };
  for (int ref = 0; ref < c->max_refinements; ++ref) {
    float* d = nullptr;
    int outcome = SERIES_RUNNING;
    if (gmres) {
      rc = gmres_inner_solve(c, ncol, r32, da, max_sweeps, inner_target(kGmresTarget, tol, prev_res), rep, mv);
      d = da;
      rep->inner_gmres = 1;
    } else {
      // the first right-hand side lives on the source sites: truncate its sweeps
      const int* act = ref == 0 && c->support_trunc && c->use_tc && precision == DYSON_PREC_TF32X3_F64REF
                           ? support_table(c, ncol)
                           : nullptr;
      rc = inner_solve(c, ncol, gs, precision, r32, da, db, max_sweeps, rref, &d, rep,
                       may_switch ? kSeriesPeakMax : std::numeric_limits<double>::infinity(), act, &outcome,
                       inner_target(kInnerTarget, tol, prev_res), ref == 0, plateau);
      if (rc == DYSON_ERR_DIVERGED && may_switch && !(prev_res <= tol)) {
        gmres = true;                                    // redo this refinement with GMRES
        --ref;
        continue;
      }
      // a series that used its whole sweep budget converges too slowly (spectral radius
      // near 1): its correction is kept, the following refinements use GMRES
      if (rc == DYSON_OK && outcome == SERIES_EXHAUSTED && may_switch) gmres = true;
    }
    if (rc == DYSON_ERR_DIVERGED) {
      status = prev_res <= tol ? DYSON_OK : rc;            // (the refinement beyond the tolerance adds nothing)
      break;
    }
    if (rc) return rc;
    launch_accumulate(G, d, c->Nr, c->Nc, c->Ns, ncol, c->stream);
    c->launches += 1;
    DY_CUDA(c, cudaMemsetAsync(c->d_norm, 0, (size_t)ng * sizeof(unsigned long long), c->stream));
    if ((rc = enqueue_residual(c, ncol, gs, G, r32))) return rc;
    if (c->use_oz && (rc = oz_error_enqueue(c))) return rc;   // read with the norms: one synchronisation
    if ((rc = read_norms(c, ng, false))) return rc;
    if (c->use_oz && (rc = oz_error_status(c))) return rc;
    rep->refinements += 1;
    rep->gemm_flops += sweep_flops(c, ncol);
    double res = rel_max(c->h_norm, scale.data(), ng);
    rep->residual = res;
    for (int q = 0; q < ng; ++q) rref[q] = std::max(bits_to_double(c->h_norm[q]), 1e-300);
    if (!(res < kDivergedGrowth)) {
      if (c->use_oz64 && (rc = oz64_check_error(c))) return rc;
      status = DYSON_ERR_DIVERGED;
      break;
    }
    if (res <= tol && !refine_once_more(res, tol, prev_res, c->accept, ref + 1 == c->max_refinements)) {
      status = DYSON_OK;
      break;
    }
    if (outcome == SERIES_PLATEAU && !plateau_served(res, prev_res)) {
      plateau = false;
      if (may_switch) gmres = true;
    }
    if (res > tol && res > kRefineContract * prev_res) {
      if (may_switch && !gmres) {
        gmres = true;                                    // the series does not contract: use GMRES
      } else if (++strikes >= kRefineStrikes) {
        status = DYSON_ERR_DIVERGED;
        break;
      }
    }
    prev_res = res;
  }
  return status;
}

}  // namespace dyson_detail

using namespace dyson_detail;

int ctx_fail(dyson_ctx* c, int code, const std::string& msg) {
  if (c) c->err = msg;
  else g_noctx_err = msg;
  return code;
}

extern "C" {

const char* dyson_version(void) { return "gb300-dyson 0.1 (sm_103a)"; }

const char* dyson_last_error(const dyson_ctx* ctx) { return ctx ? ctx->err.c_str() : g_noctx_err.c_str(); }

int dyson_init(dyson_ctx** out, const dyson_lattice* L, const dyson_contour* C, const dyson_trap* T,
               const dyson_drive* D, int device, void* stream) {
  if (!out) return fail_noctx(DYSON_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!L || !C || !T || !D || !D->U || !D->J) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL argument");
  if (L->Lx < 1 || L->Ly < 1 || (int64_t)L->Lx * L->Ly > 65535)
    return fail_noctx(DYSON_ERR_INVALID_ARG, "lattice must have 1..65535 sites");
  if (C->Nt < 1 || C->Nm < 1 || 2 * (int64_t)C->Nt + C->Nm > 2048)
    return fail_noctx(DYSON_ERR_INVALID_ARG, "need Nt >= 1, Nm >= 1 and 2*Nt+Nm <= 2048");
  if (!(C->dt > 0) || !(C->beta > 0) || !std::isfinite(C->dt) || !std::isfinite(C->beta))
    return fail_noctx(DYSON_ERR_INVALID_ARG, "dt and beta must be positive and finite");
  if (!std::isfinite(T->curvature) || !std::isfinite(T->mu))
    return fail_noctx(DYSON_ERR_INVALID_ARG, "trap parameters must be finite");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev)
    return fail_noctx(DYSON_ERR_INVALID_ARG, "no such CUDA device");
  DeviceGuard g(device);
  // commit the allocation-free entry point's static scratch on this device now, not at
  // its first call (lazy module loading); optional, so a failure only clears the error
  if (noalloc_reserve_scratch(device) != DYSON_OK) cudaGetLastError();
  auto* c = new dyson_ctx;
  c->device = device;
  c->stream = (cudaStream_t)stream;
  c->Lx = L->Lx;
  c->Ly = L->Ly;
  c->Nr = L->Lx * L->Ly;
  c->Nb = L->Ly * (L->Lx - 1) + L->Lx * (L->Ly - 1);
  c->Nt = C->Nt;
  c->Nm = C->Nm;
  c->Nc = 2 * C->Nt + C->Nm;
  c->dt = C->dt;
  c->beta = C->beta;
  c->curvature = T->curvature;
  c->mu = T->mu;
  c->U.assign(D->U, D->U + (size_t)c->Nr * c->Nt);
  c->J.assign(D->J, D->J + (size_t)c->Nb * c->Nt);
  for (double v : c->U)
    if (!std::isfinite(v)) {
      delete c;
      return fail_noctx(DYSON_ERR_INVALID_ARG, "U table holds a non-finite value");
    }
  for (double v : c->J)
    if (!std::isfinite(v)) {
      delete c;
      return fail_noctx(DYSON_ERR_INVALID_ARG, "J table holds a non-finite value");
    }
  for (double v : c->J) c->j_max = std::max(c->j_max, (float)(std::fabs(v) * 1.000001));
  double u_min = std::numeric_limits<double>::infinity(), eps_max = 0.0;
  for (double v : c->U) u_min = std::min(u_min, std::fabs(v));
  for (int i = 0; i < c->Nr; ++i) {
    const double x = i % c->Lx - 0.5 * (c->Lx - 1), y = i / c->Lx - 0.5 * (c->Ly - 1);
    eps_max = std::max(eps_max, std::fabs(c->curvature * (x * x + y * y) - 0.5 * c->U[(size_t)i * c->Nt] - c->mu));
  }
  c->accept = accept_share(c->dt, u_min, eps_max, c->j_max);
  c->j_uniform = true;
  for (int b = 1; b < c->Nb && c->j_uniform; ++b)
    c->j_uniform = std::equal(c->J.begin() + (size_t)b * c->Nt, c->J.begin() + (size_t)(b + 1) * c->Nt, c->J.begin());

  // neighbour slots (+x, -x, +y, -y) with their bond indices
  std::vector<int> nbr((size_t)c->Nr * 4, -1), nbond((size_t)c->Nr * 4, -1);
  for (int y = 0; y < c->Ly; ++y)
    for (int x = 0; x < c->Lx; ++x) {
      int i = y * c->Lx + x;
      if (x + 1 < c->Lx) { nbr[i * 4 + 0] = i + 1; nbond[i * 4 + 0] = y * (c->Lx - 1) + x; }
      if (x > 0) { nbr[i * 4 + 1] = i - 1; nbond[i * 4 + 1] = y * (c->Lx - 1) + x - 1; }
      int vb = c->Ly * (c->Lx - 1);
      if (y + 1 < c->Ly) { nbr[i * 4 + 2] = i + c->Lx; nbond[i * 4 + 2] = vb + y * c->Lx + x; }
      if (y > 0) { nbr[i * 4 + 3] = i - c->Lx; nbond[i * 4 + 3] = vb + (y - 1) * c->Lx + x; }
    }
  c->h_nbr = nbr;
  c->h_nbond = nbond;
  const size_t NcNc = (size_t)c->Nc * c->Nc;
  auto bail = [&](cudaError_t e, const char* what) {
    int code = e == cudaErrorMemoryAllocation ? DYSON_ERR_OOM : DYSON_ERR_CUDA;
    cudaGetLastError();
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    dyson_destroy(c);
    return fail_noctx(code, m);
  };
  cudaError_t e;
  if ((e = dalloc(&c->dU, c->U.size())) || (e = dalloc(&c->dJ, c->J.size())) ||
      (e = dalloc(&c->d_nbr, nbr.size())) || (e = dalloc(&c->d_nbond, nbond.size())) ||
      (e = dalloc(&c->d_eps, (size_t)c->Nr)) || (e = dalloc(&c->d_phase, (size_t)c->Nr * (2 * c->Nc + 2))) ||
      (e = dalloc(&c->d_trig, (size_t)c->Nr * (2 * c->Nc + 2))) || (e = dalloc(&c->d_lam, (size_t)c->Nr * NcNc)) || (e = dalloc(&c->d_JW, (size_t)c->Nb * c->Nc)) ||
      (e = dalloc(&c->d_Jz, (size_t)c->Nb * contour_stride(c))) || (e = dalloc(&c->d_obs, 3 * (size_t)c->Nr * c->Nt)))
    return bail(e, "device allocation");
  std::vector<double> nan_obs(3 * (size_t)c->Nr * c->Nt, std::numeric_limits<double>::quiet_NaN());
  if ((e = cudaMemcpyAsync(c->dU, c->U.data(), c->U.size() * 8, cudaMemcpyHostToDevice, c->stream)) ||
      (e = cudaMemcpyAsync(c->dJ, c->J.data(), c->J.size() * 8, cudaMemcpyHostToDevice, c->stream)) ||
      (e = cudaMemcpyAsync(c->d_nbr, nbr.data(), nbr.size() * 4, cudaMemcpyHostToDevice, c->stream)) ||
      (e = cudaMemcpyAsync(c->d_nbond, nbond.data(), nbond.size() * 4, cudaMemcpyHostToDevice, c->stream)) ||
      (e = cudaMemcpyAsync(c->d_obs, nan_obs.data(), nan_obs.size() * 8, cudaMemcpyHostToDevice, c->stream)) ||
      (e = cudaStreamSynchronize(c->stream)))
    return bail(e, "table upload");
  *out = c;
  return DYSON_OK;
}

int dyson_build_sigma(dyson_ctx* c) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  DeviceGuard g(c->device);
  launch_build_sigma(c->dU, c->Lx, c->Ly, c->Nt, c->Nm, c->dt, c->beta, c->curvature, c->mu, c->d_eps,
                     c->d_phase, c->d_trig, c->d_lam, c->stream);
  launch_hopping_tables(c->dJ, c->Nb, c->Nt, c->Nm, c->dt, c->beta, c->d_JW, c->d_Jz, contour_stride(c),
                        c->stream);
  c->launches += c->Nb > 0 ? 4 : 3;
  DY_CUDA(c, cudaGetLastError());
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  c->sigma_built = true;
  c->lam32_built = c->lam_split_built = c->lam16_built = false;
  oz_invalidate(c);
  oz64_invalidate(c);
  se_invalidate(c);                                      // Sigma = 0: Lambda is the atomic G0 again
  return DYSON_OK;
}

int dyson_copy_sigma(dyson_ctx* c, double* dst, int on_device) {
  if (!c || !dst) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL argument");
  if (!c->sigma_built) return ctx_fail(c, DYSON_ERR_STATE, "dyson_build_sigma has not run");
  DeviceGuard g(c->device);
  DY_CUDA(c, cudaMemcpyAsync(dst, c->d_lam, (size_t)c->Nr * c->Nc * c->Nc * sizeof(double2),
                             on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  return DYSON_OK;
}

}  // extern "C"

namespace dyson_detail {

// Scratch that a solve sizes for itself and leaves with the context.  What one precision holds is free memory to
// another (release_scratch), so that a solve gets the same chunks whatever ran before it.
size_t scratch_bytes(const dyson_ctx* c) {
  return c->work_bytes + oz_x_bytes(c) + oz64_x_bytes(c) + tc_x_bytes(c) + gmres_bytes(c);
}

void release_scratch(dyson_ctx* c) {
  cudaFree(c->work);
  c->work = nullptr;
  c->work_bytes = 0;
  oz_release_x(c);
  oz64_release_x(c);
  tc_release_x(c);
  gmres_release(c);
}

// (site, vector column) pairs from which 64 contour points take the unfused sweep (prepare_tables)
constexpr int64_t kManySiteColumns = 32768;

// share of the free memory that cudaMalloc is taken to deliver in a few blocks
constexpr double kFreeShare = 0.95;

// FP64 sweeps and residuals on the tensor cores where the slices of Lambda fit (sets c->use_oz64);
// the FP64-pipe kernel otherwise.  hold: the scratch is in use and stays.
int prepare_oz64(dyson_ctx* c, bool hold) {
  size_t more = 0, free_b = 0, total_b = 0;
  c->use_oz64 = oz64_usable(c, &more);
  if (!c->use_oz64) return DYSON_OK;
  if (more > 0 && cudaMemGetInfo(&free_b, &total_b) == cudaSuccess && more > kFreeShare * free_b) {
    if (hold) c->use_oz64 = false;
    else release_scratch(c);
  }
  if (!c->use_oz64) return DYSON_OK;
  const int rc = oz64_prepare(c);
  if (rc == DYSON_ERR_OOM) c->use_oz64 = false;
  return rc == DYSON_ERR_OOM ? DYSON_OK : rc;
}

// Build the reduced-precision copies of Lambda a solve needs and pick the sweep
// and residual kernels (sets c->use_tc, c->use_oz, c->use_oz64).
// The residual of a mixed solve: five slices (15 products) for tolerances down to 1e-8, where they run at
// 85 TFLOP/s of the contraction (16x16, Nc = 256, 4096 columns: 6.5 ms); eight (36 products, 53 TFLOP/s) below.
int prepare_tables(dyson_ctx* c, int precision, double tol, int64_t columns, bool batch, bool hold) {
  // A fused tile of 256 rows is half empty at 64 contour points (128 rows of the embedding), so from
  // kManySiteColumns on the unfused form is the faster one although its series waits for every sweep:
  // single CTA / fused, us a sweep: 8x8 sites, 512 columns 34 / 46, 1024 57 / 83; 12x12, 512 62 / 85;
  // 16x16, 128 36 / 52; 5x5, 1024 33 / 43.  A form that the tuner measured is the one that runs.
  c->many_of_64 = !c->tc_tuned && c->Nc == 64 && c->Nr * columns >= kManySiteColumns;
  c->use_tc = c->use_oz = c->use_oz64 = false;
  c->Ns = c->Nc;
  if (precision == DYSON_PREC_F64) return prepare_oz64(c, hold);
  const bool tc = tc_supported(c);
  const bool fused = tc && (batch || tc_uses_fused(c));
  if (tc) c->Ns = contour_stride(c);
  if (!tc && !c->lam32_built) {
    if (!c->d_lam32) DY_CUDA(c, dalloc(&c->d_lam32, (size_t)c->Nr * c->Nc * c->Nc));
    launch_lam_c64(c->d_lam, c->Nr, c->Nt, c->Nm, c->dt, c->beta, c->d_lam32, c->stream);
    c->launches += 1;
    c->lam32_built = true;
  }
  if (fused && !c->lam16_built) {
    const size_t n = (size_t)c->Nr * 4 * c->Ns * c->Ns;
    if (!c->d_lam16_hi) DY_CUDA(c, dalloc(&c->d_lam16_hi, n));
    if (!c->d_lam16_lo) DY_CUDA(c, dalloc(&c->d_lam16_lo, n));
    if (!c->d_a_down) DY_CUDA(c, dalloc(&c->d_a_down, (size_t)c->Nr * 2 * c->Ns));
    launch_lam_split16(c->d_lam, c->Nr, c->Nt, c->Nm, c->Ns, c->dt, c->beta, c->d_lam16_hi, c->d_lam16_lo,
                       c->d_a_down, c->stream);
    c->launches += 1;
    c->lam16_built = true;
  }
  if (tc && !fused && !c->lam_split_built) {
    size_t n = (size_t)c->Nr * 4 * c->Nc * c->Nc;
    if (!c->d_lam_hi) DY_CUDA(c, dalloc(&c->d_lam_hi, n));
    if (!c->d_lam_lo) DY_CUDA(c, dalloc(&c->d_lam_lo, n));
    launch_lam_emb_split(c->d_lam, c->Nr, c->Nt, c->Nm, c->dt, c->beta, c->d_lam_hi, c->d_lam_lo, c->stream);
    c->launches += 1;
    c->lam_split_built = true;
  }
  c->use_tc = tc;
  c->use_oz = tc && tol >= kOzTol && c->slice_memory != 0 && oz_supported(c);
  return c->use_oz ? DYSON_OK : prepare_oz64(c, hold);
}

// r32 = B + K G - G with the residual kernel that prepare_tables picked; c->d_norm[q] = max |r|
int enqueue_residual(dyson_ctx* c, int ncol, int gs, const double2* G, float* r32) {
  int rc = DYSON_OK;
  KernelTimer t(c, c->use_oz || c->use_oz64 ? DYSON_KERNEL_RESIDUAL_SPLIT : DYSON_KERNEL_RESIDUAL_F64);
  if (c->use_oz) {
    rc = oz_residual(c, ncol, gs, G, r32);
  } else if (c->use_oz64) {
    rc = oz64_sweep(c, ncol, gs, G, nullptr, r32, 1);
  } else {
    launch_sweep_f64(c->d_lam, c->d_JW, c->d_nbr, c->d_nbond, G, nullptr, r32, c->Ns, c->d_src_site, c->d_src_time,
                     c->Nr, c->Nc, ncol, gs, 1, c->d_norm, c->stream);
    c->launches += 1;
  }
  if (rc) return rc;
  DY_CUDA(c, cudaGetLastError());
  return DYSON_OK;
}

// Largest number of vector columns, a multiple of `unit` and at most `want`, whose
// work state fits in 85 % of the device memory that is free or scratch of the context.  F64: two complex128
// states; mixed: complex128 G + three FP32 states (*bytes_per_col: these, the work buffer); besides it
// the FP32 gather buffer of the tensor-core sweep and the BF16 slices of the split-product
// residual or FP64 sweep (*total_per_col: all).  Frees the scratch where the buffers for these columns would not
// fit beside what it holds.
int64_t chunk_columns(dyson_ctx* c, int precision, int64_t unit, int64_t want, size_t* bytes_per_col,
                      size_t* total_per_col) {
  const double col_el = c->Nr * (double)c->Nc;
  const struct { double per_col; size_t held; } buf[4] = {
      {col_el * (precision == DYSON_PREC_F64 ? 32.0 : 16.0 + 24.0 * c->Ns / c->Nc), c->work_bytes},
      {col_el * (c->use_tc && !tc_uses_fused(c) ? 8.0 : 0.0), tc_x_bytes(c)},
      {col_el * (c->use_oz ? (double)oz_bytes_per_element() : 0.0), oz_x_bytes(c)},
      {col_el * (c->use_oz64 ? oz64_bytes_per_element(c) : 0.0), oz64_x_bytes(c)}};
  double col_bytes = 0.0;
  for (const auto& b : buf) col_bytes += b.per_col;
  *bytes_per_col = (size_t)std::ceil(buf[0].per_col);
  if (total_per_col) *total_per_col = (size_t)col_bytes;
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return 0;
  const double budget = 0.85 * (double)(free_b + scratch_bytes(c));
  int64_t cols = (int64_t)(budget / col_bytes);
  if (c->chunk_override > 0) cols = std::min<int64_t>(cols, (int64_t)c->chunk_override * unit);
  cols = std::min<int64_t>(cols, want);
  cols = std::min<int64_t>(cols, (int64_t)1 << 24);
  cols = (cols / unit) * unit;
  double more = 0.0;                                       // (a buffer that grows is freed first)
  for (const auto& b : buf) more += std::max(0.0, cols * b.per_col - (double)b.held);
  if (more > kFreeShare * free_b) release_scratch(c);
  return cols;
}

// Tables for a solve of `want` columns, *cols of them at once where memory allows; *cols becomes what it allows.
// The sweep is picked by the columns that really go through at once.
int prepare_chunk(dyson_ctx* c, int precision, double tol, int64_t unit, int64_t want, int64_t* cols, size_t* bytes_per_col) {
  int rc = prepare_tables(c, precision, tol, *cols);
  if (rc) return rc;
  *cols = chunk_columns(c, precision, unit, want, bytes_per_col);
  if (!c->many_of_64 || c->Nr * *cols >= kManySiteColumns) return DYSON_OK;
  if ((rc = prepare_tables(c, precision, tol, *cols))) return rc;
  *cols = chunk_columns(c, precision, unit, want, bytes_per_col);
  return DYSON_OK;
}

// Buffers of a chunk of ncol columns in groups of gs: work state, sources and norms, and what the sweeps and the
// residual need besides, ahead of the GMRES basis, which takes most of what is left.  Where the residual's or the
// FP64 sweep's slices cannot be had, the FP64-pipe kernel runs.
int reserve_chunk(dyson_ctx* c, int ncol, int gs, size_t bytes_per_col, bool batch) {
  int rc;
  if ((rc = ensure_work(c, (size_t)ncol * bytes_per_col)) || (rc = ensure_cols(c, ncol, ncol / gs))) return rc;
  if (c->use_tc && (rc = tc_prepare_sweep(c, ncol, batch))) return rc;
  if (c->use_oz && (rc = oz_reserve(c, ncol)) == DYSON_ERR_OOM) c->use_oz = false;
  else if (c->use_oz && rc) return rc;
  if (c->use_oz64 && (rc = oz64_reserve(c, ncol)) == DYSON_ERR_OOM) c->use_oz64 = false;
  else if (c->use_oz64 && rc) return rc;
  return DYSON_OK;
}

int solve_chunk(dyson_ctx* c, int ncol, int gs, int precision, double tol, int max_sweeps, double2** G,
                dyson_report* rep) {
  int rc = upload_sources(c, ncol);
  if (rc) return rc;
  return precision == DYSON_PREC_F64 ? solve_f64(c, ncol, gs, tol, max_sweeps, G, rep)
                                     : solve_mixed(c, ncol, gs, precision, tol, max_sweeps, G, rep);
}

int check_solve_args(dyson_ctx* c, int precision, double tol, int max_sweeps) {
  if (!c->sigma_built) return ctx_fail(c, DYSON_ERR_STATE, "dyson_build_sigma has not run");
  if (precision != DYSON_PREC_F64 && precision != DYSON_PREC_TF32X3_F64REF)
    return ctx_fail(c, DYSON_ERR_INVALID_ARG, "unknown precision");
  if (!(tol > 0) || max_sweeps < 1) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "need tol > 0 and max_sweeps >= 1");
  return DYSON_OK;
}

struct ReportScope {
  dyson_ctx* c;
  dyson_report rep;
  dyson_report* out;
  int64_t launches0, syncs0;
  std::chrono::steady_clock::time_point t0;
  ReportScope(dyson_ctx* cc, dyson_report* o) : c(cc), out(o), launches0(cc->launches), syncs0(cc->host_syncs) {
    std::memset(&rep, 0, sizeof rep);
    t0 = std::chrono::steady_clock::now();
  }
  int finish(int code) {
    rep.status = code;
    rep.kernel_launches = c->launches - launches0;
    rep.host_syncs = (int32_t)(c->host_syncs - syncs0);
    rep.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (out) *out = rep;
    return code;
  }
};

int fold_status(int status, int st) {
  if (st != DYSON_OK && status == DYSON_OK) return st;
  return status;
}

}  // namespace dyson_detail

extern "C" {

namespace {

// block-column solves; g_out: full block columns, gloc: diagonal blocks G_ss at row s (either may be NULL)
int solve_columns_impl(dyson_ctx* c, const int32_t* src, int64_t n_src, int precision, double tol,
                       int32_t max_sweeps, double* g_out, double* gloc, dyson_report* rep_out) {
  ReportScope R(c, rep_out);
  int rc = check_solve_args(c, precision, tol, max_sweeps);
  if (rc) return R.finish(rc);
  if (c->sigma_transposed)
    return R.finish(ctx_fail(c, DYSON_ERR_STATE, "Lambda is transposed: block columns and observables need it upright"));
  if (n_src < 1 || !src) return R.finish(ctx_fail(c, DYSON_ERR_INVALID_ARG, "need at least one source site"));
  for (int64_t q = 0; q < n_src; ++q)
    if (src[q] < 0 || src[q] >= c->Nr) return R.finish(ctx_fail(c, DYSON_ERR_INVALID_ARG, "source site out of range"));
  DeviceGuard g(c->device);
  const int64_t at_once = c->chunk_override > 0 ? std::min<int64_t>(n_src, c->chunk_override) : n_src;
  size_t col_bytes = 0;
  int64_t cols = at_once * c->Nc;
  if ((rc = prepare_chunk(c, precision, tol, c->Nc, n_src * (int64_t)c->Nc, &cols, &col_bytes))) return R.finish(rc);
  if (cols < c->Nc) return R.finish(ctx_fail(c, DYSON_ERR_OOM, "one block column does not fit in device memory"));
  const int64_t chunk = cols / c->Nc;
  if ((rc = reserve_chunk(c, (int)cols, c->Nc, col_bytes))) return R.finish(rc);

  int status = DYSON_OK;
  for (int64_t start = 0; start < n_src; start += chunk) {
    const int nq = (int)std::min<int64_t>(chunk, n_src - start);
    const int ncol = nq * c->Nc;
    c->h_src_site.resize(ncol);
    c->h_src_time.resize(ncol);
    for (int q = 0; q < nq; ++q)
      for (int z = 0; z < c->Nc; ++z) {
        c->h_src_site[q * c->Nc + z] = src[start + q];
        c->h_src_time[q * c->Nc + z] = z;
      }
    double2* G = nullptr;
    int st = solve_chunk(c, ncol, c->Nc, precision, tol, max_sweeps, &G, &R.rep);
    if (st != DYSON_OK && st != DYSON_ERR_NOT_CONVERGED && st != DYSON_ERR_DIVERGED) return R.finish(st);
    if (!G) return R.finish(ctx_fail(c, DYSON_ERR_STATE, "solve produced no state"));
    status = fold_status(status, st);
    R.rep.chunks += 1;
    launch_observables(G, c->d_src_site, nq, c->d_nbr, c->d_nbond, c->dJ, c->d_eps, c->dU, c->Nr, c->Nt, c->Nc,
                       ncol, c->dt, c->d_obs, c->stream);
    c->launches += 1;
    if (g_out) {
      launch_export(G, c->Nr, c->Nc, nq, (double2*)g_out + (size_t)start * c->Nr * c->Nc * c->Nc, c->stream);
      c->launches += 1;
    }
    if (gloc) {
      launch_export_diagonal(G, c->d_src_site, c->Nc, ncol, nq, (double2*)gloc, c->stream);
      c->launches += 1;
    }
    DY_CUDA(c, cudaGetLastError());
  }
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  flush_timers(c);
  if (status == DYSON_ERR_NOT_CONVERGED) ctx_fail(c, status, "max_sweeps or refinement limit reached above tolerance");
  if (status == DYSON_ERR_DIVERGED) ctx_fail(c, status, "series diverged (update not finite or past the rounding limit, or refinement residual growing)");
  return R.finish(status);
}

}  // namespace

int dyson_solve_columns(dyson_ctx* c, const int32_t* src, int64_t n_src, int precision, double tol,
                        int32_t max_sweeps, double* g_out, dyson_report* rep_out) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (c->symmetry == DYSON_SYMMETRY_C4V)
    return solve_columns_c4v(c, src, n_src, precision, tol, max_sweeps, g_out, rep_out);
  return solve_columns_impl(c, src, n_src, precision, tol, max_sweeps, g_out, nullptr, rep_out);
}

int dyson_local_greens(dyson_ctx* c, const int32_t* src, int64_t n_src, int precision, double tol,
                       int32_t max_sweeps, double* gloc, dyson_report* rep_out) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (!gloc) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "gloc is NULL");
  if (c->symmetry == DYSON_SYMMETRY_C4V)
    return local_greens_c4v(c, src, n_src, precision, tol, max_sweeps, gloc, rep_out);
  return solve_columns_impl(c, src, n_src, precision, tol, max_sweeps, nullptr, gloc, rep_out);
}

int dyson_solve_vector_columns(dyson_ctx* c, const int32_t* sites, const int32_t* times, int64_t n, int precision,
                               double tol, int32_t max_sweeps, double* g_out, dyson_report* rep_out) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  ReportScope R(c, rep_out);
  int rc = check_solve_args(c, precision, tol, max_sweeps);
  if (rc) return R.finish(rc);
  if (n < 1 || !sites || !times) return R.finish(ctx_fail(c, DYSON_ERR_INVALID_ARG, "need at least one column"));
  for (int64_t q = 0; q < n; ++q)
    if (sites[q] < 0 || sites[q] >= c->Nr || times[q] < 0 || times[q] >= c->Nc)
      return R.finish(ctx_fail(c, DYSON_ERR_INVALID_ARG, "column source out of range"));
  DeviceGuard g(c->device);
  constexpr int GS = 32;                                   // norm group; columns padded to a multiple
  const int64_t padded = (n + GS - 1) / GS * GS;
  size_t col_bytes = 0;
  int64_t chunk = n;
  if ((rc = prepare_chunk(c, precision, tol, GS, padded, &chunk, &col_bytes))) return R.finish(rc);
  if (chunk < GS) return R.finish(ctx_fail(c, DYSON_ERR_OOM, "32 vector columns do not fit in device memory"));
  if ((rc = reserve_chunk(c, (int)chunk, GS, col_bytes))) return R.finish(rc);
  int status = DYSON_OK;
  for (int64_t start = 0; start < padded; start += chunk) {
    const int ncol = (int)std::min<int64_t>(chunk, padded - start);
    c->h_src_site.assign(ncol, -1);
    c->h_src_time.assign(ncol, 0);
    const int nv = (int)std::min<int64_t>(ncol, n - start);
    for (int k = 0; k < nv; ++k) {
      c->h_src_site[k] = sites[start + k];
      c->h_src_time[k] = times[start + k];
    }
    double2* G = nullptr;
    int st = solve_chunk(c, ncol, GS, precision, tol, max_sweeps, &G, &R.rep);
    if (st != DYSON_OK && st != DYSON_ERR_NOT_CONVERGED && st != DYSON_ERR_DIVERGED) return R.finish(st);
    if (!G) return R.finish(ctx_fail(c, DYSON_ERR_STATE, "solve produced no state"));
    status = fold_status(status, st);
    R.rep.chunks += 1;
    if (g_out) {
      launch_export_vectors(G, c->Nr, c->Nc, ncol, nv, (double2*)g_out + (size_t)start * c->Nr * c->Nc, c->stream);
      c->launches += 1;
    }
    DY_CUDA(c, cudaGetLastError());
  }
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  flush_timers(c);
  if (status == DYSON_ERR_NOT_CONVERGED) ctx_fail(c, status, "max_sweeps or refinement limit reached above tolerance");
  if (status == DYSON_ERR_DIVERGED) ctx_fail(c, status, "series diverged (update not finite or past the rounding limit, or refinement residual growing)");
  return R.finish(status);
}

int dyson_adjoint_obs(dyson_ctx* c, const double* w_density, const double* w_docc, int32_t t_index, int precision,
                      double tol, int32_t max_sweeps, double* loss, double* grad_U, double* grad_J,
                      dyson_report* rep_out) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  ReportScope R(c, rep_out);
  int rc = check_solve_args(c, precision, tol, max_sweeps);
  if (rc) return R.finish(rc);
  if (c->sigma_transposed) return R.finish(ctx_fail(c, DYSON_ERR_STATE, "Lambda is transposed"));
  if (c->se_installed)
    return R.finish(ctx_fail(c, DYSON_ERR_STATE, "the adjoint differentiates the atomic Lambda: rebuild it first"));
  if ((!w_density && !w_docc) || t_index < 0 || t_index >= c->Nt || (w_docc && t_index < 1))
    return R.finish(ctx_fail(c, DYSON_ERR_INVALID_ARG, "need weights, 0 <= t_index < Nt (>= 1 with D weights)"));
  DeviceGuard g(c->device);
  const int Nr = c->Nr, Nc = c->Nc, Nt = c->Nt;
  const bool docc = w_docc != nullptr;
  const size_t colbuf = (size_t)Nr * Nr * Nc;                 // double2 elements of C (and the rows, psi, gamma, rho)
  const size_t nbuf = docc ? 6 : 5;
  const size_t need = (nbuf * colbuf + (size_t)Nr * Nc * Nc) * sizeof(double2) + (size_t)Nr * sizeof(AdjCoef) +
                      ((size_t)3 * Nr + 1 + (size_t)Nr * Nt + (size_t)std::max(c->Nb, 1) * Nt) * sizeof(double);
  if (c->adj_bytes < need) {
    if (c->adj) cudaFree(c->adj);
    c->adj = nullptr;
    c->adj_bytes = 0;
    cudaError_t e = cudaMalloc(&c->adj, need);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return R.finish(ctx_fail(c, DYSON_ERR_OOM, "adjoint buffers"));
    }
    c->adj_bytes = need;
  }
  double2* C = (double2*)c->adj;
  double2* R1 = C + colbuf;
  double2* R2 = docc ? R1 + colbuf : nullptr;
  double2* psi = (docc ? R2 : R1) + colbuf;
  double2* gam = psi + colbuf;
  double2* rho = gam + colbuf;
  double2* M = rho + colbuf;
  AdjCoef* coef_dev = (AdjCoef*)(M + (size_t)Nr * Nc * Nc);
  double* wn_dev = (double*)(coef_dev + Nr);
  double* wd_dev = wn_dev + Nr;
  double* ones_dev = wd_dev + Nr;
  double* loss_dev = ones_dev + Nr;
  double* gU_dev = loss_dev + 1;
  double* gJ_dev = gU_dev + (size_t)Nr * Nt;
  // coefficients beta'_i = i beta_i of the rows (see k_adjoint.cu): the density
  // n_i = Im c_i(i, kf) gives b0 += w; the double occupancy D_i of Eq. (docc) gives
  // b0 += i v / (dt U) - v eps / U, b1 = -i v / (dt U), bj = -v J_ij / U
  std::vector<double> eps(Nr);
  DY_CUDA(c, cudaMemcpyAsync(eps.data(), c->d_eps, Nr * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  std::vector<AdjCoef> coef(Nr);
  std::vector<double> ones(Nr, 1.0);
  for (int i = 0; i < Nr; ++i) {
    AdjCoef& k = coef[i];
    std::memset(&k, 0, sizeof k);
    if (w_density) k.b0.x += w_density[i];
    if (docc && w_docc[i] != 0.0) {
      const double v = w_docc[i], U = c->U[(size_t)i * Nt + t_index];
      k.b0.x += -v * eps[i] / U;
      k.b0.y += v / (c->dt * U);
      k.b1.y = -v / (c->dt * U);
      for (int s = 0; s < 4; ++s)
        if (c->h_nbr[i * 4 + s] >= 0) k.bj[s].x = -v * c->J[(size_t)c->h_nbond[i * 4 + s] * Nt + t_index] / U;
    }
  }
  DY_CUDA(c, cudaMemcpyAsync(coef_dev, coef.data(), Nr * sizeof(AdjCoef), cudaMemcpyHostToDevice, c->stream));
  DY_CUDA(c, cudaMemcpyAsync(ones_dev, ones.data(), Nr * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  if (w_density)
    DY_CUDA(c, cudaMemcpyAsync(wn_dev, w_density, Nr * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  if (docc) DY_CUDA(c, cudaMemcpyAsync(wd_dev, w_docc, Nr * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  // columns G e_i at (i, kf); rows of G (columns of G^T) at (i, kf) and, for D, (i, kf - 1)
  std::vector<int32_t> sites(2 * (size_t)Nr), times(2 * (size_t)Nr);
  for (int i = 0; i < Nr; ++i) {
    sites[i] = sites[Nr + i] = i;
    times[i] = t_index;
    times[Nr + i] = t_index - 1;
  }
  dyson_report r1, r2;
  int st1 = dyson_solve_vector_columns(c, sites.data(), times.data(), Nr, precision, tol, max_sweeps,
                                       (double*)C, &r1);
  if (st1 != DYSON_OK && st1 != DYSON_ERR_NOT_CONVERGED) return R.finish(st1);
  if ((rc = dyson_transpose_sigma(c))) return R.finish(rc);
  int st2 = dyson_solve_vector_columns(c, sites.data(), times.data(), docc ? 2 * Nr : Nr, precision, tol,
                                       max_sweeps, (double*)R1, &r2);
  if ((rc = dyson_transpose_sigma(c))) return R.finish(rc);
  if (st2 != DYSON_OK && st2 != DYSON_ERR_NOT_CONVERGED) return R.finish(st2);
  R.rep.sweeps = r1.sweeps + r2.sweeps;
  R.rep.refinements = r1.refinements + r2.refinements;
  R.rep.chunks = r1.chunks + r2.chunks;
  R.rep.gemm_flops = r1.gemm_flops + r2.gemm_flops;
  R.rep.update = std::max(r1.update, r2.update);
  R.rep.residual = std::max(r1.residual, r2.residual);
  R.rep.inner_gmres = r1.inner_gmres | r2.inner_gmres;
  if ((rc = adjoint_contract_obs(c, C, R1, R2, coef_dev, w_density ? wn_dev : nullptr, docc ? wd_dev : nullptr,
                                 ones_dev, t_index, psi, gam, rho, M, loss_dev, gU_dev, gJ_dev)))
    return R.finish(rc);
  if (loss) DY_CUDA(c, cudaMemcpyAsync(loss, loss_dev, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  if (grad_U)
    DY_CUDA(c, cudaMemcpyAsync(grad_U, gU_dev, (size_t)Nr * Nt * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  if (grad_J && c->Nb > 0)
    DY_CUDA(c, cudaMemcpyAsync(grad_J, gJ_dev, (size_t)c->Nb * Nt * sizeof(double), cudaMemcpyDeviceToHost,
                               c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  const int status = fold_status(st1, st2);
  if (status == DYSON_ERR_NOT_CONVERGED) ctx_fail(c, status, "max_sweeps or refinement limit reached above tolerance");
  return R.finish(status);
}

int dyson_adjoint(dyson_ctx* c, const double* w, int32_t t_index, int precision, double tol, int32_t max_sweeps,
                  double* loss, double* grad_U, double* grad_J, dyson_report* rep_out) {
  if (c && !w) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "bad weights or time");
  return dyson_adjoint_obs(c, w, nullptr, t_index, precision, tol, max_sweeps, loss, grad_U, grad_J, rep_out);
}

int dyson_transpose_sigma(dyson_ctx* c) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (!c->sigma_built) return ctx_fail(c, DYSON_ERR_STATE, "dyson_build_sigma has not run");
  DeviceGuard g(c->device);
  launch_transpose_blocks(c->d_lam, c->Nr, c->Nc, c->stream);
  c->launches += 1;
  DY_CUDA(c, cudaGetLastError());
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  c->sigma_transposed = !c->sigma_transposed;
  c->lam32_built = c->lam_split_built = c->lam16_built = false;
  oz_invalidate(c);
  oz64_invalidate(c);
  return DYSON_OK;
}

int dyson_observables(dyson_ctx* c, double* n, double* ekin, double* docc, int on_device) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  DeviceGuard g(c->device);
  size_t cnt = (size_t)c->Nr * c->Nt;
  double* dst[3] = {n, ekin, docc};
  for (int k = 0; k < 3; ++k)
    if (dst[k])
      DY_CUDA(c, cudaMemcpyAsync(dst[k], c->d_obs + k * cnt, cnt * sizeof(double),
                                 on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, c->stream));
  DY_CUDA(c, cudaStreamSynchronize(c->stream));
  return DYSON_OK;
}

int dyson_profile(dyson_ctx* c, int enable) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  flush_timers(c);
  c->profiling = enable != 0;
  for (int k = 0; k < DYSON_KERNEL_KINDS; ++k) {
    c->prof_ms[k] = 0.0;
    c->prof_launches[k] = 0;
  }
  return DYSON_OK;
}

int dyson_profile_query(dyson_ctx* c, int kind, int64_t* launches, double* total_ms) {
  if (!c || kind < 0 || kind >= DYSON_KERNEL_KINDS) return fail_noctx(DYSON_ERR_INVALID_ARG, "bad kernel kind");
  flush_timers(c);
  if (launches) *launches = c->prof_launches[kind];
  if (total_ms) *total_ms = c->prof_ms[kind];
  return DYSON_OK;
}

int64_t dyson_launch_count(const dyson_ctx* c) { return c ? c->launches : -1; }

int dyson_set_chunk(dyson_ctx* c, int32_t block_columns) {
  if (!c || block_columns < 0) return fail_noctx(DYSON_ERR_INVALID_ARG, "bad chunk size");
  c->chunk_override = block_columns;
  return DYSON_OK;
}

int dyson_set_inner_solver(dyson_ctx* c, int solver, int32_t restart) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (solver != DYSON_INNER_SERIES && solver != DYSON_INNER_GMRES && solver != DYSON_INNER_AUTO)
    return ctx_fail(c, DYSON_ERR_INVALID_ARG, "unknown inner solver");
  if (restart < 0 || restart > 60) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "restart length must be 0..60");
  c->inner_solver = solver;
  c->gmres_restart = restart > 0 ? restart : 40;
  return DYSON_OK;
}

int dyson_set_support_truncation(dyson_ctx* c, int enable) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  c->support_trunc = enable != 0;
  return DYSON_OK;
}

int dyson_set_wait_limit(dyson_ctx* c, double seconds) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (!(seconds >= 0.0) || seconds > 60.0) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "limit must be in [0, 60] s");
  DeviceGuard g(c->device);
  const unsigned long long ns = seconds == 0.0 ? 2000000000ull : (unsigned long long)(seconds * 1e9);
  int rc = tc_set_wait_limit(c, ns);
  if (rc) return rc;
  if ((rc = oz_set_wait_limit(c, ns))) return rc;
  return oz64_set_wait_limit(c, ns);
}

int dyson_set_slice_memory(dyson_ctx* c, int64_t bytes) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (bytes < -1) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "need a number of bytes, or -1");
  c->slice_memory = bytes;
  return DYSON_OK;
}

int dyson_set_graph_sweeps(dyson_ctx* c, int sweeps) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (sweeps < 0 || sweeps > 64 || sweeps % 2) return ctx_fail(c, DYSON_ERR_INVALID_ARG, "sweeps must be even, 0..64");
  c->graph_sweeps = sweeps;
  return DYSON_OK;
}

int dyson_set_sweep_variant(dyson_ctx* c, int variant) {
  if (!c) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context");
  if (variant < DYSON_SWEEP_SINGLE_CTA || variant > DYSON_SWEEP_FUSED_PAIR_WIDE)
    return ctx_fail(c, DYSON_ERR_INVALID_ARG, "unknown sweep variant");
  c->tc_variant = variant;
  c->tc_tuned = false;
  return DYSON_OK;
}

void dyson_destroy(dyson_ctx* c) {
  if (!c) return;
  DeviceGuard g(c->device);
  cudaStreamSynchronize(c->stream);
  flush_timers(c);
  tc_release(c);
  oz_release(c);
  oz64_release(c);
  gmres_release(c);
  se_release(c);
  if (c->d_sym_perm) cudaFree(c->d_sym_perm);
  void* ptrs[] = {c->dU, c->dJ, c->d_nbr, c->d_nbond, c->d_eps, c->d_phase, c->d_trig, c->d_lam, c->d_JW, c->d_Jz,
                  c->d_lam32, c->d_lam_hi, c->d_lam_lo, c->d_obs, c->work, c->d_src_site, c->d_src_time,
                  c->d_norm, c->adj, c->d_act, c->d_series, c->d_rref, c->d_xscale, c->d_lam16_hi,
                  c->d_lam16_lo, c->d_a_down};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (c->h_norm) cudaFreeHost(c->h_norm);
  if (c->d_f64_run) cudaFree(c->d_f64_run);
  if (c->h_f64_upd) cudaFreeHost(c->h_f64_upd);
  for (cudaEvent_t e : c->f64_ev)
    if (e) cudaEventDestroy(e);
  if (c->h_series) cudaFreeHost(c->h_series);
  delete c;
}

}  // extern "C"
