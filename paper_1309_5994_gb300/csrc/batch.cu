// Batched mixed-precision solves of several problem instances (dyson_batch_*).
//
// Each instance is a context of its own (lattice, contour, trap, drive, Lambda)
// solving its block columns with the series of App. C refined by FP64 residuals,
// exactly as dyson_solve_columns(precision = TF32X3_F64REF) does: the same sweeps, stopping rule and
// residuals.  What is shared is the device: the inner series run side by side on BATCH_LANES streams, a number
// of sweeps enqueued at a time for every instance still iterating, and the host waits once for all of them.  An
// instance that has stopped takes no more part.  The FP64 residual refinement (split-product
// residual, k_oz.cu or k_oz64.cu) runs per instance between inner solves.  An instance whose
// series diverges (spectral radius of K above 1) is then solved alone with the
// GMRES of App. C (k_gmres.cu).
// Six instances of 8x8 to 16x16 sites to 1e-10: 52.7 ms (one by one 62.5).  As a graph of S sweeps of all instances,
// captured for every call, each sweep ended by a check of all, 60.4; twelve drawn batches of 2 to 8 instances were
// 1.14 to 1.27 times as long so.
#include <algorithm>
#include <chrono>
#include <limits>
#include <vector>

#include "common.cuh"
#include "detail.cuh"
#include "oz.cuh"
#include "oz64.cuh"
#include "tc.cuh"

using namespace dyson_detail;

namespace {

// Streams that the instances' series run on: the tail of one instance's sweep overlaps another's.
constexpr int BATCH_LANES = 4;
// More instances than this have their launches overlap as a single solve's do.  A sweep that waits for its turn holds
// its SMs meanwhile: two instances of 4x4 and 10x10 sites 3.43 ms without, 3.75 with; three 8.94 and 8.95, eight
// 35.4 and 34.9, six large ones 53.9 and 52.7.
constexpr size_t OVERLAP_ABOVE = 2;

// per-instance host state of one batched solve
struct Inst {
  dyson_ctx* c = nullptr;
  int nq = 0, ncol = 0, ng = 0;
  double2* G = nullptr;
  float *r32 = nullptr, *da = nullptr, *db = nullptr;
  SeriesRun run{};
  std::vector<double> scale, rref;
  double prev_res = std::numeric_limits<double>::infinity();
  int strikes = 0;
  bool plateau = true;               // the series may end on a plateau
  int status = DYSON_ERR_NOT_CONVERGED;
  bool done = false;
  int64_t launches0 = 0;
  dyson_report rep{};
};

}  // namespace

struct dyson_batch {
  std::vector<dyson_ctx*> ctx;
  int device = 0;
  cudaStream_t stream = nullptr;     // the contexts' stream
  std::string err;
  int64_t launches = 0;
  cudaStream_t lane[BATCH_LANES] = {};
  cudaEvent_t ready = nullptr;
};

namespace {

int bfail(dyson_batch* b, int code, const std::string& m) {
  if (b) b->err = m;
  else fail_noctx(code, m);
  return code;
}

#define DYB_CUDA(b, call)                                                          \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess) {                                                       \
      cudaGetLastError();                                                          \
      return bfail(b, DYSON_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    }                                                                              \
  } while (0)

// The contexts' streams while their series run on the lanes; back on the batch's stream, and nothing of them in
// flight, when it goes.
struct OnLanes {
  dyson_batch* b;
  explicit OnLanes(dyson_batch* bb) : b(bb) {
    for (size_t k = 0; k < b->ctx.size(); ++k) b->ctx[k]->stream = b->lane[k % BATCH_LANES];
  }
  cudaError_t wait() const {
    cudaError_t e = cudaSuccess;
    for (cudaStream_t s : b->lane) {
      const cudaError_t e1 = cudaStreamSynchronize(s);
      if (e == cudaSuccess) e = e1;
    }
    return e;
  }
  ~OnLanes() {
    wait();
    for (dyson_ctx* c : b->ctx) c->stream = b->stream;
  }
};

}  // namespace

extern "C" {

int dyson_batch_create(dyson_batch** out, dyson_ctx* const* ctxs, int32_t n) {
  if (!out) return fail_noctx(DYSON_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!ctxs || n < 1 || n > DYSON_BATCH_MAX_INSTANCES)
    return fail_noctx(DYSON_ERR_INVALID_ARG, "a batch holds 1.." + std::to_string(DYSON_BATCH_MAX_INSTANCES) +
                                                 " contexts");
  for (int k = 0; k < n; ++k) {
    if (!ctxs[k]) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL context in the batch");
    if (ctxs[k]->device != ctxs[0]->device || ctxs[k]->stream != ctxs[0]->stream)
      return fail_noctx(DYSON_ERR_INVALID_ARG, "batched contexts must share one device and one stream");
    for (int j = 0; j < k; ++j)
      if (ctxs[j] == ctxs[k]) return fail_noctx(DYSON_ERR_INVALID_ARG, "a context appears twice in the batch");
  }
  DeviceGuard g(ctxs[0]->device);
  auto* b = new dyson_batch;
  b->ctx.assign(ctxs, ctxs + n);
  b->device = ctxs[0]->device;
  b->stream = ctxs[0]->stream;
  cudaError_t e = cudaEventCreateWithFlags(&b->ready, cudaEventDisableTiming);
  for (cudaStream_t& l : b->lane)
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&l, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    cudaGetLastError();
    dyson_batch_destroy(b);
    return fail_noctx(e == cudaErrorMemoryAllocation ? DYSON_ERR_OOM : DYSON_ERR_CUDA,
                      std::string("batch set-up: ") + cudaGetErrorString(e));
  }
  *out = b;
  return DYSON_OK;
}

int dyson_batch_solve(dyson_batch* b, const int32_t* const* src, const int32_t* n_src, double tol,
                      int32_t max_sweeps, int32_t graph_sweeps, double* const* g_out, dyson_report* reports) {
  if (!b) return fail_noctx(DYSON_ERR_INVALID_ARG, "NULL batch");
  const int n = (int)b->ctx.size();
  if (!src || !n_src) return bfail(b, DYSON_ERR_INVALID_ARG, "NULL source arrays");
  if (!(tol > 0) || max_sweeps < 1 || graph_sweeps < 0)
    return bfail(b, DYSON_ERR_INVALID_ARG, "need tol > 0, max_sweeps >= 1 and graph_sweeps >= 0");
  // sweeps enqueued at a time; even, so that each time starts from the first state
  int S = graph_sweeps > 0 ? graph_sweeps : 8;
  S += S & 1;
  const auto t0 = std::chrono::steady_clock::now();
  DeviceGuard g(b->device);
  std::vector<Inst> I(n);
  int rc;
  // ---- per-instance set-up: tables, work buffers, right-hand sides ----
  for (int k = 0; k < n; ++k) {
    Inst& X = I[k];
    dyson_ctx* c = X.c = b->ctx[k];
    X.launches0 = c->launches;
    if (!c->sigma_built || c->sigma_transposed)
      return bfail(b, DYSON_ERR_STATE, "instance " + std::to_string(k) + ": Lambda not built or transposed");
    if (n_src[k] < 1 || !src[k]) return bfail(b, DYSON_ERR_INVALID_ARG, "every instance needs a source site");
    for (int q = 0; q < n_src[k]; ++q)
      if (src[k][q] < 0 || src[k][q] >= c->Nr) return bfail(b, DYSON_ERR_INVALID_ARG, "source site out of range");
    if ((rc = prepare_tables(c, DYSON_PREC_TF32X3_F64REF, tol, 0, true))) return bfail(b, rc, c->err);
    if (!c->use_tc || !oz_supported(c) || !tc_fused_runs(c))
      return bfail(b, DYSON_ERR_INVALID_ARG,
                   "instance " + std::to_string(k) + ": batched solves need Nc % 64 == 0 and 2 Nc <= 512");
    X.nq = n_src[k];
    X.ncol = X.nq * c->Nc;
    X.ng = X.nq;
    size_t col_bytes = 0;
    if (chunk_columns(c, DYSON_PREC_TF32X3_F64REF, c->Nc, X.ncol, &col_bytes) < X.ncol)
      return bfail(b, DYSON_ERR_OOM, "instance " + std::to_string(k) + ": its block columns do not fit at once");
    if ((rc = reserve_chunk(c, X.ncol, c->Nc, col_bytes, true))) return bfail(b, rc, c->err);
    c->h_src_site.resize(X.ncol);
    c->h_src_time.resize(X.ncol);
    for (int q = 0; q < X.nq; ++q)
      for (int z = 0; z < c->Nc; ++z) {
        c->h_src_site[q * c->Nc + z] = src[k][q];
        c->h_src_time[q * c->Nc + z] = z;
      }
    if ((rc = upload_sources(c, X.ncol))) return bfail(b, rc, c->err);
    const size_t n_el = (size_t)c->Nr * X.ncol * c->Nc, n32 = (size_t)c->Nr * X.ncol * 2 * c->Ns;
    X.G = (double2*)c->work;
    X.r32 = (float*)(X.G + n_el);
    X.da = X.r32 + n32;
    X.db = X.da + n32;
    DYB_CUDA(b, cudaMemsetAsync(X.G, 0, n_el * sizeof(double2), c->stream));
    DYB_CUDA(b, cudaMemsetAsync(c->d_norm, 0, 2 * (size_t)X.ng * sizeof(unsigned long long), c->stream));
    launch_init_rhs(c->d_lam, c->d_src_site, c->d_src_time, c->Nr, c->Nc, X.ncol, c->Nc, X.G, c->d_norm + X.ng,
                    c->stream);
    launch_to_planar32(X.G, X.r32, (size_t)c->Nr * X.ncol, c->Nc, c->Ns, c->stream);
    c->launches += 2;
    DYB_CUDA(b, cudaMemsetAsync(X.G, 0, n_el * sizeof(double2), c->stream));
    if ((rc = read_norms(c, X.ng, true))) return bfail(b, rc, c->err);
    X.scale.resize(X.ng);
    for (int q = 0; q < X.ng; ++q) X.scale[q] = bits_to_double(c->h_norm[X.ng + q]);
    X.rref = X.scale;
  }
  // ---- refinements: batched inner series, per-instance FP64 residuals ----
  dyson_ctx* c0 = b->ctx[0];
  const int max_ref = c0->max_refinements;
  for (int ref = 0; ref < max_ref; ++ref) {
    std::vector<int> live;
    for (int k = 0; k < n; ++k) {
      Inst& X = I[k];
      if (X.done) continue;
      dyson_ctx* c = X.c;
      live.push_back(k);
      const size_t n32 = (size_t)c->Nr * X.ncol * 2 * c->Ns;
      DYB_CUDA(b, cudaMemcpyAsync(X.da, X.r32, n32 * sizeof(float), cudaMemcpyDeviceToDevice, b->stream));
      // the first right-hand side lives on the source sites (skipped tiles stay 0)
      const int* act = ref == 0 && c->support_trunc ? support_table(c, X.ncol) : nullptr;
      if (act) DYB_CUDA(b, cudaMemsetAsync(X.db, 0, n32 * sizeof(float), b->stream));
      X.run = SeriesRun{c, X.ncol, c->Nc, max_sweeps, S, X.r32, X.da, X.db, act, ref == 0 ? TC_R_ON_SOURCES : TC_R_DENSE,
                        inner_target(kInnerTarget, tol, X.prev_res), kSeriesPeakMax, &X.rep};
      if ((rc = seed_series(c, X.rref)) || (rc = X.run.begin(X.plateau))) return bfail(b, rc, c->err);
    }
    if (live.empty()) break;
    {
      DYB_CUDA(b, cudaEventRecord(b->ready, b->stream));
      for (cudaStream_t l : b->lane) DYB_CUDA(b, cudaStreamWaitEvent(l, b->ready, 0));
      OnLanes lanes(b);
      std::vector<int> going = live;
      while (!going.empty()) {
        for (int k : going) {
          if ((rc = I[k].run.enqueue(going.size() > OVERLAP_ABOVE))) return bfail(b, rc, I[k].c->err);
          b->launches += 2 * (int64_t)S;
        }
        DYB_CUDA(b, lanes.wait());
        std::vector<int> next;
        for (int k : going) {
          I[k].run.collect(&rc);
          if (rc) return bfail(b, rc, I[k].c->err);
          if (I[k].run.running()) next.push_back(k);
        }
        going.swap(next);
      }
    }
    // G += d, then the FP64-accurate residual, per live instance
    for (int k = 0; k < n; ++k) {
      Inst& X = I[k];
      if (X.done) continue;
      dyson_ctx* c = X.c;
      const int outcome = X.run.state()->outcome;
      if (outcome == SERIES_ABORTED || outcome == SERIES_NOT_FINITE) {
        X.status = X.prev_res <= tol ? DYSON_OK : DYSON_ERR_DIVERGED;
        X.done = true;
        continue;
      }
      const float* d = X.run.da;
      launch_accumulate(X.G, d, c->Nr, c->Nc, c->Ns, X.ncol, c->stream);
      c->launches += 1;
      DYB_CUDA(b, cudaMemsetAsync(c->d_norm, 0, (size_t)X.ng * sizeof(unsigned long long), c->stream));
      if ((rc = enqueue_residual(c, X.ncol, c->Nc, X.G, X.r32))) return bfail(b, rc, c->err);
    }
    for (int k = 0; k < n; ++k) {
      Inst& X = I[k];
      if (X.done) continue;
      dyson_ctx* c = X.c;
      if ((rc = read_norms(c, X.ng, false))) return bfail(b, rc, c->err);
      if ((rc = oz_check_error(c))) return bfail(b, rc, c->err);
      X.rep.refinements += 1;
      X.rep.gemm_flops += sweep_flops(c, X.ncol);
      const double res = rel_max(c->h_norm, X.scale.data(), X.ng);
      X.rep.residual = res;
      for (int q = 0; q < X.ng; ++q) X.rref[q] = std::max(bits_to_double(c->h_norm[q]), 1e-300);
      if (!(res < kDivergedGrowth)) {
        if (c->use_oz64 && (rc = oz64_check_error(c))) return bfail(b, rc, c->err);
        X.status = DYSON_ERR_DIVERGED;
        X.done = true;
      } else if (res <= tol) {
        if (!refine_once_more(res, tol, X.prev_res, c->accept, ref + 1 == max_ref)) {
          X.status = DYSON_OK;
          X.done = true;
        }
      } else if (res > kRefineContract * X.prev_res && ++X.strikes >= kRefineStrikes) {
        X.status = DYSON_ERR_DIVERGED;
        X.done = true;
      }
      if (X.run.state()->outcome == SERIES_PLATEAU && !plateau_served(res, X.prev_res)) X.plateau = false;
      X.prev_res = res;
    }
  }
  // ---- instances whose series diverged: the GMRES of App. C, one context at a
  //      time (unless the context asked for the series alone) ----
  for (int k = 0; k < n; ++k) {
    Inst& X = I[k];
    dyson_ctx* c = X.c;
    if (X.status != DYSON_ERR_DIVERGED || c->inner_solver == DYSON_INNER_SERIES) continue;
    const int saved = c->inner_solver;
    c->inner_solver = DYSON_INNER_GMRES;
    double2* G = nullptr;
    if ((rc = prepare_tables(c, DYSON_PREC_TF32X3_F64REF, tol, 0, false, true))) return bfail(b, rc, c->err);
    rc = solve_mixed(c, X.ncol, c->Nc, DYSON_PREC_TF32X3_F64REF, tol, max_sweeps, &G, &X.rep);
    c->inner_solver = saved;
    if (rc != DYSON_OK && rc != DYSON_ERR_NOT_CONVERGED && rc != DYSON_ERR_DIVERGED) return bfail(b, rc, c->err);
    X.status = rc;
    X.G = G;
  }
  // ---- observables and optional export per instance ----
  int status = DYSON_OK;
  const double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  for (int k = 0; k < n; ++k) {
    Inst& X = I[k];
    dyson_ctx* c = X.c;
    launch_observables(X.G, c->d_src_site, X.nq, c->d_nbr, c->d_nbond, c->dJ, c->d_eps, c->dU, c->Nr, c->Nt, c->Nc,
                       X.ncol, c->dt, c->d_obs, c->stream);
    c->launches += 1;
    if (g_out && g_out[k]) {
      launch_export(X.G, c->Nr, c->Nc, X.nq, (double2*)g_out[k], c->stream);
      c->launches += 1;
    }
    if (X.status != DYSON_OK && status == DYSON_OK) status = X.status;
    X.rep.status = X.status;
    X.rep.chunks = 1;
    X.rep.seconds = secs;
    X.rep.kernel_launches = c->launches - X.launches0;
    if (reports) reports[k] = X.rep;
  }
  DYB_CUDA(b, cudaGetLastError());
  DYB_CUDA(b, cudaStreamSynchronize(b->stream));
  if (status == DYSON_ERR_NOT_CONVERGED) b->err = "an instance reached its refinement limit above tolerance";
  if (status == DYSON_ERR_DIVERGED) b->err = "an instance's series diverged";
  return status;
}

int64_t dyson_batch_launch_count(const dyson_batch* b) { return b ? b->launches : -1; }

const char* dyson_batch_last_error(const dyson_batch* b) { return b ? b->err.c_str() : ""; }

void dyson_batch_destroy(dyson_batch* b) {
  if (!b) return;
  DeviceGuard g(b->device);
  for (cudaStream_t l : b->lane)
    if (l) {
      cudaStreamSynchronize(l);
      cudaStreamDestroy(l);
    }
  if (b->ready) cudaEventDestroy(b->ready);
  delete b;
}

}  // extern "C"
