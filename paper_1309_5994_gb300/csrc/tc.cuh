// Tensor-core (tcgen05) sweep: interface used by the host driver.
#pragma once
#include <cuda.h>

#include "common.cuh"

// Arguments of a fused sweep (a kernel parameter).
struct FusedInst {
  const float* r;                    // right-hand side of the series [Nr][ncol][2 Ns] (nullptr: 0)
  const float* din;                  // the two FP32 states
  float* dout;
  const float* Jz;                   // [Nb][Ns] hopping on the contour
  const int* nbr;                    // [Nr][4] neighbour sites (-1: none)
  const int* nbond;                  // [Nr][4] bond of each neighbour slot
  unsigned long long* norm;          // update max-norm per group of gs columns
  const float* adown;                // [Nr][2 Ns] inverse row scales of the FP16 Lambda
  TcScale* sc;                       // scales per group of gs columns
  const int* rsrc;                   // r is non-zero only where column n has its source (site rsrc[n]); or nullptr
  const int* act;                    // support truncation table; or nullptr
  int Lx, Ly, Ns, ncol, gs;
};

// Contour points a column of the FP32 planar state holds, Ns: Nc rounded up to 64 (the rest are
// zeros) on the tensor-core sweeps
int contour_stride(const dyson_ctx* c);

// FP16 scales of the fused sweep: before the first sweep of a chain, seed the bound on |d_in| per
// column group, with ref (device, [ng]) or one bound for all, or by reading the state; the
// sweeps after it take the bound from the maxima that the previous one left.
int tc_seed_scale(dyson_ctx* c, int ng, const double* ref, double bound);
int tc_seed_scale_scan(dyson_ctx* c, int ncol, int gs, const float* d);
// turn the seeded maxima into scales (tc_sweep does this itself outside a batch of sweeps)
int tc_set_scale(dyson_ctx* c, int ng);
float tc_jbound(const dyson_ctx* c);              // 4 max|J|, the factor of set_scale
// true when a tcgen05 sweep serves this context
bool tc_supported(dyson_ctx* c);
// true when tc_sweep runs the CTA-pair (cta_group::2) kernel for this context
bool tc_uses_pair(dyson_ctx* c);
// true when tc_sweep runs the fused gather + GEMM kernel (k_tc_fused) for this context: unless
// its variant is DYSON_SWEEP_SINGLE_CTA or DYSON_SWEEP_CTA_PAIR and Nc a multiple of 64;
// TC_GATHER alone then launches nothing
bool tc_uses_fused(dyson_ctx* c);
// tensor maps and buffers of tc_sweep (fused: of tc_fused_sweep) for ncol columns, set up ahead of
// a stream capture
int tc_prepare_sweep(dyson_ctx* c, int ncol, bool fused = false);
// one sweep d_out = r + K d_in over the FP32 planar chunk state of ncol vector columns;
// writes c->d_norm[q] for groups of gs columns (unfused forms: gs a multiple of 32).
// phases: TC_GATHER launches X = J d_in, TC_GEMM launches the tensor-core product and
// epilogue (in that order; both = one whole sweep).
// act (optional, device [Nr][ceil(ncol / 256)]): support truncation (App. C, Sec. IV.D):
// the first sweep at which each (site, 256-column tile) can be non-zero; tiles with
// act > sweep are skipped, so their d_out must already hold zeros.
// rform: what the caller knows of r, for the fused kernel to skip loads of zeros:
// TC_R_DENSE (general), TC_R_ZERO (r = 0: a matvec), TC_R_ON_SOURCES (r non-zero only
// on the rows of each column's source site, c->d_src_site: the first right-hand side)
enum { TC_GATHER = 1, TC_GEMM = 2 };
enum { TC_R_DENSE = 0, TC_R_ZERO = 1, TC_R_ON_SOURCES = 2 };
constexpr int TC_TILE_COLS = 256;
int tc_sweep(dyson_ctx* c, int ncol, int gs, const float* r, const float* d_in, float* d_out, int phases,
             const int* act = nullptr, int sweep = 0, int rform = TC_R_DENSE);
// DYSON_ERR_TIMEOUT if a bounded pipeline wait of an earlier sweep expired (clears the flag);
// synchronises the context's stream
int tc_check_error(dyson_ctx* c);
// the same in two halves around a synchronisation the caller makes anyway: enqueue the
// copy of the flag to pinned host memory, then, after the stream has synchronised, read it
int tc_error_enqueue(dyson_ctx* c);
// time limit (ns) of the pipeline waits of this file's kernels on the context's device
int tc_set_wait_limit(dyson_ctx* c, unsigned long long ns);
int tc_error_status(dyson_ctx* c);
// bytes held by the unfused forms' gather buffer; give it back
size_t tc_x_bytes(const dyson_ctx* c);
void tc_release_x(dyson_ctx* c);
// free tensor-core module state
void tc_release(dyson_ctx* c);

// true when the fused sweep can run on this context's device
bool tc_fused_runs(dyson_ctx* c);
// The fused sweep of tc_sweep on a stream of the caller's, with scales set (tc_set_scale, or by a
// check kernel): run (or nullptr): device flag, 0 skips the sweep; sweeps_done (or nullptr):
// device count that gives the sweep number
int tc_fused_sweep(dyson_ctx* c, int ncol, int gs, const float* r, const float* din, float* dout, const int* act,
                   int sweep, int rform, const int* run, const int* sweeps_done, cudaStream_t stream);
