// FP64 series sweep and FP64 Dyson residual on the BF16 tensor cores (slice-split products).
#pragma once
#include "common.cuh"

// true when the split-product FP64 sweep can serve this context: its slices of Lambda exist or
// fit in a third of the device memory that is free or scratch (it takes every contour length); *more: bytes
// that oz64_prepare would allocate
bool oz64_usable(dyson_ctx* c, size_t* more);
// X slices for ncol columns (oz64_sweep makes them where they are missing); bytes held by them; give them back
int oz64_reserve(dyson_ctx* c, int ncol);
size_t oz64_x_bytes(const dyson_ctx* c);
void oz64_release_x(dyson_ctx* c);
// device bytes of the X slices per complex state element
double oz64_bytes_per_element(const dyson_ctx* c);
// forget the Lambda slices (after Lambda changed)
void oz64_invalidate(dyson_ctx* c);
// build the Lambda slices now (so that the free memory a caller sizes its chunk by is what is left)
int oz64_prepare(dyson_ctx* c);
// mode 0: out = B + K Gin, c->d_norm[q] = max |out - Gin| (complex modulus; 24 bits, relative to the scale
// c->d_norm[ncol / gs + q]);
// mode 1: r32 = B + K Gin - Gin (FP32 planar of stride c->Ns; only the Nc points are written), c->d_norm[q] = max |r|.
// Groups of gs columns as launch_sweep_f64; two kernel launches, counted on the context.
int oz64_sweep(dyson_ctx* c, int ncol, int gs, const double2* Gin, double2* out, float* r32, int mode,
               const int* run = nullptr);
// DYSON_ERR_TIMEOUT if a bounded pipeline wait of an earlier sweep expired (clears the flag);
// synchronises.  Such a sweep also leaves norm word 0 infinite: to be asked where a norm is.
int oz64_check_error(dyson_ctx* c);
// out[b][u][t] = sum_{i < nk} X[b][i][u] A[b][i][t] (complex128, t, u < Nc) for b < batch, as accurate as
// the sweep; DYSON_ERR_OOM (no message) where the slices' scratch does not fit.  Synchronises.
int oz64_batched_product(dyson_ctx* c, int batch, int nk, int Nc, const double2* A, const double2* X, double2* out);
int oz64_set_wait_limit(dyson_ctx* c, unsigned long long ns);
void oz64_release(dyson_ctx* c);
