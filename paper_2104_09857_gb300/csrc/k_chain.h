// Launchers of the FP64 screening-chain kernels (k_chain.cu).
#pragma once

#include <cuda_runtime.h>

#include "gw_internal.h"

namespace gw {

// out[e] = sum_j w[j] in[j][e], n elements per matrix
void chain_lincomb(const double* in, int nin, const double* w, long long n, double* out, cudaStream_t st);
// x = w - v on the lower triangles of two n x n matrices, taken as symmetric:
// out[j] += d[j * ldd] x for j < nout, both triangles of out written
void chain_add_symmetric(const double* w, const double* v, const double* d, int ldd, int nout, int n, double* out,
                         cudaStream_t st);
// a[i][i] += x
void chain_add_diagonal(double* a, int n, double x, cudaStream_t st);
// a = identity
void chain_set_identity(double* a, int n, cudaStream_t st);
// a[rows][n], rows >= n: the leading n x n block (its lower triangle is read)
// becomes its Cholesky factor R, the rows below become B R^-T; the strict
// upper triangle of the leading block is zeroed.  nz such matrices z_stride
// elements apart in one sweep.  err[0] |= 1 on a pivot that is not positive.
// Uses the context's work buffers (emu_begin before).
int chain_cholesky(gw_ctx* ctx, double* a, long long rows, int n, int nz, long long z_stride, int* err,
                   cudaStream_t st);

}  // namespace gw
