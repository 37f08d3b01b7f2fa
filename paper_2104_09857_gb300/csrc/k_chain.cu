// FP64 kernels of the screening chain between chi(i tau) and W^c(i tau):
// cosine transforms (weighted sums over the time or frequency grid) and the
// Cholesky factorisation with its triangular solve; the dense products are
// k_emu.cu's.
//
// Everything is FP64: the transform weights are large and of both signs (the
// sums cancel), and the factorisation of eps needs the precision.  Row-major
// n x n matrices throughout.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "k_chain.h"
#include "k_emu.h"

namespace gw {
namespace chain {

// out[e] = sum_j w[j] * in[j][e]   (fixed j order)
__global__ void k_lincomb(const double* __restrict__ in, int nin, const double* __restrict__ w, long long n,
                          double* __restrict__ out) {
  long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  for (; e < n; e += stride) {
    double acc = 0.0;
    for (int j = 0; j < nin; ++j) acc = fma(w[j], in[static_cast<long long>(j) * n + e], acc);
    out[e] = acc;
  }
}

// One 32 x 32 tile of the lower triangle and its mirror per CTA: the tile is
// read once and added into both places of every output matrix.
__global__ void __launch_bounds__(256) k_add_symmetric(const double* __restrict__ w, const double* __restrict__ v,
                                                       const double* __restrict__ d, int ldd, int nout, int n,
                                                       double* __restrict__ out) {
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double t[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + tx;
    if (r < n && c <= r) {
      const long long e = static_cast<long long>(r) * n + c;
      t[i][tx] = w[e] - v[e];
    }
  }
  __syncthreads();
  const long long nn = static_cast<long long>(n) * n;
  const bool diag = r0 == c0;
  for (int i = ty; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + tx;
    const bool on = r < n && c < n;
    const double x = on ? (diag && tx > i ? t[tx][i] : t[i][tx]) : 0.0;
    const int rm = c0 + i, cm = r0 + tx;  // the mirrored tile, row by row
    const bool onm = !diag && rm < n && cm < n;
    const double xm = onm ? t[tx][i] : 0.0;
    for (int j = 0; j < nout; ++j) {
      const double f = d[static_cast<long long>(j) * ldd];
      double* o = out + j * nn;
      if (on) o[static_cast<long long>(r) * n + c] += f * x;
      if (onm) o[static_cast<long long>(rm) * n + cm] += f * xm;
    }
  }
}

__global__ void k_add_diagonal(double* __restrict__ a, int n, double x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[static_cast<long long>(i) * n + i] += x;
}

__global__ void k_set_identity(double* __restrict__ a, int n) {
  long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long nn = static_cast<long long>(n) * n;
  if (i < nn) a[i] = (i / n == i % n) ? 1.0 : 0.0;
}

// ---------------------------------------------------------------------------
// Cholesky
// ---------------------------------------------------------------------------
// Blocks of 64 columns in two steps of 32.  A step factors the 32 x 32
// diagonal block, then solves for the rows below; the first 32 columns are
// applied to the other 32 on the FP64 pipe, the 64 then to everything to their
// right as one product of the digit engine.  Several matrices go through the
// sweep together (blockIdx.z): at the sizes where it matters the chain of
// small dependent kernels is what takes the time, not their work.  The FP64
// pipe of an SM quarter takes 64 cycles for one warp-wide operation, so every
// phase spreads its work over the four warps of a CTA and over many CTAs:
// with one warp per diagonal block and a row per thread a step took 88 us.
// 64 columns and not 128: the FP64 work inside a block grows with its width
// (rows x 32 x 32 multiply-adds here, six times that at 128).
constexpr int kNb = 32;
constexpr int kOuter = 2 * kNb;

// Cholesky factor of the b x b diagonal block at (k0, k0) of every matrix, to
// fac[k0 * 32..] (row-major, pitch 32) and the reciprocals of its diagonal to
// fac[(n + 32) * 32 + k0..].  One CTA per matrix; formed by every CTA of the
// solve below instead, the CTAs of an SM would queue for its FP64 pipe.  The
// columns of the block are scaled by rsqrt (one unit in the last place), a
// square root and a division per pivot would lie on the serial chain; the
// diagonal and its reciprocals are rounded roots and quotients, taken for all
// pivots at once at the end.
__global__ void __launch_bounds__(128) k_chol_factor(const double* __restrict__ a0, int n, long long z_stride, int k0,
                                                     int b, double* __restrict__ fac0, long long fac_z,
                                                     int* __restrict__ err) {
  __shared__ double d[kNb][kNb + 1];
  __shared__ double piv[kNb];
  const double* a = a0 + blockIdx.x * z_stride;
  double* fac = fac0 + blockIdx.x * fac_z;
  double* rd = fac + (static_cast<long long>(n) + kNb) * kNb + k0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kNb * kNb; i += blockDim.x) {
    const int r = i >> 5, c = i & 31;
    d[r][c] = (r < b && c <= r) ? a[static_cast<long long>(k0 + r) * n + k0 + c] : (r == c ? 1.0 : 0.0);
  }
  __syncthreads();
  bool bad = false;
  for (int j = 0; j < b; ++j) {
    double p = d[j][j];
    if (!(p > 0.0) || !isfinite(p)) {
      bad = true;
      p = 1.0;
    }
    const double y = rsqrt(p);
    if (warp == 0) {
      if (lane > j) d[lane][j] *= y;
      if (lane == j) piv[j] = p;
    }
    __syncthreads();
    const double l = d[lane][j];
    for (int c = j + 1 + warp; c < b; c += 4)
      if (lane >= c) d[lane][c] = fma(-l, d[c][j], d[lane][c]);
    __syncthreads();
  }
  if (bad && threadIdx.x == 0) atomicOr(err, 1);
  if (warp == 0 && lane < b) {
    const double r = sqrt(piv[lane]);
    d[lane][lane] = r;
    rd[lane] = 1.0 / r;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kNb * kNb; i += blockDim.x)
    fac[static_cast<long long>(k0) * kNb + i] = d[i >> 5][i & 31];
}

// Rows i >= k0 + b: a[i][k0:k0+b] <- a[i][k0:k0+b] D^-T, D the factor.  32
// rows per CTA, 8 per warp, a row on four lanes that hold every fourth column.
__global__ void __launch_bounds__(128) k_chol_solve(double* __restrict__ a0, long long rows, int n, long long z_stride,
                                                    int k0, int b, const double* __restrict__ fac0, long long fac_z) {
  __shared__ double d[kNb][kNb + 1];
  __shared__ double rd[kNb];
  double* a = a0 + blockIdx.z * z_stride;
  const double* fac = fac0 + blockIdx.z * fac_z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kNb * kNb; i += blockDim.x)
    d[i >> 5][i & 31] = fac[static_cast<long long>(k0) * kNb + i];
  if (threadIdx.x < b) rd[threadIdx.x] = fac[(static_cast<long long>(n) + kNb) * kNb + k0 + threadIdx.x];
  // this thread's part of a row: columns g, g + 4, ...
  const long long row = k0 + b + static_cast<long long>(blockIdx.x) * kNb + warp * 8 + (lane >> 2);
  const int g = lane & 3;
  double x[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = (row < rows && g + 4 * i < b) ? a[row * n + k0 + g + 4 * i] : 0.0;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kNb; ++j) {
    if (j >= b) break;
    if (g == (j & 3)) x[j >> 2] *= rd[j];
    const double xj = __shfl_sync(0xffffffffu, x[j >> 2], (lane & ~3) | (j & 3));
#pragma unroll
    for (int i = j >> 2; i < 8; ++i)
      if (g + 4 * i > j) x[i] = fma(-xj, d[g + 4 * i][j], x[i]);
  }
  if (row < rows)
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (g + 4 * i < b) a[row * n + k0 + g + 4 * i] = x[i];
}

// a[r][c] -= sum_{t < 32} a[r][k0 + t] a[c][k0 + t] for rows r >= c0 and the
// columns c of [c0, c1), c1 - c0 <= 32: 16 x 32 tiles (small, so that the FP64
// pipes of all SMs take part), nothing above the diagonal.
__global__ void __launch_bounds__(128) k_chol_update(double* __restrict__ a0, long long rows, int n,
                                                     long long z_stride, int k0, int c0, int c1) {
  double* a = a0 + blockIdx.z * z_stride;
  const long long rb = c0 + static_cast<long long>(blockIdx.x) * 16;
  __shared__ double x[16][33], y[32][33];
  for (int i = threadIdx.x; i < 32 * 32; i += blockDim.x) {
    const int r = i >> 5, t = i & 31;
    if (r < 16) x[r][t] = rb + r < rows ? a[(rb + r) * n + k0 + t] : 0.0;
    y[r][t] = c0 + r < c1 ? a[static_cast<long long>(c0 + r) * n + k0 + t] : 0.0;
  }
  __syncthreads();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  double acc[4] = {};
#pragma unroll
  for (int t = 0; t < 32; ++t) {
    const double v = y[tx][t];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = fma(x[ty + 4 * i][t], v, acc[i]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long long r = rb + ty + 4 * i;
    const int c = c0 + tx;
    if (r < rows && c < c1 && r >= c) a[r * n + c] -= acc[i];
  }
}

// the factored diagonal blocks into place, zeros above the diagonal
__global__ void k_chol_finish(double* __restrict__ a0, int n, long long z_stride, const double* __restrict__ fac0,
                              long long fac_z) {
  double* a = a0 + blockIdx.z * z_stride;
  const double* fac = fac0 + blockIdx.z * fac_z;
  long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long nn = static_cast<long long>(n) * n;
  if (i >= nn) return;
  const int r = static_cast<int>(i / n), c = static_cast<int>(i % n);
  if (c > r)
    a[i] = 0.0;
  else if (c / kNb == r / kNb)
    a[i] = fac[static_cast<long long>(c / kNb * kNb) * kNb + (r % kNb) * kNb + c % kNb];
}

}  // namespace chain

namespace {
inline unsigned blocks_for(long long n, int threads, long long cap = 152LL * 16) {
  long long b = (n + threads - 1) / threads;
  if (b > cap) b = cap;
  return static_cast<unsigned>(b < 1 ? 1 : b);
}
}  // namespace

void chain_lincomb(const double* in, int nin, const double* w, long long n, double* out, cudaStream_t st) {
  chain::k_lincomb<<<blocks_for(n, 256), 256, 0, st>>>(in, nin, w, n, out);
}

void chain_add_symmetric(const double* w, const double* v, const double* d, int ldd, int nout, int n, double* out,
                         cudaStream_t st) {
  const unsigned t = (n + 31) / 32;
  chain::k_add_symmetric<<<dim3(t, t), 256, 0, st>>>(w, v, d, ldd, nout, n, out);
}

void chain_add_diagonal(double* a, int n, double x, cudaStream_t st) {
  chain::k_add_diagonal<<<(n + 255) / 256, 256, 0, st>>>(a, n, x);
}

void chain_set_identity(double* a, int n, cudaStream_t st) {
  const long long nn = static_cast<long long>(n) * n;
  chain::k_set_identity<<<static_cast<unsigned>((nn + 255) / 256), 256, 0, st>>>(a, n);
}

int chain_cholesky(gw_ctx* ctx, double* a, long long rows, int n, int nz, long long z_stride, int* err,
                   cudaStream_t st) {
  void* p;
  int rc;
  const long long fac_z = (static_cast<long long>(n) + chain::kNb) * (chain::kNb + 1);
  if ((rc = work_buffer(ctx, "w.chol.fac", static_cast<size_t>(fac_z) * nz * sizeof(double), &p))) return rc;
  double* fac = static_cast<double*>(p);
  for (int k0 = 0; k0 < n; k0 += chain::kOuter) {
    const int k1 = std::min(n, k0 + chain::kOuter);
    for (int j0 = k0; j0 < k1; j0 += chain::kNb) {
      const int b = std::min(chain::kNb, k1 - j0);
      const long long below = rows - j0 - b;
      chain::k_chol_factor<<<nz, 128, 0, st>>>(a, n, z_stride, j0, b, fac, fac_z, err);
      if (below > 0)
        chain::k_chol_solve<<<dim3(static_cast<unsigned>((below + 31) / 32), 1, nz), 128, 0, st>>>(
            a, rows, n, z_stride, j0, b, fac, fac_z);
      if (j0 + b < k1)
        chain::k_chol_update<<<dim3(static_cast<unsigned>((below + 15) / 16), 1, nz), 128, 0, st>>>(
            a, rows, n, z_stride, j0, j0 + b, k1);
    }
    if (k1 < n) {
      // a[k1:, k1:n] -= X X^T, X = a[k1:, k0:k1]
      EmuOp x, y;
      EmuSrc s;
      s.src = a + static_cast<long long>(k1) * n + k0;
      s.ld = n;
      s.rows = rows - k1;
      s.K = k1 - k0;
      s.nz = nz;
      s.z_stride = z_stride;
      if ((rc = emu_prep(ctx, "panel", s, &x, st))) return rc;
      y = x;
      y.s.rows = n - k1;
      EmuGemm g;
      g.alpha = -1.0;
      g.beta = 1.0;
      g.C = a + static_cast<long long>(k1) * n + k1;
      g.ldc = n;
      g.c_zstride = z_stride;
      g.tri = 1;
      if ((rc = emu_mm(ctx, x, y, g, st))) return rc;
    }
  }
  const long long nn = static_cast<long long>(n) * n;
  chain::k_chol_finish<<<dim3(static_cast<unsigned>((nn + 255) / 256), 1, nz), 256, 0, st>>>(a, n, z_stride, fac,
                                                                                          fac_z);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    ctx->err = std::string("Cholesky factorisation: ") + cudaGetErrorString(e);
    return GW_ERR_CUDA;
  }
  return GW_OK;
}

}  // namespace gw
