// CUDA-core kernels of the chi(i tau) path: 3c block norms and panel build,
// Green's functions (Eq. 2), the two brackets of Eq. 3 as grouped panel
// GEMMs (steps A and B), the block filter of the intermediates, per-tile task
// lists, the step-C contraction in FP64 and FP32, and the final mirror.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "gw_internal.h"
#include "k_simt.h"

#include <cooperative_groups.h>

namespace gw {

// ---------------------------------------------------------------------------
// three-centre tensor: per-block Frobenius norm, finiteness, symmetry of
// (A, A, P) blocks
// ---------------------------------------------------------------------------
__global__ void k_block_norms_3c(const double* __restrict__ t3, long long base_off,
                                 const int* __restrict__ blk, const long long* __restrict__ off,
                                 const int* __restrict__ n_ao, const int* __restrict__ n_ri,
                                 long long n_blocks, double* __restrict__ norms, int* __restrict__ bad) {
  long long b = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  int lane = threadIdx.x & 31;
  if (b >= n_blocks) return;
  const double* x = t3 + (off[b] - base_off);
  long long n = off[b + 1] - off[b];
  double s = 0.0;
  bool nonfinite = false;
  for (long long i = lane; i < n; i += 32) {
    double v = x[i];
    if (!isfinite(v)) nonfinite = true;
    s += v * v;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  unsigned nf = __ballot_sync(0xffffffffu, nonfinite);
  int a = blk[3 * b], bb = blk[3 * b + 1], p = blk[3 * b + 2];
  bool asym = false;
  if (a == bb) {
    int na = n_ao[a], np = n_ri[p];
    double mx = 0.0, md = 0.0;
    for (long long i = lane; i < n; i += 32) {
      int pl = (int)(i % np);
      long long r = i / np;
      int j = (int)(r % na), k = (int)(r / na);
      double v = x[i];
      double w = x[((long long)j * na + k) * np + pl];
      mx = fmax(mx, fabs(v));
      md = fmax(md, fabs(v - w));
    }
    for (int o = 16; o > 0; o >>= 1) {
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
    }
    asym = md > 1e-12 * mx;
  }
  if (lane == 0) {
    norms[b] = sqrt(s);
    if (nf) atomicOr(bad, 1);
    if (asym) atomicOr(bad, 2);
  }
}

// Scatter the kept A <= B blocks into the owner panels:
//   block (A, B, p) -> panel(B) rows of A (value blk[a][b][P]),
//                      panel(A) rows of B (value blk[a][b][P]) if A != B.
__global__ void k_panel_scatter(const double* __restrict__ t3, const int* __restrict__ blk,
                                const long long* __restrict__ off, const int* __restrict__ n_ao,
                                const int* __restrict__ n_ri, const int* __restrict__ ri_off,
                                const int* __restrict__ kept_idx, int n_kept,
                                const long long* __restrict__ dstB, const long long* __restrict__ dstA,
                                const int* __restrict__ ldB, const int* __restrict__ ldA,
                                double* __restrict__ pool) {
  int kb = blockIdx.x;
  if (kb >= n_kept) return;
  int b = kept_idx[kb];
  int A = blk[3 * b], B = blk[3 * b + 1], p = blk[3 * b + 2];
  int na = n_ao[A], nb = n_ao[B], np = n_ri[p];
  const double* x = t3 + off[b];
  long long n = (long long)na * nb * np;
  // dstB[kb]: element offset of (row of alpha = 0, pw = ri_off[p] - p0(B), s' = 0)
  // in panel(B); row stride ldB = npw(B) * nb.
  for (long long i = threadIdx.x; i < n; i += blockDim.x) {
    int pl = (int)(i % np);
    long long r = i / np;
    int be = (int)(r % nb), al = (int)(r / nb);
    double v = x[i];
    pool[dstB[kb] + (long long)al * ldB[kb] + (long long)pl * nb + be] = v;
    if (A != B) pool[dstA[kb] + (long long)be * ldA[kb] + (long long)pl * na + al] = v;
  }
}

__global__ void k_cast_f64_f32(const double* __restrict__ x, float* __restrict__ y, long long n) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long stride = (long long)gridDim.x * blockDim.x;
  for (; i < n; i += stride) y[i] = (float)x[i];
}

// ---------------------------------------------------------------------------
// Eq. 2: scaled orbital columns.  occupied: C[mu][i] exp((eps_i - mu_F) tau/2),
// virtual: C[mu][a] exp(-(eps_a - mu_F) tau/2); G = Cs Cs^T.
// ---------------------------------------------------------------------------
// One exponential per column and CTA: an FP64 exponential is some 25 operations
// on the FP64 pipe, and one per element took 18 us at 602 functions.
__global__ void __launch_bounds__(256) k_scale_orbitals(const double* __restrict__ C, const double* __restrict__ eps,
                                                        int nao, int n_occ, double mu, double tau,
                                                        double* __restrict__ cso, double* __restrict__ csv) {
  __shared__ double f[32];
  const int col = blockIdx.x * 32 + (threadIdx.x & 31);
  if (threadIdx.x < 32 && col < nao) {
    const double e = eps[col] - mu;
    f[threadIdx.x] = col < n_occ ? exp(0.5 * e * tau) : exp(-0.5 * e * tau);
  }
  __syncthreads();
  if (col >= nao) return;
  const double w = f[threadIdx.x & 31];
  const int nv = nao - n_occ;
  for (int row = blockIdx.y * 8 + (threadIdx.x >> 5); row < nao; row += 8 * gridDim.y) {
    const double v = C[static_cast<long long>(row) * nao + col] * w;
    if (col < n_occ)
      cso[static_cast<long long>(row) * n_occ + col] = v;
    else
      csv[static_cast<long long>(row) * nv + (col - n_occ)] = v;
  }
}

// Frobenius norms of the (A <= B) atom blocks of two symmetric matrices
// (blockIdx.y); blocks with norm < thr are zeroed together with their mirror.
// flags[A*n+B] = flags[B*n+A] = kept.  A warp per block: blocks are a few
// hundred elements, and a CTA for each (and for each mirror) took 16 us at 58
// atoms where this takes 3.
__global__ void __launch_bounds__(256) k_sym_block_filter(double* __restrict__ g0, double* __restrict__ g1, int nao,
                                                          const int* __restrict__ ao_off, int n_at, double thr,
                                                          unsigned char* __restrict__ f0,
                                                          unsigned char* __restrict__ f1) {
  double* g = blockIdx.y ? g1 : g0;
  unsigned char* flags = blockIdx.y ? f1 : f0;
  const int lane = threadIdx.x & 31;
  const long long pair = static_cast<long long>(blockIdx.x) * 8 + threadIdx.x / 32;
  if (pair >= static_cast<long long>(n_at) * n_at) return;
  const int A = static_cast<int>(pair / n_at), B = static_cast<int>(pair % n_at);
  if (A > B) return;
  const int a0 = ao_off[A], na = ao_off[A + 1] - a0;
  const int b0 = ao_off[B], nb = ao_off[B + 1] - b0;
  double s = 0.0;
  for (int i = lane; i < na * nb; i += 32) {
    const double v = g[(long long)(a0 + i / nb) * nao + b0 + i % nb];
    s += v * v;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const bool keep = !(sqrt(s) < thr);
  if (lane == 0) {
    flags[(long long)A * n_at + B] = keep;
    flags[(long long)B * n_at + A] = keep;
  }
  if (!keep) {
    for (int i = lane; i < na * nb; i += 32) {
      g[(long long)(a0 + i / nb) * nao + b0 + i % nb] = 0.0;
      g[(long long)(b0 + i % nb) * nao + a0 + i / nb] = 0.0;
    }
  }
}

// ---------------------------------------------------------------------------
// CUDA-core tile GEMM, both operands K-major:
//   C[m][n] += alpha * sum_{k in runs} A[m][k] * B[n][k]
// 64 x 64 tile, 256 threads, thread (tx, ty) owns rows ty + 16 i and columns
// tx + 16 j (i, j < 4).  Accumulation in AccT per run; runs are added into
// FP64 registers, so FP32 products are summed in FP32 within a run only.
// ---------------------------------------------------------------------------
template <typename T, typename AccT>
__device__ __forceinline__ void tile_nt_run(const T* __restrict__ A, long long lda, int mrows,
                                            const T* __restrict__ B, long long ldb, int nrows,
                                            long long k0, int klen, T (*As)[65], T (*Bs)[65],
                                            double (&acc64)[4][4]) {
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  AccT acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = AccT(0);
  for (int kk0 = 0; kk0 < klen; kk0 += 16) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int idx = tid + 256 * e;
      int row = idx >> 4, kk = idx & 15;
      bool kin = kk0 + kk < klen;
      As[kk][row] = (row < mrows && kin) ? A[(long long)row * lda + k0 + kk0 + kk] : T(0);
      Bs[kk][row] = (row < nrows && kin) ? B[(long long)row * ldb + k0 + kk0 + kk] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma((AccT)a[i], (AccT)b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc64[i][j] += (double)acc[i][j];
}

// G = Cs Cs^T for the occupied (blockIdx.z = 0) and virtual (1) orbitals:
// tiles on and above the diagonal are computed and also stored transposed, so
// G is exactly symmetric (inside a diagonal tile both halves use the same k
// order and commutative products).  16 x 16 tiles of 64 threads: two FMAs per
// cycle and SM is all there is, so a small G must spread over every SM (124
// functions: 72 CTAs of 6 us, where 64 x 64 tiles took 80 us on three SMs).
__global__ void __launch_bounds__(64) k_syrk64(const double* __restrict__ cso, const double* __restrict__ csv,
                                               int nao, int n_occ, double* __restrict__ go,
                                               double* __restrict__ gv) {
  if (blockIdx.x < blockIdx.y) return;
  const double* cs = blockIdx.z ? csv : cso;
  double* g = blockIdx.z ? gv : go;
  const int K = blockIdx.z ? nao - n_occ : n_occ;
  __shared__ double As[16][33], Bs[16][33];
  const int m0 = blockIdx.y * 16, n0 = blockIdx.x * 16;
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  double acc[2][2] = {};
  for (int k0 = 0; k0 < K; k0 += 32) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int row = (threadIdx.x >> 5) + 2 * e, kk = threadIdx.x & 31;
      const bool kin = k0 + kk < K;
      As[row][kk] = (kin && m0 + row < nao) ? cs[static_cast<long long>(m0 + row) * K + k0 + kk] : 0.0;
      Bs[row][kk] = (kin && n0 + row < nao) ? cs[static_cast<long long>(n0 + row) * K + k0 + kk] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk)
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[i][j] = fma(As[ty + 8 * i][kk], Bs[tx + 8 * j][kk], acc[i][j]);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int m = m0 + ty + 8 * i, n = n0 + tx + 8 * j;
      if (m < nao && n < nao) {
        g[static_cast<long long>(m) * nao + n] = acc[i][j];
        if (m0 != n0) g[static_cast<long long>(n) * nao + m] = acc[i][j];
      }
    }
}

// ---------------------------------------------------------------------------
// FP32: 64 x 64 tile, 64 threads; thread (tx, ty) owns rows 4 ty + i and
// 32 + 4 ty + i, columns 4 tx + j and 32 + 4 tx + j (i, j < 4), two products per
// instruction (fma.rn.f32x2).  Four 16-byte shared loads feed 64 multiply-adds,
// where the 4 x 4 tile of tile_nt_run needs eight 4-byte ones for 16: alone the
// loop runs at 63 TFLOP/s with 8 warps per SM (8 x 4 per thread: 55).  Per
// element the products enter one by one in the order of k, as there: the sums
// are the same to the bit.
// ---------------------------------------------------------------------------
constexpr int kF32K = 16;       // reduction elements per stage
constexpr int kF32Pitch = 68;   // floats per k row of a stage (16-byte aligned)
constexpr int kF32Threads = 64;
using F32Stage = float[kF32K][kF32Pitch];
using F32Acc = unsigned long long[4][8];

// column of row or column r of the tile in k row k: the swap of 8 columns keeps
// four k rows apart in the banks when a warp stores 4 consecutive k of 8 rows
__device__ __forceinline__ int f32_col(int k, int r) { return k & 8 ? r ^ 8 : r; }
__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
  return v;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
// row or column of the tile of a thread's element i (or j) < 8
__device__ __forceinline__ int f32_at(int t8, int i) { return (i & 4) * 8 + 4 * t8 + (i & 3); }
// acc[i][j]: row elements 2 i and 2 i + 1, column element j
__device__ __forceinline__ void f32_stage(const F32Stage& A, const F32Stage& B, int tx, int ty, F32Acc& acc) {
#pragma unroll
  for (int kk = 0; kk < kF32K; ++kk) {
    const int ca = f32_col(kk, 4 * ty), cb = f32_col(kk, 4 * tx);
    const float4 a0 = *reinterpret_cast<const float4*>(&A[kk][ca]);
    const float4 a1 = *reinterpret_cast<const float4*>(&A[kk][32 + ca]);
    const float4 b0 = *reinterpret_cast<const float4*>(&B[kk][cb]);
    const float4 b1 = *reinterpret_cast<const float4*>(&B[kk][32 + cb]);
    const unsigned long long av[4] = {pack2(a0.x, a0.y), pack2(a0.z, a0.w), pack2(a1.x, a1.y), pack2(a1.z, a1.w)};
    const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) fma2(acc[i][j], av[i], pack2(bv[j], bv[j]));
  }
}

// Step C in FP32: chi[P][Q] -= sum over the tile's slab list of X[P][k] Y[Q][k],
// each slab summed in FP32 and the slabs in FP64.  ldk and every slab's start
// and length are multiples of 64 elements.  A cluster shares a tile, each block
// a contiguous part of its slabs: 58 atoms have 272 tiles of work, less than two
// blocks per SM.  The FP64 sums stay in shared memory (64 of them would take 128
// registers of each thread).  58 atoms, 858 GFLOP: 61 ms in 4 x 4 tiles of one
// block, 25.8 with one stage of loads in flight, 22.3 with two.  What remains is
// the latency of those loads (a third of them miss the L2 cache) at 8 warps per SM.
// Clusters of 1, 2, 4 and 8, ms: 12-atom ring 0.92, 0.57, 0.29, 0.16; ribbons of 20
// atoms 2.96, 1.56, 0.93, 0.80, of 40 11.9, 9.0, 8.4, 6.5, of 58 37, 34, 21.1, 22.3,
// of 100 181, 151, 146, 150; 45-atom cluster 13.3, 9.7, 8.9, 7.2.  Eight loses 6 %
// at most where there are many tiles (shorter parts that end together keep the CTAs
// on the same slabs), so it is taken at every size.
constexpr int kF32Split = 8;
struct F32ChiShared {
  double sum[64][kF32Threads];  // element 8 i + j of each thread
  F32Stage a[2], b[2];
};
__global__ void __cluster_dims__(1, 1, kF32Split) __launch_bounds__(kF32Threads)
    k_chi_tiles_f32(const float* __restrict__ X, const float* __restrict__ Y, long long ldk, int P0, int prow, int nri,
                    const int* __restrict__ tasks, const int* __restrict__ counts, int max_slab, int nqt,
                    const long long* __restrict__ slab_k0, const int* __restrict__ slab_len,
                    double* __restrict__ chi) {
  extern __shared__ __align__(16) unsigned char f32_smem[];
  F32ChiShared& sm = *reinterpret_cast<F32ChiShared*>(f32_smem);
  const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank());
  const int tile = blockIdx.y * nqt + blockIdx.x;
  const int total = counts[tile];
  if (total == 0) return;  // the whole cluster
  const int p0 = blockIdx.y * 64, q0 = blockIdx.x * 64;
  const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
  // this thread fetches k 4 (t % 4) .. + 3 of rows t / 4 + 16 h
  const int fr = t >> 2, fk = (t & 3) * 4;
  const float* xr = X + static_cast<long long>(p0 + fr) * ldk + fk;
  const float* yr = Y + static_cast<long long>(q0 + fr) * ldk + fk;
  float4 f0[8], f1[8];
  auto fetch = [&](float4(&f)[8], long long k) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const long long o = k + 16 * h * ldk;
      f[h] = p0 + fr + 16 * h < prow ? *reinterpret_cast<const float4*>(xr + o) : make_float4(0.f, 0.f, 0.f, 0.f);
      f[4 + h] = q0 + fr + 16 * h < nri ? *reinterpret_cast<const float4*>(yr + o) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto put = [&](const float4(&f)[8], F32Stage& a, F32Stage& b) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int c = f32_col(fk, fr + 16 * h);
      a[fk][c] = f[h].x;
      a[fk + 1][c] = f[h].y;
      a[fk + 2][c] = f[h].z;
      a[fk + 3][c] = f[h].w;
      b[fk][c] = f[4 + h].x;
      b[fk + 1][c] = f[4 + h].y;
      b[fk + 2][c] = f[4 + h].z;
      b[fk + 3][c] = f[4 + h].w;
    }
  };
  const int first = static_cast<int>(static_cast<long long>(total) * rank / kF32Split);
  const int cnt = static_cast<int>(static_cast<long long>(total) * (rank + 1) / kF32Split) - first;
  const int* list = tasks + static_cast<long long>(tile) * max_slab + first;
#pragma unroll 8
  for (int e = 0; e < 64; ++e) sm.sum[e][t] = 0.0;
  if (cnt > 0) {
    const long long k0 = slab_k0[list[0]];
    fetch(f0, k0);
    fetch(f1, k0 + kF32K);
    put(f0, sm.a[0], sm.b[0]);
  }
  __syncthreads();
  for (int i = 0; i < cnt; ++i) {
    const long long k0 = slab_k0[list[i]];
    const int len = slab_len[list[i]];
    const long long next = i + 1 < cnt ? slab_k0[list[i + 1]] : -1;
    F32Acc acc = {};
    for (int kk = 0; kk < len; kk += 2 * kF32K) {
      // two stages on their way while this one is multiplied
      const long long k = kk + 2 * kF32K < len ? k0 + kk + 2 * kF32K : next;
      if (k >= 0) fetch(f0, k);
      f32_stage(sm.a[0], sm.b[0], tx, ty, acc);
      put(f1, sm.a[1], sm.b[1]);
      __syncthreads();
      if (k >= 0) fetch(f1, k + kF32K);
      f32_stage(sm.a[1], sm.b[1], tx, ty, acc);
      if (k >= 0) put(f0, sm.a[0], sm.b[0]);
      __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 v = unpack2(acc[a][j]);
        sm.sum[16 * a + j][t] += static_cast<double>(v.x);
        sm.sum[16 * a + 8 + j][t] += static_cast<double>(v.y);
      }
  }
  // the partial tiles, row element `rank` of every thread added up by this rank
  // in the order of the slabs
  cluster.sync();
  const int m = p0 + f32_at(ty, rank);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int n = q0 + f32_at(tx, j);
    double v = 0.0;
#pragma unroll
    for (int o = 0; o < kF32Split; ++o) v += *cluster.map_shared_rank(&sm.sum[8 * rank + j][t], o);
    if (m < prow && n < nri) chi[static_cast<long long>(P0 + m) * nri + n] -= v;
  }
  cluster.sync();  // no rank leaves while its tile is read
}

// Step C: chi[P][Q] -= sum over the tile's slab list of X[P][k] Y[Q][k].
// Tile (pt, qt) covers P in [P0 + 64 pt, ...) and Q in [64 qt, ...).
template <typename T, typename AccT>
__global__ void k_chi_tiles(const T* __restrict__ X, const T* __restrict__ Y, long long ldk, int P0,
                            int prow, int nri, const int* __restrict__ tasks,
                            const int* __restrict__ counts, int max_slab, int nqt,
                            const long long* __restrict__ slab_k0, const int* __restrict__ slab_len,
                            double* __restrict__ chi) {
  __shared__ T As[16][65];
  __shared__ T Bs[16][65];
  int pt = blockIdx.y, qt = blockIdx.x;
  int tile = pt * nqt + qt;
  int cnt = counts[tile];
  if (cnt == 0) return;
  int p0 = pt * 64, q0 = qt * 64;
  int mrows = min(64, prow - p0), nrows = min(64, nri - q0);
  double acc[4][4] = {};
  const int* list = tasks + (long long)tile * max_slab;
  for (int t = 0; t < cnt; ++t) {
    int s = list[t];
    tile_nt_run<T, AccT>(X + (long long)p0 * ldk, ldk, mrows, Y + (long long)q0 * ldk, ldk, nrows,
                         slab_k0[s], slab_len[s], As, Bs, acc);
  }
  int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int m = p0 + ty + 16 * i, n = q0 + tx + 16 * j;
      if (m < prow && n < nri) chi[(long long)(P0 + m) * nri + n] -= acc[i][j];
    }
}

// ---------------------------------------------------------------------------
// Steps A / B: grouped panel GEMM Z[r][n] = sum_k G[lam[k]][r] * panel[k][n],
// scattered into the K-major operands.
//   mode 0 (X, Eq. 3 first bracket, G = G^occ, r = mu over all AOs):
//     X[(p0 + pw - P0b) * ldk + seg + r * nsig + s']
//   mode 1 (Y, Eq. 3 second bracket, G = G^virt, r = sigma of the batch):
//     Y[(p0 + pw) * ldk + rowbase[r] + (aom + s') * rowmul[r]]
// with n = pw * nsig + s'.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_panel_gemm(const T* __restrict__ G, int nao, const T* __restrict__ pool,
                             const int* __restrict__ lam, const PanelTask* __restrict__ tasks,
                             int mode, int r0, int R, int P0b, long long ldk,
                             const long long* __restrict__ rowbase, const int* __restrict__ rowmul,
                             T* __restrict__ out) {
  __shared__ T As[16][65];
  __shared__ T Bs[16][65];
  const PanelTask tk = tasks[blockIdx.z];
  int n0 = blockIdx.x * 64, m0 = blockIdx.y * 64;
  if (n0 >= tk.N || m0 >= R) return;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const T* P = pool + tk.panel_off;
  const int* lk = lam + tk.lam_off;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
  for (int k0 = 0; k0 < tk.K; k0 += 16) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int idx = tid + 256 * e;
      int kk = idx >> 6, c = idx & 63;
      bool kin = k0 + kk < tk.K;
      int r = m0 + c;
      As[kk][c] = (kin && r < R) ? G[(long long)lk[k0 + kk] * nao + r0 + r] : T(0);
      int n = n0 + c;
      Bs[kk][c] = (kin && n < tk.N) ? P[(long long)(k0 + kk) * tk.N + n] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    int n = n0 + tx + 16 * j;
    if (n >= tk.N) continue;
    int pw = n / tk.nsig, sp = n - pw * tk.nsig;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int r = m0 + ty + 16 * i;
      if (r >= R) continue;
      long long dst;
      if (mode == 0) {
        dst = (long long)(tk.p0 + pw - P0b) * ldk + tk.seg + (long long)(r0 + r) * tk.nsig + sp;
      } else {
        dst = (long long)(tk.p0 + pw) * ldk + rowbase[r] + (long long)(tk.aom + sp) * rowmul[r];
      }
      out[dst] = acc[i][j];
    }
  }
}

// The same in FP32 on the tiles of f32_stage: rows r of G along the tile's rows,
// panel columns n along its columns.  The results pass through shared memory, so
// that a warp's stores run along the operand's memory: n in mode 0, r in mode 1.
// 58 atoms, 585 GFLOP: 24 ms in 4 x 4 tiles, 15.1 in these.
__global__ void __launch_bounds__(kF32Threads)
    k_panel_gemm_f32(const float* __restrict__ G, int nao, const float* __restrict__ pool, const int* __restrict__ lam,
                     const PanelTask* __restrict__ tasks, int mode, int r0, int R, int P0b, long long ldk,
                     const long long* __restrict__ rowbase, const int* __restrict__ rowmul, float* __restrict__ out) {
  __shared__ __align__(16) union {
    struct {
      F32Stage a[2], b[2];
    } st;
    float out[64][65];  // after the last stage
  } sm;
  const PanelTask tk = tasks[blockIdx.z];
  const int n0 = blockIdx.x * 64, m0 = blockIdx.y * 64;
  if (n0 >= tk.N || m0 >= R) return;
  const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
  // this thread fetches column t of every k row
  const bool rin = m0 + t < R, nin = n0 + t < tk.N;
  const float* g = G + r0 + m0 + t;
  const float* P = pool + tk.panel_off + n0 + t;
  const int* lk = lam + tk.lam_off;
  float fa[kF32K], fb[kF32K];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int e = 0; e < kF32K; ++e) {
      const int k = k0 + e;
      const bool kin = k < tk.K;
      fa[e] = (kin && rin) ? g[static_cast<long long>(lk[k]) * nao] : 0.f;
      fb[e] = (kin && nin) ? P[static_cast<long long>(k) * tk.N] : 0.f;
    }
  };
  auto put = [&](int s) {
#pragma unroll
    for (int e = 0; e < kF32K; ++e) {
      sm.st.a[s][e][f32_col(e, t)] = fa[e];
      sm.st.b[s][e][f32_col(e, t)] = fb[e];
    }
  };
  F32Acc acc = {};
  int s = 0;
  fetch(0);
  put(0);
  __syncthreads();
  for (int k0 = 0; k0 < tk.K; k0 += kF32K) {
    const bool more = k0 + kF32K < tk.K;
    if (more) fetch(k0 + kF32K);
    f32_stage(sm.st.a[s], sm.st.b[s], tx, ty, acc);
    if (more) put(s ^ 1);
    __syncthreads();
    s ^= 1;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float2 v = unpack2(acc[i][j]);
      sm.out[f32_at(ty, 2 * i)][f32_at(tx, j)] = v.x;
      sm.out[f32_at(ty, 2 * i + 1)][f32_at(tx, j)] = v.y;
    }
  __syncthreads();
  if (mode == 0) {
    if (!nin) return;
    const int n = n0 + t, pw = n / tk.nsig, sp = n - pw * tk.nsig;
    float* o = out + static_cast<long long>(tk.p0 + pw - P0b) * ldk + tk.seg + sp +
               static_cast<long long>(r0 + m0) * tk.nsig;
    const int mr = min(64, R - m0);
#pragma unroll 4
    for (int i = 0; i < mr; ++i) o[static_cast<long long>(i) * tk.nsig] = sm.out[i][t];
  } else {
    if (!rin) return;
    const int r = m0 + t;
    const long long base = rowbase[r];
    const int mul = rowmul[r];
    int pw = n0 / tk.nsig, sp = n0 - pw * tk.nsig;
    const int nr = min(64, tk.N - n0);
#pragma unroll 4
    for (int i = 0; i < nr; ++i) {
      out[static_cast<long long>(tk.p0 + pw) * ldk + base + static_cast<long long>(tk.aom + sp) * mul] = sm.out[t][i];
      if (++sp == tk.nsig) {
        sp = 0;
        ++pw;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Block filter of the intermediates and slab/tile occupancy.
// Block (m, s, p) of an operand buffer Z[row][k]: rows = RI functions of atom
// p (offset by rowoff), columns [seg(s) + ao(m) nsig(s), + n_ao(m) nsig(s)).
// Norm < thr -> zeroed.  Kept and nonzero -> flag byte of the block and of
// every (slab, row tile) it touches.
// ---------------------------------------------------------------------------
// |v| as FP32 within 2^-22, by integer operations (an FP64 conversion takes the
// SM quarter's FP64 pipe for 64 cycles per warp); below FP32's range 0.
__device__ __forceinline__ float magnitude(float v) { return fabsf(v); }
__device__ __forceinline__ float magnitude(double v) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(v)) & 0x7fffffffu;
  if (hi < 0x38100000u) return 0.f;
  if (hi >= 0x47f00000u) return INFINITY;
  return __uint_as_float(((hi - 0x38000000u) << 3) | (static_cast<unsigned>(__double2loint(v)) >> 29));
}

// One warp per block.  The norm is first taken in FP32 (a relative error below
// 1e-3 for blocks of up to 10^4 rows); only a block within 1 % of the threshold, one
// outside FP32's range or one with an Inf or NaN has it taken in FP64, so every decision is the FP64 one.
// In FP64 throughout, the kernel was bound by that pipe: 5.5 ms at 58 atoms, now 1.7.
template <typename T>
__global__ void k_operand_block_filter(T* __restrict__ Z, long long ldk, int rowoff,
                                       const int* __restrict__ ri_off, const int* __restrict__ ao_off,
                                       const int* __restrict__ n_ao, int s0, int ns,
                                       const long long* __restrict__ seg, int pa0, int npa, int n_at,
                                       double thr, int naop, unsigned char* __restrict__ blockflag,
                                       unsigned char* __restrict__ tileflag, int ntile,
                                       int tile_rows) {
  long long w = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  int lane = threadIdx.x & 31;
  long long nblk = (long long)ns * n_at * npa;
  if (w >= nblk) return;
  int pl = (int)(w % npa);
  long long t = w / npa;
  int m = (int)(t % n_at);
  int sl = (int)(t / n_at);
  int s = s0 + sl, p = pa0 + pl;
  int nsig = n_ao[s];
  int rows0 = ri_off[p] - rowoff, nrows = ri_off[p + 1] - ri_off[p];
  long long c0 = seg[sl] + (long long)ao_off[m] * nsig;
  int ncols = n_ao[m] * nsig;
  float sum = 0.f;
  bool any = false;
  for (int r = 0; r < nrows; ++r) {
    const T* row = Z + (long long)(rows0 + r) * ldk + c0;
    float part = 0.f;
#pragma unroll 4
    for (int c = lane; c < ncols; c += 32) {
      const T v = row[c];
      any = any || !(v == T(0));
      const float m = magnitude(v);
      part = fmaf(m, m, part);
    }
    sum += part;
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  any = __any_sync(0xffffffffu, any);
  const float t2 = (float)(thr * thr);
  bool kept, nz = false;
  if (!any) {
    kept = !(0.0 < thr);
  } else if (sum > fmaxf(1.01f * t2, 1e-30f) && sum < 1e37f) {
    kept = nz = true;
  } else if (t2 > 1e-30f && sum < 0.99f * t2) {
    kept = false;
  } else {
    double acc = 0.0;
    for (int r = 0; r < nrows; ++r) {
      const T* row = Z + (long long)(rows0 + r) * ldk + c0;
      for (int c = lane; c < ncols; c += 32) {
        const double v = (double)row[c];
        acc += v * v;
      }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const double nrm = sqrt(acc);
    kept = !(nrm < thr);
    nz = kept && nrm > 0.0;
  }
  if (!kept) {
    for (int r = 0; r < nrows; ++r) {
      T* row = Z + (long long)(rows0 + r) * ldk + c0;
      for (int c = lane; c < ncols; c += 32) row[c] = T(0);
    }
  }
  if (lane == 0) blockflag[w] = nz;
  if (nz) {
    // flag (sigma-atom, mu-atom, tile) for every tile the block's rows touch
    int ts = rows0 / tile_rows, te = (rows0 + nrows - 1) / tile_rows;
    for (int tt = ts + lane; tt <= te; tt += 32) tileflag[((long long)sl * n_at + m) * ntile + tt] = 1;
    (void)naop;
  }
}

// Task list per (P tile, Q tile): slabs whose X part touches the P tile and
// whose Y part touches the Q tile.  Tiles entirely below the atom-block
// diagonal (atom(first P) > atom(last Q)) get no tasks.
__global__ void k_build_tasks(const unsigned char* __restrict__ fx, const unsigned char* __restrict__ fy,
                              int nslab, int npt, int nqt, int P0, int prow, int Q0, int qrow,
                              const int* __restrict__ atom_of_ri, const int* __restrict__ slab_len,
                              int* __restrict__ tasks, int* __restrict__ counts,
                              long long* __restrict__ kacc, int tile_rows, int tile_cols, int per,
                              int m0, int nmc, int mu0, int nmu, const int* __restrict__ atom_of_ao) {
  int tile = blockIdx.x;
  int pt = tile / nqt, qt = tile % nqt;
  int pfirst = P0 + pt * tile_rows;
  int qlast = Q0 + min(qrow, (qt + 1) * tile_cols) - 1;
  bool upper = atom_of_ri[pfirst] <= atom_of_ri[qlast];
  // warp-serial compaction in slab order (deterministic)
  if (threadIdx.x >= 32) return;
  int lane = threadIdx.x;
  int cnt = 0;
  long long ksum = 0;
  if (upper) {
    for (int base = 0; base < nslab; base += 32) {
      int s = base + lane;
      bool on = false;
      if (s < nslab) {
        // a slab is a task iff one of its mu atoms has both an X block in the
        // row tile and a Y block in the column tile (otherwise the product is
        // exactly zero)
        const int sl = s / per, c = s % per;
        const int a_lo = c * kSlabAO;  // chunk-local AO
        if (a_lo < nmu) {
          const int ma = atom_of_ao[mu0 + a_lo] - m0;
          const int mb = atom_of_ao[mu0 + min(nmu, a_lo + kSlabAO) - 1] - m0;
          for (int m = ma; m <= mb && !on; ++m)
            on = fx[((long long)sl * nmc + m) * npt + pt] && fy[((long long)sl * nmc + m) * nqt + qt];
        }
      }
      unsigned m = __ballot_sync(0xffffffffu, on);
      if (on) {
        tasks[(long long)tile * nslab + cnt + __popc(m & ((1u << lane) - 1))] = s;
        ksum += slab_len[s];
      }
      cnt += __popc(m);
    }
  }
  for (int o = 16; o > 0; o >>= 1) ksum += __shfl_xor_sync(0xffffffffu, ksum, o);
  if (lane == 0) {
    counts[tile] = cnt;
    kacc[tile] = ksum;
  }
  (void)prow;
}

// Useful flops of step C for one batch: for each (s, m) pair of the batch's
// sigma-atoms and the chunk's mu-atoms,
//   sum_{p <= q} 2 n(m) n(s) nP nQ [X(m,s,p) kept][Y(m,s,q) kept],
// X flags over RI atoms [pa0, pa0 + npa), Y flags over [qa0, qa0 + nqa).
__global__ void k_count_c(const unsigned char* __restrict__ bx, const unsigned char* __restrict__ by,
                          int ns, int m0, int nmc, int pa0, int npa, int qa0, int nqa,
                          const int* __restrict__ n_ri, const int* __restrict__ n_ao, int s0,
                          double* __restrict__ out) {
  int pair = blockIdx.x * blockDim.x + threadIdx.x;
  if (pair >= ns * nmc) return;
  int sl = pair / nmc, ml = pair % nmc;
  const unsigned char* fx = bx + ((long long)sl * nmc + ml) * npa;
  const unsigned char* fy = by + ((long long)sl * nmc + ml) * nqa;
  // suffix sums of Y over q
  double tot = 0.0, suffix = 0.0;
  int q = qa0 + nqa - 1;
  for (int pl = npa - 1; pl >= 0; --pl) {
    int p = pa0 + pl;
    while (q >= p && q >= qa0) {
      if (fy[q - qa0]) suffix += n_ri[q];
      --q;
    }
    if (fx[pl]) tot += (double)n_ri[p] * suffix;
  }
  out[pair] = 2.0 * tot * n_ao[m0 + ml] * n_ao[s0 + sl];
}

// chi_out[P][Q] = acc[P][Q] if atom(P) <= atom(Q) else acc[Q][P]
__global__ void k_mirror(const double* __restrict__ acc, double* __restrict__ out, int nri,
                         const int* __restrict__ atom_of_ri) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long n = (long long)nri * nri;
  if (i >= n) return;
  int P = (int)(i / nri), Q = (int)(i % nri);
  out[i] = atom_of_ri[P] <= atom_of_ri[Q] ? acc[i] : acc[(long long)Q * nri + P];
}

// ---------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------
void launch_block_norms_3c(const double* t3, long long base_off, const int* blk, const long long* off,
                           const int* n_ao, const int* n_ri, long long n_blocks, double* norms, int* bad,
                           cudaStream_t st) {
  if (n_blocks == 0) return;
  long long grid = (n_blocks + 7) / 8;
  k_block_norms_3c<<<(unsigned)grid, 256, 0, st>>>(t3, base_off, blk, off, n_ao, n_ri, n_blocks, norms,
                                                    bad);
}

void launch_panel_scatter(const double* t3, const int* blk, const long long* off, const int* n_ao,
                          const int* n_ri, const int* ri_off, const int* kept_idx, int n_kept,
                          const long long* dstB, const long long* dstA, const int* ldB,
                          const int* ldA, double* pool, cudaStream_t st) {
  if (n_kept == 0) return;
  k_panel_scatter<<<n_kept, 256, 0, st>>>(t3, blk, off, n_ao, n_ri, ri_off, kept_idx, n_kept, dstB,
                                          dstA, ldB, ldA, pool);
}

void launch_cast_f64_f32(const double* x, float* y, long long n, cudaStream_t st) {
  if (n == 0) return;
  long long blocks = (n + 255) / 256;
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_cast_f64_f32<<<(unsigned)blocks, 256, 0, st>>>(x, y, n);
}

void launch_scale_orbitals(const double* C, const double* eps, int nao, int n_occ, double mu, double tau,
                           double* cso, double* csv, cudaStream_t st) {
  const unsigned gx = (nao + 31) / 32;
  k_scale_orbitals<<<dim3(gx, (304 + gx - 1) / gx), 256, 0, st>>>(C, eps, nao, n_occ, mu, tau, cso, csv);
}

void launch_greens(const double* C, const double* eps, int nao, int n_occ, double mu, double tau,
                   double* cso, double* csv, double* g_occ, double* g_virt, cudaStream_t st) {
  launch_scale_orbitals(C, eps, nao, n_occ, mu, tau, cso, csv, st);
  const unsigned t = (nao + 15) / 16;
  k_syrk64<<<dim3(t, t, 2), 64, 0, st>>>(cso, csv, nao, n_occ, g_occ, g_virt);
}

void launch_sym_block_filter(double* g0, double* g1, int nao, const int* ao_off, int n_at, double thr,
                             unsigned char* flags0, unsigned char* flags1, cudaStream_t st) {
  const long long pairs = static_cast<long long>(n_at) * n_at;
  k_sym_block_filter<<<dim3(static_cast<unsigned>((pairs + 7) / 8), 2), 256, 0, st>>>(g0, g1, nao, ao_off, n_at, thr,
                                                                                      flags0, flags1);
}

template <typename T>
void launch_panel_gemm(const T* G, int nao, const T* pool, const int* lam, const PanelTask* tasks,
                       int ntasks, int maxN, int mode, int r0, int R, int P0b, long long ldk,
                       const long long* rowbase, const int* rowmul, T* out, cudaStream_t st) {
  if (ntasks == 0 || R == 0 || maxN == 0) return;
  for (int z0 = 0; z0 < ntasks; z0 += 65535) {
    int nz = ntasks - z0 < 65535 ? ntasks - z0 : 65535;
    dim3 grid((maxN + 63) / 64, (R + 63) / 64, nz);
    if constexpr (sizeof(T) == 4)
      k_panel_gemm_f32<<<grid, kF32Threads, 0, st>>>(G, nao, pool, lam, tasks + z0, mode, r0, R, P0b, ldk, rowbase, rowmul,
                                             out);
    else
      k_panel_gemm<T><<<grid, 256, 0, st>>>(G, nao, pool, lam, tasks + z0, mode, r0, R, P0b, ldk,
                                           rowbase, rowmul, out);
  }
}
template void launch_panel_gemm<double>(const double*, int, const double*, const int*,
                                        const PanelTask*, int, int, int, int, int, int, long long,
                                        const long long*, const int*, double*, cudaStream_t);
template void launch_panel_gemm<float>(const float*, int, const float*, const int*,
                                       const PanelTask*, int, int, int, int, int, int, long long,
                                       const long long*, const int*, float*, cudaStream_t);

template <typename T>
void launch_operand_block_filter(T* Z, long long ldk, int rowoff, const int* ri_off,
                                 const int* ao_off, const int* n_ao, int s0, int ns,
                                 const long long* seg, int pa0, int npa, int n_at, double thr,
                                 int naop, unsigned char* blockflag, unsigned char* tileflag,
                                 int ntile, int tile_rows, cudaStream_t st) {
  long long nblk = (long long)ns * n_at * npa;
  if (nblk == 0) return;
  k_operand_block_filter<T><<<(unsigned)((nblk + 7) / 8), 256, 0, st>>>(
      Z, ldk, rowoff, ri_off, ao_off, n_ao, s0, ns, seg, pa0, npa, n_at, thr, naop, blockflag,
      tileflag, ntile, tile_rows);
}
template void launch_operand_block_filter<double>(double*, long long, int, const int*, const int*,
                                                  const int*, int, int, const long long*, int, int,
                                                  int, double, int, unsigned char*, unsigned char*,
                                                  int, int, cudaStream_t);
template void launch_operand_block_filter<float>(float*, long long, int, const int*, const int*,
                                                 const int*, int, int, const long long*, int, int,
                                                 int, double, int, unsigned char*, unsigned char*,
                                                 int, int, cudaStream_t);

void launch_build_tasks(const unsigned char* fx, const unsigned char* fy, int nslab, int npt,
                        int nqt, int P0, int prow, int Q0, int qrow, const int* atom_of_ri,
                        const int* slab_len, int* tasks, int* counts, long long* kacc,
                        int tile_rows, int tile_cols, int per, int m0, int nmc, int mu0, int nmu,
                        const int* atom_of_ao, cudaStream_t st) {
  if (npt * nqt == 0) return;
  k_build_tasks<<<npt * nqt, 32, 0, st>>>(fx, fy, nslab, npt, nqt, P0, prow, Q0, qrow, atom_of_ri,
                                          slab_len, tasks, counts, kacc, tile_rows, tile_cols, per, m0, nmc, mu0,
                                          nmu, atom_of_ao);
}

void launch_count_c(const unsigned char* bx, const unsigned char* by, int ns, int m0, int nmc, int pa0,
                    int npa, int qa0, int nqa, const int* n_ri, const int* n_ao, int s0, double* out,
                    cudaStream_t st) {
  int n = ns * nmc;
  if (n == 0) return;
  k_count_c<<<(n + 127) / 128, 128, 0, st>>>(bx, by, ns, m0, nmc, pa0, npa, qa0, nqa, n_ri, n_ao, s0,
                                             out);
}

template <typename T, typename AccT>
void launch_chi_tiles(const T* X, const T* Y, long long ldk, int P0, int prow, int nri,
                      const int* tasks, const int* counts, int max_slab, int npt, int nqt,
                      const long long* slab_k0, const int* slab_len, double* chi, cudaStream_t st) {
  dim3 grid(nqt, npt);
  if constexpr (sizeof(T) == 4) {
    constexpr int smem = static_cast<int>(sizeof(F32ChiShared));
    cudaFuncSetAttribute(k_chi_tiles_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    k_chi_tiles_f32<<<dim3(nqt, npt, kF32Split), kF32Threads, smem, st>>>(
        X, Y, ldk, P0, prow, nri, tasks, counts, max_slab, nqt, slab_k0, slab_len, chi);
  } else {
    k_chi_tiles<T, AccT><<<grid, 256, 0, st>>>(X, Y, ldk, P0, prow, nri, tasks, counts, max_slab, nqt,
                                               slab_k0, slab_len, chi);
  }
}
template void launch_chi_tiles<double, double>(const double*, const double*, long long, int, int, int,
                                               const int*, const int*, int, int, int,
                                               const long long*, const int*, double*, cudaStream_t);
template void launch_chi_tiles<float, float>(const float*, const float*, long long, int, int, int,
                                             const int*, const int*, int, int, int,
                                             const long long*, const int*, double*, cudaStream_t);

void launch_mirror(const double* acc, double* out, int nri, const int* atom_of_ri, cudaStream_t st) {
  long long n = (long long)nri * nri;
  k_mirror<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(acc, out, nri, atom_of_ri);
}

}  // namespace gw
