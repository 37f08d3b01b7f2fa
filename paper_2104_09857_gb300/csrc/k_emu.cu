// FP64 products on the tensor cores (tcgen05) from exact integer digits.
//
// The FP64 pipe of this chip gives 1.26 TFLOP/s for all 152 SMs (two FMAs per
// cycle and SM); the 16-bit tensor cores give 1900.  Each row of an operand
// is scaled by a power of two above its largest magnitude and every element
// is rounded to an integer of 62 bits and sign, written as eight signed
// digits
//   x = 2^(e - 62) sum_{i<8} d_i 2^(8 (7 - i)),   |d_i| <= 128,
// which binary16 holds exactly.  A product a b is formed from the 36 digit
// pairs with i + j <= 7; the left-out pairs are together below 2^-61 of the
// two rows' largest magnitudes, the rounding of an element below 2^-63.  The
// pairs of one diagonal i + j = d have the same weight and share one
// accumulator: over 128 reduction elements its magnitude is at most
// 8 * 128 * 2^14 = 2^24, so the FP32 accumulation is exact integer
// arithmetic.  After every 128 elements the epilogue adds the eight
// diagonals into two 64-bit integers (diagonals 0-3 and 4-7), exactly, and
// rounds once at the end.  Against a sequential FP64 sum (error about
// 0.2 * 2^-53 |a| |b| of the rows' 2-norms for random signs) the result is
// closer to the exact value, and it does not depend on how K is split:
// partial sums are integers, so split units may add in any order.
//
// Layout of a tile: 128 x 64 outputs; stages of 32 reduction elements with
// all eight digits of both operands (96 KB, two stages), one TMA box per
// operand and stage.  64 columns and not 128: the two integers of 128 x 128
// outputs would take the whole register file.  Each diagonal has its own 64
// accumulator columns; a diagonal of the next 128 elements starts as soon as
// the epilogue has drained it.  Eight-bit digits and not nine: seven nine-bit
// digits need 28 products but a drain every 32 elements, and the drains'
// float-to-integer conversions (16 per cycle and SM) were then the limit.
// The MMA warp runs converged with one elected thread issuing, so that the
// descriptors stay in uniform registers: issued from a divergent branch an
// MMA took 85 cycles, now the 48 that its 6 KB of operands need.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "gw_internal.h"
#include "k_emu.h"
#include "k_tc.h"
#include "tc_ptx.h"

namespace gw {
namespace emu {

using namespace gw::tc;

constexpr int kS = kEmuSlices;
constexpr int kM = kEmuTileM, kN = kEmuTileN;
constexpr int kChunk = 32;  // reduction elements of a stage (64-byte rows)
constexpr int kSub = kChunk / kMmaK;
constexpr int kStages = 2;
constexpr int kGroup = 4;  // stages of one exact accumulation
constexpr int kTmemCols = 512;
constexpr int kEpiWarps = 16;              // 4 lane quadrants x 4 column groups
constexpr int kCols = kN / (kEpiWarps / 4);  // 16 columns per epilogue warp
constexpr int kThreads = (2 + kEpiWarps) * 32;
constexpr int kABytes = kM * kChunk * 2, kBBytes = kN * kChunk * 2;  // one digit of one operand
constexpr int kStageBytes = kS * (kABytes + kBBytes);
constexpr int kSmem = kStages * kStageBytes + 256 + 1024;
constexpr int kLoBits = 32;   // value = (hi * 2^32 + lo) * 2^(ea + eb - 68)
constexpr int kUnit = -68;
constexpr int kBad = INT32_MAX;  // exponent of a row that holds an Inf or NaN

// K-major tile of 64-byte rows (32 binary16), 64-byte swizzle: 8-row groups
// 512 bytes apart.
__device__ __forceinline__ uint64_t desc_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(512 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(4) << 61;
  return d;
}

// ---------------------------------------------------------------------------
// digits
// ---------------------------------------------------------------------------
// e with |x| < 2^e for every x whose largest biased exponent is be.
__device__ __forceinline__ int row_exp(int be) { return be == 2047 ? kBad : (be == 0 ? -1021 : be - 1022); }

// x * 2^(62 - e) rounded to an integer (|.| <= 2^62).
__device__ __forceinline__ long long fixed62(double x, int e) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int be = static_cast<int>((b >> 52) & 0x7ff);
  unsigned long long m = b & ((1ull << 52) - 1);
  if (be) m |= 1ull << 52;
  const int sh = (be ? be : 1) - 1013 - e;  // <= 9
  unsigned long long t = 0;
  if (sh >= 0)
    t = m << sh;
  else if (sh >= -53)
    t = (m + (1ull << (-sh - 1))) >> -sh;
  return (b >> 63) ? -static_cast<long long>(t) : static_cast<long long>(t);
}
// Digits of eight elements, packed for one 16-byte store per digit: q[i]
// holds digit i of the eight elements as binary16.
__device__ __forceinline__ void digits8(const double (&x)[8], int e, uint4 (&q)[kS]) {
  uint32_t w[kS][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    long long t0 = e == kBad ? 0 : fixed62(x[2 * p], e), t1 = e == kBad ? 0 : fixed62(x[2 * p + 1], e);
#pragma unroll
    for (int i = kS - 1; i >= 0; --i) {
      int d0, d1;
      if (i > 0) {
        d0 = static_cast<int>((t0 + 128) & 255) - 128;
        d1 = static_cast<int>((t1 + 128) & 255) - 128;
        t0 = (t0 - d0) >> 8;
        t1 = (t1 - d1) >> 8;
      } else {
        d0 = static_cast<int>(t0);
        d1 = static_cast<int>(t1);
      }
      // binary16 1536 + d has bits 0x6600 + d; the subtraction is exact
      const uint32_t u = static_cast<uint32_t>(0x6600 + d0) | (static_cast<uint32_t>(0x6600 + d1) << 16);
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&u), __float2half2_rn(1536.f));
      w[i][p] = *reinterpret_cast<const uint32_t*>(&h);
    }
  }
#pragma unroll
  for (int i = 0; i < kS; ++i) q[i] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}
__device__ __forceinline__ int biased_exp(double x) {
  return static_cast<int>((static_cast<unsigned long long>(__double_as_longlong(x)) >> 52) & 0x7ff);
}

// Rows of a row-major matrix: kWarps warps per row, which they read twice
// (the second time from cache): its exponent, then the digits, eight
// consecutive elements per lane.
template <int kWarps>
__global__ void __launch_bounds__(256) k_prep_rows(const double* __restrict__ src, long long ld, long long rows,
                                                   int K, int kp, long long zrows, long long z_stride,
                                                   __half* __restrict__ dig, int* __restrict__ exps) {
  constexpr int kPer = 8 / kWarps;  // rows of a CTA
  __shared__ int red[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = threadIdx.x % (32 * kWarps), nt = 32 * kWarps;
  for (long long r0 = static_cast<long long>(blockIdx.x) * kPer; r0 < rows;
       r0 += static_cast<long long>(gridDim.x) * kPer) {
    const long long r = r0 + warp / kWarps;
    const bool on = r < rows;
    const double* x = zrows == rows ? src + r * ld : src + r / zrows * z_stride + r % zrows * ld;
    int be = 0;
    if (on)
      for (int k = t; k < K; k += nt) be = max(be, biased_exp(x[k]));
    be = __reduce_max_sync(0xffffffffu, be);
    if (kWarps > 1) {
      __syncthreads();
      if (lane == 0) red[warp] = be;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kWarps; ++i) be = max(be, red[i]);
    }
    if (!on) continue;
    const int e = row_exp(be);
    if (t == 0) exps[r] = e;
    for (int k = 8 * t; k < kp; k += 8 * nt) {
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = k + i < K ? x[k + i] : 0.0;
      uint4 q[kS];
      digits8(v, e, q);
#pragma unroll
      for (int i = 0; i < kS; ++i)
        *reinterpret_cast<uint4*>(dig + (i * rows + r) * kp + k) = q[i];
    }
  }
}

// Columns of a row-major [K][rows] matrix as operand rows: largest biased
// exponent per column (be zeroed before), then the digits through a
// transposed 64 x 32 tile.
__global__ void __launch_bounds__(256) k_col_exps(const double* __restrict__ src, long long ld, long long rows,
                                                  int K, int* __restrict__ be) {
  const int c = threadIdx.x & 31, kk = threadIdx.x >> 5;
  const long long col = static_cast<long long>(blockIdx.x) * 32 + c;
  int m = 0;
  if (col < rows)
    for (int k = blockIdx.y * 8 + kk; k < K; k += 8 * gridDim.y) m = max(m, biased_exp(src[k * ld + col]));
  __shared__ int red[8][32];
  red[kk][c] = m;
  __syncthreads();
  if (kk == 0 && col < rows) {
#pragma unroll
    for (int i = 1; i < 8; ++i) m = max(m, red[i][c]);
    if (m) atomicMax(be + col, m);
  }
}
__global__ void __launch_bounds__(256) k_prep_cols(const double* __restrict__ src, long long ld, long long rows,
                                                   int K, int kp, const int* __restrict__ be,
                                                   __half* __restrict__ dig, int* __restrict__ exps) {
  __shared__ double t[64][33];
  const long long c0 = static_cast<long long>(blockIdx.x) * 32;
  const int k0 = blockIdx.y * 64;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = (threadIdx.x >> 5) + 8 * i, c = threadIdx.x & 31;
    t[k][c] = (k0 + k < K && c0 + c < rows) ? src[(k0 + k) * ld + c0 + c] : 0.0;
  }
  __syncthreads();
  const int c = threadIdx.x >> 3, g = threadIdx.x & 7;
  const long long r = c0 + c;
  if (r >= rows) return;
  const int e = row_exp(be[r]);
  if (blockIdx.y == 0 && g == 0) exps[r] = e;
  double v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = t[8 * g + i][c];
  uint4 q[kS];
  digits8(v, e, q);
#pragma unroll
  for (int i = 0; i < kS; ++i)
    *reinterpret_cast<uint4*>(dig + (i * rows + r) * kp + k0 + 8 * g) = q[i];
}

// The same for the owner panels of the 3c tensor ([K][N] each, blockIdx.z =
// panel): operand row row0[panel] + n, pitch kp.
__global__ void __launch_bounds__(256) k_panel_exps(const double* __restrict__ pool, const PanelDesc* __restrict__ pd,
                                                    const long long* __restrict__ row0, int* __restrict__ be) {
  const PanelDesc d = pd[blockIdx.z];
  const int N = d.npw * d.nsig;
  if (static_cast<int>(blockIdx.x) * 32 >= N) return;
  const int c = threadIdx.x & 31, kk = threadIdx.x >> 5;
  const int col = blockIdx.x * 32 + c;
  int m = 0;
  if (col < N)
    for (int k = blockIdx.y * 8 + kk; k < d.K; k += 8 * gridDim.y)
      m = max(m, biased_exp(pool[d.off + static_cast<long long>(k) * N + col]));
  __shared__ int red[8][32];
  red[kk][c] = m;
  __syncthreads();
  if (kk == 0 && col < N) {
#pragma unroll
    for (int i = 1; i < 8; ++i) m = max(m, red[i][c]);
    if (m) atomicMax(be + row0[blockIdx.z] + col, m);
  }
}
__global__ void __launch_bounds__(256) k_panel_prep(const double* __restrict__ pool, const PanelDesc* __restrict__ pd,
                                                    const long long* __restrict__ row0, long long rows, int kp,
                                                    const int* __restrict__ be, __half* __restrict__ dig,
                                                    int* __restrict__ exps) {
  const PanelDesc d = pd[blockIdx.z];
  const int N = d.npw * d.nsig, c0 = blockIdx.x * 32, k0 = blockIdx.y * 64;
  if (c0 >= N || k0 >= d.K) return;
  __shared__ double t[64][33];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = (threadIdx.x >> 5) + 8 * i, c = threadIdx.x & 31;
    t[k][c] = (k0 + k < d.K && c0 + c < N) ? pool[d.off + static_cast<long long>(k0 + k) * N + c0 + c] : 0.0;
  }
  __syncthreads();
  const int c = threadIdx.x >> 3, g = threadIdx.x & 7;
  if (c0 + c >= N) return;
  const long long r = row0[blockIdx.z] + c0 + c;
  const int e = row_exp(be[r]);
  if (blockIdx.y == 0 && g == 0) exps[r] = e;
  double v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = t[8 * g + i][c];
  uint4 q[kS];
  digits8(v, e, q);
#pragma unroll
  for (int i = 0; i < kS; ++i) *reinterpret_cast<uint4*>(dig + (i * rows + r) * kp + k0 + 8 * g) = q[i];
}

// Digits of G gathered on each task's lambda functions: out row
// g_row0 + r, column k = digits of G[rbase + r][lam[lam_off + k]], zero for
// k >= K up to the task's last 64 columns.  blockIdx.y = task, z = digit.
__global__ void __launch_bounds__(256) k_gather_digits(const __half* __restrict__ g, int nao, int gkp, int rbase,
                                                       int R, const PanelTask64* __restrict__ tasks,
                                                       const int* __restrict__ lam, long long out_rows, int kp,
                                                       __half* __restrict__ out) {
  const PanelTask64 tk = tasks[blockIdx.y];
  const int kt = (tk.K + 63) / 64 * 64;
  const __half* src = g + (static_cast<long long>(blockIdx.z) * nao + rbase) * gkp;
  __half* dst = out + (blockIdx.z * out_rows + tk.g_row0) * kp;
  const int n = R * kt;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int r = i / kt, k = i - r * kt;
    dst[static_cast<long long>(r) * kp + k] =
        k < tk.K ? src[static_cast<long long>(r) * gkp + lam[tk.lam_off + k]] : __half(0.f);
  }
}

// ---------------------------------------------------------------------------
// integers back to FP64
// ---------------------------------------------------------------------------
// lo into [0, 2^32), the carry into hi.
__device__ __forceinline__ void carry(long long& hi, long long& lo) {
  hi += lo >> kLoBits;
  lo &= (1ll << kLoBits) - 1;
}
// (hi 2^32 + lo) 2^e rounded to nearest even, in 32-bit integer arithmetic:
// the FP64 pipe takes 16 cycles per warp and operation.
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int e) {
  carry(hi, lo);
  uint32_t w2 = static_cast<uint32_t>(static_cast<unsigned long long>(hi) >> 32);
  uint32_t w1 = static_cast<uint32_t>(hi), w0 = static_cast<uint32_t>(lo);
  const uint32_t sign = w2 & 0x80000000u;
  if (sign) {  // 96-bit negation
    w0 = 0u - w0;
    w1 = ~w1 + (w0 == 0u);
    w2 = ~w2 + (w0 == 0u && w1 == 0u);
  }
  const bool z2 = w2 == 0u, z1 = z2 && w1 == 0u;
  if (z1 && w0 == 0u) return 0.0;
  // leading word first
  const uint32_t a = z1 ? w0 : (z2 ? w1 : w2), b = z1 ? 0u : (z2 ? w0 : w1), c = z2 ? 0u : w0;
  const int s = __clz(static_cast<int>(a));
  const uint32_t m1 = __funnelshift_l(b, a, s), m0 = __funnelshift_l(c, b, s), rest = c << s;
  uint32_t f1 = m1 >> 11, f0 = __funnelshift_l(m0, m1, 21);
  const uint32_t cut = m0 & 0x7ffu;
  const uint32_t up = cut > 0x400u || (cut == 0x400u && (rest != 0u || (f0 & 1u)));
  f0 += up;
  f1 += up && f0 == 0u;
  // (f1 : f0) in [2^52, 2^53], value (f1 : f0) 2^ex
  const int ex = 43 - s - (z1 ? 64 : (z2 ? 32 : 0)) + e;
  const int be = ex + 1075;
  if (be > 0 && be < 2046)
    return __hiloint2double(static_cast<int>(((static_cast<uint32_t>(be - 1) << 20) + f1) | sign),
                            static_cast<int>(f0));
  const double d = ldexp(__hiloint2double(static_cast<int>((1074u << 20) + f1), static_cast<int>(f0)), ex);
  return sign ? -d : d;
}

// ---------------------------------------------------------------------------
// dense products
// ---------------------------------------------------------------------------
struct GemmJob {
  int m, n, K, nt, n_items, ks, stages, tri, ktri, tri_off;
  double alpha, beta;
  double* C;
  long long ldc, cblk_stride, col0;
  int cblk;
  const int *ea, *eb;
  int per_z, za, zb;         // items and operand rows of one product of a batch
  long long c_z, a_z, b_z;   // C, A, B from one product to the next
  unsigned long long* part;  // ks > 1: [nz][m][n][2] integer sums
  const double *A, *B;
  long long lda, ldb;
  int ta, tb;

  struct Tile {
    int ya, yb, c0, n;  // rows of the stacked digits
    int ra, rb, z;      // ... and of the product's own operands
  };
  __device__ int items() const { return n_items; }
  __device__ Tile tile(int t) const {
    Tile T;
    T.z = t / per_z;
    const int u = t - T.z * per_z, s = u % ks, x = u / ks;
    T.ra = x / nt * kM;
    T.rb = x % nt * kN;
    T.ya = T.ra + T.z * za;
    T.yb = T.rb + T.z * zb;
    const int from = ktri ? min(max(T.ra + tri_off, 0) / kChunk, stages) : 0;
    const int per = (stages - from + ks - 1) / ks;
    T.c0 = from + s * per;
    T.n = max(min(per, stages - T.c0), 0);
    // an unsplit product writes every element, also where no stage is left
    if (ks == 1 && T.n == 0) {
      T.c0 = stages - 1;
      T.n = 1;
    }
    if (skip(T.ra, T.rb)) T.n = 0;
    return T;
  }
  __device__ bool skip(int ya, int yb) const { return tri && yb >= ya + kM + tri_off; }
  __device__ int nchunks(const Tile& T) const { return T.n; }
  struct Iter {
    int x;
    __device__ void init(const GemmJob*, const Tile& T) { x = T.c0 * kChunk; }
    __device__ int next() {
      const int v = x;
      x += kChunk;
      return v;
    }
  };
  __device__ double at(const double* p, long long ld, int t, int r, int k) const {
    return t ? p[k * ld + r] : p[r * ld + k];
  }
  // the element from the FP64 operands (a row with an Inf or NaN)
  __device__ double direct(int z, int r, int c) const {
    double s = 0.0;
    for (int k = 0; k < K; ++k) s = fma(at(A + z * a_z, lda, ta, r, k), at(B + z * b_z, ldb, tb, c, k), s);
    return s;
  }
  __device__ void store(int z, int r, int c, double v) const {
    long long at = c;
    if (cblk) {
      const uint32_t q = static_cast<uint32_t>(c + col0), b = static_cast<uint32_t>(cblk);
      at = q / b * cblk_stride + q % b;
    }
    double* p = C + z * c_z + r * ldc + at;
    const double w = alpha == 1.0 ? v : (alpha == -1.0 ? -v : alpha * v);  // most calls spare the FP64 pipe
    *p = beta == 0.0 ? w : fma(beta, *p, w);
  }
  __device__ void write(long long (&hi)[kCols], long long (&lo)[kCols], const Tile& T, int row, int c0) const {
    const int r = T.ra + row;
    if (r >= m) return;
    if (part) {
      unsigned long long* p = part + ((static_cast<long long>(T.z) * m + r) * n + T.rb + c0) * 2;
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        if (T.rb + c0 + j >= n) break;
        carry(hi[j], lo[j]);
        atomicAdd(p + 2 * j, static_cast<unsigned long long>(hi[j]));
        atomicAdd(p + 2 * j + 1, static_cast<unsigned long long>(lo[j]));
      }
      return;
    }
    const int a = ea[T.z * za + r];
    unsigned bad = 0;  // columns that need the FP64 operands
#pragma unroll
    for (int j = 0; j < kCols; ++j) {
      const int c = T.rb + c0 + j;
      if (c >= n) break;
      const int b = eb[T.z * zb + c];
      if (a == kBad || b == kBad)
        bad |= 1u << j;
      else
        store(T.z, r, c, fixed_to_double(hi[j], lo[j], a + b + kUnit));
    }
    while (bad) {
      const int c = T.rb + c0 + __ffs(bad) - 1;
      store(T.z, r, c, direct(T.z, r, c));
      bad &= bad - 1;
    }
  }
};
__global__ void k_gemm_finish(const GemmJob j, int nz) {
  const long long mn = static_cast<long long>(j.m) * j.n;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < mn * nz;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int z = static_cast<int>(i / mn);
    const long long e = i - z * mn;
    const int r = static_cast<int>(e / j.n), c = static_cast<int>(e % j.n);
    if (j.skip(r / kM * kM, c / kN * kN)) continue;
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(j.part)[i];
    const int a = j.ea[z * j.za + r], b = j.eb[z * j.zb + c];
    j.store(z, r, c, a == kBad || b == kBad ? j.direct(z, r, c)
                                            : fixed_to_double(static_cast<long long>(v.x),
                                                              static_cast<long long>(v.y), a + b + kUnit));
  }
}

// ---------------------------------------------------------------------------
// steps A / B of Eq. 3 in FP64: one tile = 128 rows of the A operand x 64 of
// the B operand of one panel task
//   mode 0 (X): A = panel rows n = (pw, s'), B = G^occ rows mu
//   mode 1 (Y): A = G^virt rows sigma (batch), B = panel rows n = (pw, mu')
// A thread owns one A row, so consecutive lanes write along the contiguous
// index of the operand's K layout (s, mu, s').
// ---------------------------------------------------------------------------
struct Panel64Job {
  const int4* tiles;  // (task, A tile, B tile, 0)
  int n_tiles, mode, R, r0, P0b;
  const PanelTask64* tasks;
  long long ldk;
  const long long* rowbase;
  const int* rowmul;
  const int *pe, *ge;  // exponents of the panel rows and of G's rows
  double* out;
  const double *pool, *G;
  const int* lam;
  int nao;
  struct Tile {
    int ya, yb, n, task, a0, b0;
  };
  __device__ int items() const { return n_tiles; }
  __device__ Tile tile(int t) const {
    const int4 e = tiles[t];
    const PanelTask64& tk = tasks[e.x];
    Tile T;
    T.task = e.x;
    T.a0 = e.y * kM;
    T.b0 = e.z * kN;
    T.ya = (mode == 0 ? tk.p_row0 : tk.g_row0) + T.a0;
    T.yb = (mode == 0 ? tk.g_row0 : tk.p_row0) + T.b0;
    T.n = (tk.K + kChunk - 1) / kChunk;
    return T;
  }
  __device__ int nchunks(const Tile& T) const { return T.n; }
  struct Iter {
    int x;
    __device__ void init(const Panel64Job*, const Tile&) { x = 0; }
    __device__ int next() {
      const int v = x;
      x += kChunk;
      return v;
    }
  };
  // panel row n against G row r (global AO) from the FP64 values
  __device__ double direct(const PanelTask64& tk, int n, int r) const {
    double s = 0.0;
    for (int k = 0; k < tk.K; ++k)
      s = fma(G[static_cast<long long>(lam[tk.lam_off + k]) * nao + r],
              pool[tk.panel_off + static_cast<long long>(k) * tk.N + n], s);
    return s;
  }
  __device__ void write(long long (&hi)[kCols], long long (&lo)[kCols], const Tile& T, int row, int c0) const {
    const PanelTask64& tk = tasks[T.task];
    const int a = T.a0 + row, b = T.b0 + c0;
    const int nsig = tk.nsig;
    unsigned bad = 0;
    if (mode == 0) {
      if (a >= tk.N) return;
      const int pw = a / nsig, sp = a - pw * nsig;
      const int ea = pe[tk.p_row0 + a];
      double* o = out + static_cast<long long>(tk.p0 + pw - P0b) * ldk + tk.seg + sp;
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        const int mu = b + j;
        if (mu >= R) break;
        const int eb = ge[r0 + mu];
        if (ea == kBad || eb == kBad)
          bad |= 1u << j;
        else
          o[static_cast<long long>(r0 + mu) * nsig] = fixed_to_double(hi[j], lo[j], ea + eb + kUnit);
      }
      for (; bad; bad &= bad - 1) {
        const int mu = b + __ffs(bad) - 1;
        o[static_cast<long long>(r0 + mu) * nsig] = direct(tk, a, r0 + mu);
      }
    } else {
      if (a >= R) return;
      const int ea = ge[r0 + a];
      const long long rb = rowbase[a], rm = rowmul[a];
      int pw = b / nsig, sp = b - pw * nsig;
      double* o = out + static_cast<long long>(tk.p0 + pw - P0b) * ldk + rb + tk.aom * rm;
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        const int n = b + j;
        if (n >= tk.N) break;
        const int eb = pe[tk.p_row0 + n];
        o[sp * rm] = (ea == kBad || eb == kBad) ? direct(tk, n, r0 + a)
                                                : fixed_to_double(hi[j], lo[j], ea + eb + kUnit);
        if (++sp == nsig) {
          sp = 0;
          o += ldk;
        }
      }
    }
  }
};

// ---------------------------------------------------------------------------
// step C in FP64: chi[P][Q] -= sum over the unit's slabs of X[P][k] Y[Q][k]
// ---------------------------------------------------------------------------
struct Chi64Job {
  const int *unit_tile, *unit_first, *unit_count, *n_units;
  const int* tasks;
  const int* counts;
  int nslab, nqt, P0, prow, nri;
  const long long* slab_k0;
  const int* slab_len;
  const int *ex, *ey;
  double* chi;
  unsigned long long* part;  // units of one tile add here; null: a unit is a whole tile
  const double *X, *Y;
  long long ldk;
  struct Tile {
    int ya, yb, n, cnt, id;
    const int* list;
  };
  __device__ int items() const { return *n_units; }
  __device__ Tile tile(int u) const {
    Tile T;
    T.id = unit_tile[u];
    T.ya = T.id / nqt * kM;
    T.yb = T.id % nqt * kN;
    T.cnt = unit_count[u];
    T.list = tasks + static_cast<long long>(T.id) * nslab + unit_first[u];
    T.n = 0;
    for (int i = 0; i < T.cnt; ++i) T.n += slab_len[T.list[i]] / kChunk;
    return T;
  }
  __device__ int nchunks(const Tile& T) const { return T.n; }
  struct Iter {
    const Chi64Job* j;
    const int* list;
    int cnt, i, kk, len;
    long long k0;
    __device__ void init(const Chi64Job* jj, const Tile& T) {
      j = jj;
      list = T.list;
      cnt = T.cnt;
      i = kk = 0;
      len = cnt > 0 ? j->slab_len[list[0]] : 0;
      k0 = cnt > 0 ? j->slab_k0[list[0]] : 0;
    }
    __device__ int next() {
      const int x = static_cast<int>(k0 + kk);
      kk += kChunk;
      if (kk >= len) {
        ++i;
        kk = 0;
        if (i < cnt) {
          len = j->slab_len[list[i]];
          k0 = j->slab_k0[list[i]];
        }
      }
      return x;
    }
  };
  // the element from the FP64 operands, over the tile's whole list
  __device__ double direct(int id, int p, int q) const {
    double s = 0.0;
    const int* l = tasks + static_cast<long long>(id) * nslab;
    for (int i = 0; i < counts[id]; ++i)
      for (int k = 0; k < slab_len[l[i]]; ++k)
        s = fma(X[p * ldk + slab_k0[l[i]] + k], Y[q * ldk + slab_k0[l[i]] + k], s);
    return s;
  }
  __device__ void add(int id, int p, int q, long long hi, long long lo) const {
    const int a = ex[p], b = ey[q];
    double* c = chi + static_cast<long long>(P0 + p) * nri + q;
    *c -= (a == kBad || b == kBad) ? direct(id, p, q) : fixed_to_double(hi, lo, a + b + kUnit);
  }
  __device__ void write(long long (&hi)[kCols], long long (&lo)[kCols], const Tile& T, int row, int c0) const {
    const int p = T.ya + row;
    if (p >= prow) return;
    if (part) {
      unsigned long long* o = part + (static_cast<long long>(p) * nri + T.yb + c0) * 2;
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        if (T.yb + c0 + j >= nri) break;
        carry(hi[j], lo[j]);
        atomicAdd(o + 2 * j, static_cast<unsigned long long>(hi[j]));
        atomicAdd(o + 2 * j + 1, static_cast<unsigned long long>(lo[j]));
      }
    } else {
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        if (T.yb + c0 + j >= nri) break;
        add(T.id, p, T.yb + c0 + j, hi[j], lo[j]);
      }
    }
  }
};
__global__ void k_chi64_finish(const Chi64Job j) {
  const long long n = static_cast<long long>(j.prow) * j.nri;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int p = static_cast<int>(i / j.nri), q = static_cast<int>(i % j.nri);
    const int id = p / kM * j.nqt + q / kN;
    if (j.counts[id] == 0) continue;
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(j.part)[i];
    j.add(id, p, q, static_cast<long long>(v.x), static_cast<long long>(v.y));
  }
}

// ---------------------------------------------------------------------------
// the persistent kernel: warp 0 TMA producer, warp 1 MMA issuer, warps 2-17
// epilogue; every wait is bounded (tc_ptx.h)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}

template <class Job>
__global__ void __launch_bounds__(kThreads, 1)
    k_emu(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const Job job,
          int* __restrict__ err_flag) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;
  uint64_t* acc_empty = acc_full + kS;
  uint64_t* drain = acc_empty + kS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = __reduce_max_sync(0xffffffffu, threadIdx.x / 32), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < kS; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int n_items = job.items();

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool armed[kStages] = {};
      uint32_t armed_parity[kStages] = {};
      bool ok = true;
      for (int t = blockIdx.x; t < n_items && ok; t += gridDim.x) {
        const typename Job::Tile T = job.tile(t);
        const int n = job.nchunks(T);
        typename Job::Iter it;
        it.init(&job, T);
        for (int i = 0; i < n; ++i) {
          if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + stage * kStageBytes;
          mbar_expect_tx(&full[stage], kStageBytes);
          armed[stage] = true;
          armed_parity[stage] = phase;
          const int x = it.next();
          tma_load_3d(st, &map_a, x, T.ya, 0, &full[stage]);
          tma_load_3d(st + kS * kABytes, &map_b, x, T.yb, 0, &full[stage]);
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(err_flag, 1);
        for (int s = 0; s < kStages; ++s)
          if (armed[s]) mbar_wait_cleanup(&full[s], armed_parity[s]);
      }
    }
  } else if (warp == 1) {
    // the whole warp runs the loop: uniform control flow keeps the
    // descriptors in uniform registers; one elected lane issues
    constexpr uint32_t idesc = idesc_f32(kM, kN, true);
    const uint32_t lead = elect_one();
    const uint32_t tmu = __reduce_max_sync(0xffffffffu, tmem);
    int stage = 0;
    uint32_t phase = 0, aphase = 1;
    bool ok = true, issued = false;
    for (int t = blockIdx.x; t < n_items && ok; t += gridDim.x) {
      const typename Job::Tile T = job.tile(t);
      const int n = __reduce_max_sync(0xffffffffu, job.nchunks(T));
      for (int i = 0; i < n && ok; ++i) {
        ok = __all_sync(0xffffffffu, mbar_wait(&full[stage], phase, abort_flag));
        if (!ok) break;
        tc_fence_after();
        const bool first = (i % kGroup) == 0, last = (i % kGroup) == kGroup - 1 || i == n - 1;
        const uint64_t da = desc_sw64(smem_u32(smem + stage * kStageBytes));
        const uint32_t a_lo = static_cast<uint32_t>(da), hi = static_cast<uint32_t>(da >> 32);
        const uint32_t b_lo = a_lo + static_cast<uint32_t>((kS * kABytes) >> 4);
#pragma unroll
        for (int d = 0; d < kS; ++d) {
          if (first) {
            ok = __all_sync(0xffffffffu, mbar_wait(&acc_empty[d], aphase, abort_flag));
            if (!ok) break;
            tc_fence_after();
          }
          if (lead) {
            const uint32_t acc = tmu + static_cast<uint32_t>(d * kN);
#pragma unroll
            for (int a = 0; a <= d; ++a)
#pragma unroll
              for (int k = 0; k < kSub; ++k)
                mma_f16_lo(acc, a_lo + static_cast<uint32_t>((a * kABytes + k * kMmaK * 2) >> 4),
                           b_lo + static_cast<uint32_t>(((d - a) * kBBytes + k * kMmaK * 2) >> 4), hi, idesc,
                           (a | k) ? 1u : (first ? 0u : 1u));
            if (last) mma_commit(&acc_full[d]);
          }
          __syncwarp();
          issued = true;
        }
        if (!ok) break;
        if (lead) mma_commit(&empty[stage]);
        __syncwarp();
        if (last) aphase ^= 1u;
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok && lead) {
      *abort_flag = 1;
      atomicOr(err_flag, 2);
      if (issued) {
        mma_commit(drain);
        mbar_wait_cleanup(drain, 0);
      }
    }
    __syncwarp();
  } else {
    const int quad = warp & 3;
    const int c0 = ((warp - 2) >> 2) * kCols;
    const uint32_t row_addr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(c0);
    uint32_t aphase = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < n_items && ok; t += gridDim.x) {
      const typename Job::Tile T = job.tile(t);
      const int n = job.nchunks(T);
      if (n == 0) continue;
      long long hi[kCols], lo[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) hi[j] = lo[j] = 0;
      for (int i = 0; i < n && ok; i += kGroup, aphase ^= 1u) {
#pragma unroll
        for (int d = 0; d < kS; ++d) {
          if (!mbar_wait(&acc_full[d], aphase, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int h = 0; h < 2; ++h) {  // two halves: 16 columns at once would spill
            uint32_t r[8];
            tmem_ld8(row_addr + static_cast<uint32_t>(d * kN + 8 * h), r);
            if (h == 1) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&acc_empty[d]);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int v = __float2int_rn(__uint_as_float(r[j]));
              if (d < 4)
                hi[8 * h + j] += static_cast<long long>(v) * (1 << (24 - 8 * d));
              else
                lo[8 * h + j] += static_cast<long long>(v) * (1 << (56 - 8 * d));
            }
          }
        }
        // a group adds less than 2^48 to lo
        if ((i & 16383) == 16384 - kGroup) {
#pragma unroll
          for (int j = 0; j < kCols; ++j) carry(hi[j], lo[j]);
        }
      }
      if (!ok) break;
      job.write(hi, lo, T, quad * 32 + lane, c0);
    }
    if (!ok) {
      *abort_flag = 1;
      if (lane == 0) atomicOr(err_flag, 4);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
  }
}

template <class Job>
int launch(const CUtensorMap& ma, const CUtensorMap& mb, const Job& job, int n_items, int* err_flag,
           cudaStream_t st) {
  if (n_items <= 0) return 0;
  static std::atomic<unsigned long long> attr_set{0};  // per device, as in k_tc.cu
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (!bit || !(attr_set.load(std::memory_order_acquire) & bit)) {
    if (cudaFuncSetAttribute(k_emu<Job>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess)
      return -1;
    attr_set.fetch_or(bit, std::memory_order_release);
  }
  k_emu<Job><<<std::min(n_items, sms), kThreads, kSmem, st>>>(ma, mb, job, err_flag);
  return 0;
}

// K splits of an m x n product: the number of units that makes the last wave
// over the SMs short.  Costs in stages (about 2 us each): a unit's start and
// end about 3 (the write, or 128 KB of atomics), clearing and converting the
// partial sums about 5 in all.
int k_splits(long long m, long long n, int K, int nz) {
  const long long tiles = ((m + kM - 1) / kM) * ((n + kN - 1) / kN) * nz;
  const long long stages = (K + kChunk - 1) / kChunk;
  long long best = 1, cost = 0;
  for (long long ks = 1; ks <= 64 && ks * 4 <= std::max(stages, 4ll); ++ks) {
    const long long c = (tiles * ks + 151) / 152 * ((stages + ks - 1) / ks + 3) + (ks > 1 ? 5 : 0);
    if (ks == 1 || c < cost) {
      cost = c;
      best = ks;
    }
  }
  return static_cast<int>(best);
}

}  // namespace emu

void launch_emu_prep(EmuOp& op, const EmuSrc& s, cudaStream_t st) {
  op.s = s;
  const long long rows = s.rows * s.nz;
  op.stride_rows = rows;
  op.kp = emu_kp(s.K);
  if (rows <= 0) return;
  __half* dig = static_cast<__half*>(op.dig);
  if (!s.trans) {
    const bool wide = s.K >= 2048;  // a CTA per row, else a warp
    const long long blocks = wide ? rows : (rows + 7) / 8;
    const unsigned grid = static_cast<unsigned>(std::min<long long>(blocks, 152 * 64));
    if (wide)
      emu::k_prep_rows<8><<<grid, 256, 0, st>>>(s.src, s.ld, rows, s.K, op.kp, s.rows, s.z_stride, dig, op.exps);
    else
      emu::k_prep_rows<1><<<grid, 256, 0, st>>>(s.src, s.ld, rows, s.K, op.kp, s.rows, s.z_stride, dig, op.exps);
  } else {
    int* be = op.exps + s.rows;
    cudaMemsetAsync(be, 0, static_cast<size_t>(s.rows) * sizeof(int), st);
    const unsigned gx = static_cast<unsigned>((s.rows + 31) / 32);
    const unsigned gy = static_cast<unsigned>(std::max(1, std::min((s.K + 63) / 64, static_cast<int>(1 + 608 / gx))));
    emu::k_col_exps<<<dim3(gx, gy), 256, 0, st>>>(s.src, s.ld, s.rows, s.K, be);
    emu::k_prep_cols<<<dim3(gx, op.kp / 64), 256, 0, st>>>(s.src, s.ld, s.rows, s.K, op.kp, be, dig, op.exps);
  }
}

size_t emu_gemm_ws_bytes(long long m, long long n, int K, int nz) {
  return emu::k_splits(m, n, K, nz) > 1 ? static_cast<size_t>(m) * n * 16 * nz : 0;
}

int launch_emu_gemm(const EmuOp& A, const EmuOp& B, const EmuGemm& g, void* ws, int* err_flag,
                    cudaStream_t st) {
  const int m = static_cast<int>(A.s.rows), n = static_cast<int>(B.s.rows);
  if (m <= 0 || n <= 0) return 0;
  CUtensorMap ma, mb;
  if (make_digit_map(&ma, A.dig, A.kp, A.s.nz > 1 ? A.stride_rows : A.s.rows, A.stride_rows, kEmuSlices, emu::kChunk, emu::kM) ||
      make_digit_map(&mb, B.dig, B.kp, B.s.nz > 1 ? B.stride_rows : B.s.rows, B.stride_rows, kEmuSlices, emu::kChunk,
                     emu::kN))
    return -2;
  emu::GemmJob j{};
  j.m = m;
  j.n = n;
  j.K = A.s.K;
  j.nt = (n + emu::kN - 1) / emu::kN;
  j.stages = std::max(1, (A.s.K + emu::kChunk - 1) / emu::kChunk);
  const int nz = A.s.nz;
  j.ks = ws ? emu::k_splits(m, n, A.s.K, nz) : 1;
  j.per_z = (m + emu::kM - 1) / emu::kM * j.nt * j.ks;
  // rows of one matrix in the stacked digits (a slice of rows of each keeps the whole stack's)
  j.za = nz > 1 ? static_cast<int>(A.stride_rows / nz) : 0;
  j.zb = B.s.nz > 1 ? static_cast<int>(B.stride_rows / B.s.nz) : 0;
  j.c_z = g.c_zstride;
  j.a_z = A.s.z_stride;
  j.b_z = B.s.z_stride;
  const long long items = static_cast<long long>(j.per_z) * nz;
  if (items > INT32_MAX) return -3;
  j.n_items = static_cast<int>(items);
  j.tri = g.tri;
  j.ktri = g.ktri;
  j.tri_off = static_cast<int>(g.tri_off);
  j.alpha = g.alpha;
  j.beta = g.beta;
  j.C = g.C;
  j.ldc = g.ldc;
  j.cblk = g.cblk;
  j.cblk_stride = g.cblk_stride;
  j.col0 = g.col0;
  j.ea = A.exps;
  j.eb = B.exps;
  j.A = A.s.src;
  j.lda = A.s.ld;
  j.ta = A.s.trans;
  j.B = B.s.src;
  j.ldb = B.s.ld;
  j.tb = B.s.trans;
  if (j.ks > 1) {
    j.part = static_cast<unsigned long long*>(ws);
    cudaMemsetAsync(ws, 0, static_cast<size_t>(m) * n * 16 * nz, st);
  }
  const int rc = emu::launch(ma, mb, j, j.n_items, err_flag, st);
  if (rc) return rc;
  if (j.ks > 1) {
    const long long blocks = (static_cast<long long>(m) * n * nz + 255) / 256;
    emu::k_gemm_finish<<<static_cast<unsigned>(std::min<long long>(blocks, 152 * 16)), 256, 0, st>>>(j, nz);
  }
  return 0;
}

void launch_panel_digits(const double* pool, const PanelDesc* panels, const long long* row0, int n_panels, int max_n,
                         int max_k, long long rows, int kp, int* be, void* dig, int* exps, cudaStream_t st) {
  if (n_panels == 0 || max_n == 0) return;
  cudaMemsetAsync(be, 0, static_cast<size_t>(rows) * sizeof(int), st);
  const unsigned gx = (max_n + 31) / 32, gy = (max_k + 63) / 64;
  for (int z = 0; z < n_panels; z += 65535) {
    const unsigned nz = std::min(n_panels - z, 65535);
    emu::k_panel_exps<<<dim3(gx, std::min(gy, 4u), nz), 256, 0, st>>>(pool, panels + z, row0 + z, be);
    emu::k_panel_prep<<<dim3(gx, gy, nz), 256, 0, st>>>(pool, panels + z, row0 + z, rows, kp, be,
                                                        static_cast<__half*>(dig), exps);
  }
}

void launch_gather_digits(const EmuOp& g, int rbase, int R, const PanelTask64* tasks, int n_tasks, const int* lam,
                          long long out_rows, int kp, void* out, cudaStream_t st) {
  if (n_tasks == 0 || R == 0) return;
  const unsigned bx = static_cast<unsigned>(std::min<long long>((static_cast<long long>(R) * kp + 255) / 256, 256));
  for (int t = 0; t < n_tasks; t += 65535)
    emu::k_gather_digits<<<dim3(bx, std::min(n_tasks - t, 65535), kEmuSlices), 256, 0, st>>>(
        static_cast<const __half*>(g.dig), static_cast<int>(g.stride_rows), g.kp, rbase, R, tasks + t, lam, out_rows,
        kp, static_cast<__half*>(out));
}

int launch_panel64(const Panel64Args& p, int* err_flag, cudaStream_t st) {
  if (p.n_tiles == 0) return 0;
  CUtensorMap mp, mg;
  const bool x = p.mode == 0;
  if (make_digit_map(&mp, p.panel_dig, p.kp, p.panel_rows, p.panel_rows, kEmuSlices, emu::kChunk,
                     x ? emu::kM : emu::kN) ||
      make_digit_map(&mg, p.g_dig, p.g_kp, p.g_rows, p.g_rows, kEmuSlices, emu::kChunk, x ? emu::kN : emu::kM))
    return -2;
  emu::Panel64Job j{p.tiles, p.n_tiles, p.mode, p.R,  p.r0,   p.P0b, p.tasks, p.ldk, p.rowbase,
                    p.rowmul, p.panel_exps, p.g_exps, p.out, p.pool, p.G, p.lam, p.nao};
  return x ? emu::launch(mp, mg, j, p.n_tiles, err_flag, st) : emu::launch(mg, mp, j, p.n_tiles, err_flag, st);
}

int launch_chi64(const EmuOp& x, const EmuOp& y, const Chi64Args& c, int* err_flag, cudaStream_t st) {
  CUtensorMap mx, my;
  if (make_digit_map(&mx, x.dig, x.kp, x.s.rows, x.stride_rows, kEmuSlices, emu::kChunk, emu::kM) ||
      make_digit_map(&my, y.dig, y.kp, y.s.rows, y.stride_rows, kEmuSlices, emu::kChunk, emu::kN))
    return -2;
  emu::Chi64Job j{c.units.u_tile, c.units.u_first, c.units.u_count, c.units.n_units, c.tasks, c.counts, c.nslab,
                  c.nqt, c.P0, c.prow, c.nri, c.slab_k0, c.slab_len, x.exps, y.exps, c.chi,
                  static_cast<unsigned long long*>(c.part), x.s.src, y.s.src, x.s.ld};
  if (c.part) cudaMemsetAsync(c.part, 0, static_cast<size_t>(c.prow) * c.nri * 16, st);
  const int rc = emu::launch(mx, my, j, INT32_MAX, err_flag, st);
  if (rc) return rc;
  if (c.part) {
    const long long blocks = (static_cast<long long>(c.prow) * c.nri + 255) / 256;
    emu::k_chi64_finish<<<static_cast<unsigned>(std::min<long long>(blocks, 152 * 16)), 256, 0, st>>>(j);
  }
  return 0;
}

}  // namespace gw
