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
// partial sums are integers, so split units may add in any order.  That holds
// in the norm: the error of an element is 2^-61 of the product of its rows'
// largest magnitudes, also where the element itself is far below that product
// and an FP64 sum's error with it.  Step C of chi, whose rows fall off with
// distance, therefore has exponents per part of a row (Chi64Job).
//
// Layout: two neighbouring CTAs take 128 x 128 outputs, 64 columns each;
// stages of 32 reduction elements with all eight digits of both operands
// (96 KB, two stages).  64 columns per CTA and not 128: the two integers of
// 128 x 128 outputs would take the whole register file.  Both load the A
// operand; that they run side by side keeps its second read in the L2 cache.
// MMAs: a digit of A meets two neighbouring digits of B at once, whose rows
// follow one another in shared memory, and adds into two neighbouring
// diagonals, 64 accumulator columns each: N = 128 takes 64 cycles where two
// N = 64 take 48 each (each reads the 4 KB of A again).  32 N = 128 and 8 N =
// 64 MMAs per stage: 2430 cycles.  The diagonals go pair by pair, so that the
// epilogue drains one pair while the next is computed.  The MMA warp runs
// converged with one elected lane issuing: the descriptors stay in uniform
// registers (from a divergent branch an MMA took 85 cycles).
// Eight-bit digits and not nine: seven nine-bit digits need 28 products but a
// drain every 32 elements, and the drains' float-to-integer conversions (16
// per cycle and SM) were then the limit.
// Measured at 4096^3: 3.06 ms, 45 TFLOP/s (one digit pair per MMA: 4.2 ms;
// without the elected lane and with nine-bit digits: 6.2 ms; the FP64 pipe:
// 137 ms).
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
constexpr int kM = kEmuTileM, kN = kEmuTileN / 2;  // a CTA takes half of a tile's columns
constexpr int kN2 = kEmuTileN;
constexpr int kChunk = kEmuBlock;  // reduction elements of a stage (64-byte rows)
constexpr int kSub = kChunk / kMmaK;
constexpr int kStages = 2;
constexpr int kGroup = 4;  // stages of one exact accumulation
constexpr int kPairs = kS / 2;  // pairs of diagonals (2p, 2p + 1)
constexpr int kTmemCols = 512;
constexpr int kEpiWarps = 16;              // 4 lane quadrants x 4 column groups
constexpr int kCols = kN / (kEpiWarps / 4);  // 16 columns per epilogue warp
constexpr int kThreads = (2 + kEpiWarps) * 32;
constexpr int kABytes = kM * kChunk * 2, kBBytes = kN * kChunk * 2;  // one digit of one operand
constexpr int kStageBytes = kS * (kABytes + kBBytes);
constexpr int kStgBytes = 32 * 8 * 8;  // per epilogue warp: 32 rows x 8 values on the way out
constexpr int kSmem = kStages * kStageBytes + kEpiWarps * kStgBytes + 256 + 1024;
constexpr int kLoBits = 32;   // value = (hi * 2^32 + lo) * 2^(ea + eb - 68)
constexpr int kUnit = -68;
constexpr int kBad = INT32_MAX;  // exponent of a row that holds an Inf or NaN
constexpr int kOut = INT32_MIN;  // ... of a row outside the operand

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

// Rows of a row-major matrix with an exponent per segment of a row: segment i
// starts at element seg[i] (a multiple of 64) and ends where the next begins; seg
// null: one segment, of K elements and zeros up to a multiple of 64.  kPairs: 16
// bytes may be loaded at once (src, ld and the ends are even).  First
// exps[i * rows + r], a warp per piece of a segment of a row; with several pieces
// exps holds values below every exponent before.
constexpr int kSegPiece = 8192;
template <bool kPairs>
__global__ void __launch_bounds__(256) k_segment_exps(const double* __restrict__ src, long long ld, long long rows,
                                                      int K, const long long* __restrict__ seg, int n_seg, int pieces,
                                                      int* __restrict__ exps) {
  const int lane = threadIdx.x & 31;
  const long long r = blockIdx.x * 8LL + threadIdx.x / 32;
  if (r >= rows) return;
  for (int j = blockIdx.y; j < n_seg * pieces; j += gridDim.y) {
    const int s = pieces == 1 ? j : j / pieces;
    const long long k0 = seg ? seg[s] : 0;
    const int end = static_cast<int>((s + 1 < n_seg ? seg[s + 1] : K) - k0);
    const int from = (j - s * pieces) * kSegPiece, len = min(end - from, kSegPiece);
    const double* x = src + r * ld + k0 + from;
    int be = 0;
    if (kPairs) {
#pragma unroll 4
      for (int k = lane; k < len / 2; k += 32) {
        const double2 v = reinterpret_cast<const double2*>(x)[k];
        be = max(be, max(biased_exp(v.x), biased_exp(v.y)));
      }
    } else {
#pragma unroll 8
      for (int k = lane; k < len; k += 32) be = max(be, biased_exp(x[k]));
    }
    be = __reduce_max_sync(0xffffffffu, be);
    if (lane != 0) continue;
    if (pieces == 1)
      exps[s * rows + r] = row_exp(be);
    else
      atomicMax(exps + s * rows + r, row_exp(be));
  }
}
// Then the digits, in blocks of one stage's 32 elements, [block][digit][row][32]: a
// tile of them is eight contiguous pieces of 8 KB.  In rows of K elements a tile's
// 1024 rows lay in pages of their own from some 50 atoms on, and every CTA reads
// its own tiles: step C took 28 ms where it now takes 21 (58 atoms).  A CTA takes
// 16 rows x 512 elements of segment blockIdx.z, so that it reads and writes within
// some thirty pages: 5.4 ms for both operands with the exponents' pass.  A row's
// whole segment per CTA, in one pass, wrote to 200 pages and took 7.5 ms.
constexpr int kSegRows = 16, kSegK = 512;
template <bool kPairs>
__global__ void __launch_bounds__(256) k_segment_digits(const double* __restrict__ src, long long ld, long long rows,
                                                        int K, const long long* __restrict__ seg, int n_seg,
                                                        const int* __restrict__ exps, __half* __restrict__ dig) {
  const int s = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long k0 = seg ? seg[s] : 0;
  const int len = static_cast<int>((s + 1 < n_seg ? seg[s + 1] : K) - k0);
  // a warp: 8 rows x one block, four lanes with 8 elements each per row
  const long long r = static_cast<long long>(blockIdx.x) * kSegRows + (warp & 1) * 8 + lane / 4;
  if (r >= rows) return;
  const int e = exps[s * rows + r];
  const double* x = src + r * ld + k0;
  __half* out = dig + (k0 / kChunk * kS * rows + r) * kChunk + lane % 4 * 8;
#pragma unroll 1
  for (int b = warp / 2; b < kSegK / kChunk; b += 4) {
    const int block = static_cast<int>(blockIdx.y) * (kSegK / kChunk) + b, k = block * kChunk + lane % 4 * 8;
    if (block * kChunk >= (len + 63) / 64 * 64) break;
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      if (kPairs) {
        double2 w = make_double2(0.0, 0.0);
        if (k + j < len) w = *reinterpret_cast<const double2*>(x + k + j);
        v[j] = w.x;
        v[j + 1] = w.y;
      } else {
        v[j] = k + j < len ? x[k + j] : 0.0;
        v[j + 1] = k + j + 1 < len ? x[k + j + 1] : 0.0;
      }
    }
    uint4 q[kS];
    digits8(v, e, q);
    __half* o = out + static_cast<long long>(block) * kS * rows * kChunk;
#pragma unroll
    for (int j = 0; j < kS; ++j) *reinterpret_cast<uint4*>(o + j * rows * kChunk) = q[j];
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
// Exponents of a warp's 32 rows (one per lane) and 16 columns (lanes 0-15, and
// again 16-31), with kOut and kBad taken out.
struct Exps {
  int row, col;
  bool row_in, row_bad;
  unsigned col_in, col_bad;  // per column
  __device__ Exps(int er, int ec) {
    row_in = er != kOut;
    row_bad = er == kBad;
    row = row_in && !row_bad ? er + kUnit : 0;
    col = ec != kOut && ec != kBad ? ec : 0;
    col_in = __ballot_sync(0xffffffffu, ec != kOut);
    col_bad = __ballot_sync(0xffffffffu, ec == kBad);
  }
  __device__ int sum(int j) const { return row + __shfl_sync(0xffffffffu, col, j); }
  __device__ bool in(int j) const { return row_in && ((col_in >> j) & 1u); }
  __device__ bool bad(int j) const { return row_bad || ((col_bad >> j) & 1u); }
};
// (hi 2^32 + lo) 2^e from a sum of partial sums, whose low parts are not
// carried yet.
__device__ __forceinline__ double sums_to_double(long long hi, long long lo, int e);
// (hi 2^32 + lo) 2^e rounded to nearest (ties away from zero), in about 35
// 32-bit integer operations: three on the FP64 pipe, 64 cycles each per warp
// and SM quarter, would take longer.
__device__ __forceinline__ double fixed_to_double(long long hi, uint32_t lo, int e) {
  const uint32_t sg = static_cast<uint32_t>(static_cast<int32_t>(static_cast<unsigned long long>(hi) >> 32) >> 31);
  uint32_t w2 = static_cast<uint32_t>(static_cast<unsigned long long>(hi) >> 32) ^ sg;
  uint32_t w1 = static_cast<uint32_t>(hi) ^ sg, w0 = lo ^ sg;
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, %2, 0;"
      : "+r"(w0), "+r"(w1), "+r"(w2)
      : "r"(sg & 1u));
  // leading word first; its first 64 significant bits (what follows is below
  // the rounding by 2^-11 of a unit)
  const bool z2 = w2 == 0u, z1 = z2 && w1 == 0u;
  const uint32_t a = z1 ? w0 : (z2 ? w1 : w2), b = z1 ? 0u : (z2 ? w0 : w1), c = z2 ? 0u : w0;
  const int s = __clz(static_cast<int>(a));
  uint32_t m1 = __funnelshift_l(b, a, s), m0 = __funnelshift_l(c, b, s), over;
  asm("add.cc.u32 %0, %0, 0x400;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, 0, 0;"
      : "+r"(m0), "+r"(m1), "=r"(over));
  const uint32_t f1 = (m1 >> 11) | (over << 21), f0 = __funnelshift_r(m0, m1, 11);
  // (f1 : f0) in [2^52, 2^53], value (f1 : f0) 2^ex
  const int ex = 43 - s - (z1 ? 64 : (z2 ? 32 : 0)) + e;
  const int be = ex + 1075;
  const uint32_t sign = sg & 0x80000000u;
  if (a != 0u && static_cast<unsigned>(be - 1) < 2045u)
    return __hiloint2double(static_cast<int>(((static_cast<uint32_t>(be - 1) << 20) + f1) | sign),
                            static_cast<int>(f0));
  if (a == 0u) return 0.0;
  const double d = ldexp(__hiloint2double(static_cast<int>((1074u << 20) + f1), static_cast<int>(f0)), ex);
  return sign ? -d : d;
}

__device__ __forceinline__ double sums_to_double(long long hi, long long lo, int e) {
  return fixed_to_double(hi + (lo >> kLoBits), static_cast<uint32_t>(lo), e);
}

// FP64 operations that are not to be speculated: an FP64 instruction takes the
// SM quarter's pipe for 64 cycles per warp, also where its result is not used.
__device__ __forceinline__ double mul_here(double a, double b) {
  double d;
  asm volatile("mul.rn.f64 %0, %1, %2;" : "=d"(d) : "d"(a), "d"(b));
  return d;
}
__device__ __forceinline__ double fma_here(double a, double b, double c) {
  double d;
  asm volatile("fma.rn.f64 %0, %1, %2, %3;" : "=d"(d) : "d"(a), "d"(b), "d"(c));
  return d;
}

// A lane holds eight consecutive values of its row; they leave row by row: lane
// l takes value l % 8 of rows l / 8, + 4, ... (item i of f(i, x)), so that a
// warp's access covers four rows of 64 contiguous bytes and not 32 rows of 8.
// All lanes call it.
// load(i) first, for all items together: what the values are to be added to.
template <class L, class F>
__device__ __forceinline__ void by_rows(unsigned long long* stg, int lane, const unsigned long long (&v)[8],
                                        const L& load, const F& f) {
#pragma unroll
  for (int j = 0; j < 8; ++j) stg[lane * 8 + (j ^ (lane & 7))] = v[j];
  __syncwarp();
  double old[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) old[i] = load(i);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 4 * i + (lane >> 3);
    f(i, stg[r * 8 + ((lane & 7) ^ (r & 7))], old[i]);
  }
  __syncwarp();
}
// The (hi, lo) of 32 rows, value(j, hi, lo) for column j, into 64-bit partial
// sums: element (r, c) at part + 2 (r * n + c) for r < rows, c < n; r, c: the
// warp's first row and column.  only: the one unit of its tile, which stores
// and does not add.
template <class V>
__device__ __forceinline__ void add_partial(unsigned long long* part, bool only, long long n, int rows, int r, int c,
                                            int lane, const V& value, unsigned long long* stg) {
  const int k = lane & 7;
  unsigned long long* p = part + ((r + (lane >> 3)) * n + c + (k >> 1)) * 2 + (k & 1);
  const int left = rows - r - (lane >> 3);
#pragma unroll
  for (int h = 0; h < kCols; h += 4) {
    unsigned long long v[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      long long hi;
      uint32_t lo;
      value(h + j, hi, lo);
      v[2 * j] = static_cast<unsigned long long>(hi);
      v[2 * j + 1] = lo;
    }
    const bool in = c + h + (k >> 1) < n;
    by_rows(stg, lane, v, [](int) { return 0.0; }, [&](int i, unsigned long long x, double) {
      unsigned long long* q = p + 8 * i * n + 2 * h;
      if (!in || 4 * i >= left) return;
      if (only)
        *q = x;
      else
        atomicAdd(q, x);
    });
  }
}

// ---------------------------------------------------------------------------
// dense products
// ---------------------------------------------------------------------------
struct GemmJob {
  int m, n, K, nt, n_items, ks, stages, tri, ktri, tri_off;
  double alpha, beta;
  int a_kind, accumulate;  // alpha 1 (0), -1 (1) or another (2); beta not 0
  double* C;
  long long ldc, cblk_stride, col0;
  int cblk;
  const int *ea, *eb;
  int per_z, za, zb;         // items and operand rows of one product of a batch
  long long c_z, a_z, b_z;   // C, A, B from one product to the next
  unsigned long long* part;  // [nz][m][n][2] integer sums, or null: C is written directly
  const double *A, *B;
  long long lda, ldb;
  int ta, tb;
  int blocked_a, blocked_b;  // digits in blocks (k_segment_digits), not in rows
  __device__ bool a_blocked() const { return blocked_a; }
  __device__ bool b_blocked() const { return blocked_b; }

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
    T.rb = x % nt * kN2;
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
  __device__ bool next(Tile&) const { return false; }
  __device__ bool skip(int ya, int yb) const { return tri && yb >= ya + kM + tri_off; }
  __device__ void half(Tile& T, int side) const {
    T.yb += side * kN;
    T.rb += side * kN;
  }
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
  __device__ double* place(int z, int r, int c) const {
    long long at = c;
    if (cblk) {
      const uint32_t q = static_cast<uint32_t>(c + col0), b = static_cast<uint32_t>(cblk);
      at = q / b * cblk_stride + q % b;
    }
    return C + z * c_z + r * ldc + at;
  }
  __device__ double combine(double v, double old) const {
    double w = a_kind == 0 ? v : -v;
    if (a_kind == 2) w = mul_here(alpha, v);
    if (accumulate) w = fma_here(beta, old, w);
    return w;
  }
  __device__ void store(int z, int r, int c, double v) const {
    double* p = place(z, r, c);
    *p = combine(v, accumulate ? *p : 0.0);
  }
  __device__ int row_exp(const Tile& T, int row) const { return T.ra + row < m ? ea[T.z * za + T.ra + row] : kOut; }
  __device__ int col_exp(const Tile& T, int c) const { return T.rb + c < n ? eb[T.z * zb + T.rb + c] : kOut; }
  __device__ void write(long long (&hi)[kCols], uint32_t (&lo)[kCols], const Tile& T, int row0, int lane, int c0,
                        int er, int ec, unsigned long long* stg) const {
    const int r = T.ra + row0, c = T.rb + c0;
    if (part) {
      add_partial(part + static_cast<long long>(T.z) * m * n * 2, ks == 1, n, m, r, c, lane,
                  [&](int j, long long& h, uint32_t& l) {
                    h = hi[j];
                    l = lo[j];
                  },
                  stg);
      return;
    }
    const int left = m - r - (lane >> 3);
    const Exps ex(er, ec);
#pragma unroll
    for (int h = 0; h < kCols; h += 8) {
      unsigned long long v[8];
      unsigned bad = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        v[j] = static_cast<unsigned long long>(
            __double_as_longlong(fixed_to_double(hi[h + j], lo[h + j], ex.sum(h + j))));
        if (ex.in(h + j) && ex.bad(h + j)) bad |= 1u << j;
      }
      if (__any_sync(0xffffffffu, bad != 0)) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if ((bad >> j) & 1u) v[j] = static_cast<unsigned long long>(
              __double_as_longlong(direct(T.z, r + lane, c + h + j)));
      }
      const int cc = c + h + (lane & 7);
      const bool in = cc < n;
      double* p = place(T.z, r + (lane >> 3), cc);
      by_rows(
          stg, lane, v, [&](int i) { return accumulate && in && 4 * i < left ? p[4 * i * ldc] : 0.0; },
          [&](int i, unsigned long long x, double old) {
            if (in && 4 * i < left) p[4 * i * ldc] = combine(__longlong_as_double(static_cast<long long>(x)), old);
          });
    }
  }
};
__global__ void k_gemm_finish(const GemmJob j, int nz) {
  const long long mn = static_cast<long long>(j.m) * j.n;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < mn * nz;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    // m n nz <= 2^28 here (k_splits)
    const int z = static_cast<int>(static_cast<unsigned>(i) / static_cast<unsigned>(mn));
    const unsigned e = static_cast<unsigned>(i - z * mn);
    const int r = static_cast<int>(e / static_cast<unsigned>(j.n)), c = static_cast<int>(e % static_cast<unsigned>(j.n));
    if (j.skip(r / kM * kM, c / kN2 * kN2)) continue;
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(j.part)[i];
    const int a = j.ea[z * j.za + r], b = j.eb[z * j.zb + c];
    j.store(z, r, c, a == kBad || b == kBad ? j.direct(z, r, c)
                                            : sums_to_double(static_cast<long long>(v.x),
                                                             static_cast<long long>(v.y), a + b + kUnit));
  }
}

// ---------------------------------------------------------------------------
// steps A / B of Eq. 3 in FP64: one tile = 128 rows of the A operand x 128 of
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
  double* out_;
  const double *pool, *G;
  const int* lam;
  int nao;
  __device__ static bool a_blocked() { return false; }
  __device__ static bool b_blocked() { return false; }
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
    T.b0 = e.z * kN2;
    T.ya = (mode == 0 ? tk.p_row0 : tk.g_row0) + T.a0;
    T.yb = (mode == 0 ? tk.g_row0 : tk.p_row0) + T.b0;
    T.n = (tk.K + kChunk - 1) / kChunk;
    return T;
  }
  __device__ bool next(Tile&) const { return false; }
  __device__ void half(Tile& T, int side) const {
    T.yb += side * kN;
    T.b0 += side * kN;
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
  __device__ int row_exp(const Tile& T, int row) const {
    const PanelTask64& tk = tasks[T.task];
    const int a = T.a0 + row;
    return mode == 0 ? (a < tk.N ? pe[tk.p_row0 + a] : kOut) : (a < R ? ge[r0 + a] : kOut);
  }
  __device__ int col_exp(const Tile& T, int c) const {
    const PanelTask64& tk = tasks[T.task];
    const int b = T.b0 + c;
    return mode == 0 ? (b < R ? ge[r0 + b] : kOut) : (b < tk.N ? pe[tk.p_row0 + b] : kOut);
  }
  __device__ void write(long long (&hi)[kCols], uint32_t (&lo)[kCols], const Tile& T, int row0, int lane, int c0,
                        int er, int ec, unsigned long long*) const {
    const PanelTask64& tk = tasks[T.task];
    const int a = T.a0 + row0 + lane, b = T.b0 + c0, nsig = tk.nsig;
    const int pw = (mode == 0 ? a : b) / nsig;
    int sp = (mode == 0 ? a : b) - pw * nsig;
    double* o = out_ + static_cast<long long>(tk.p0 + pw - P0b) * ldk;  // where the first column goes,
    long long next, wrap = 0;  // from one column to the next, and (mode 1) on to the next RI row
    if (mode == 0) {
      next = nsig;
      o += tk.seg + sp + (r0 + b) * next;
    } else {
      next = er == kOut ? 0 : rowmul[a];
      o += (er == kOut ? 0 : rowbase[a]) + (tk.aom + sp) * next;
      wrap = ldk - nsig * next;
    }
    const Exps ex(er, ec);
#pragma unroll
    for (int j = 0; j < kCols; ++j) {
      double x = fixed_to_double(hi[j], lo[j], ex.sum(j));
      if (ex.in(j)) {
        if (ex.bad(j)) x = mode == 0 ? direct(tk, a, r0 + b + j) : direct(tk, b + j, r0 + a);
        *o = x;
      }
      o += next;
      if (mode == 1 && ++sp == nsig) {
        sp = 0;
        o += wrap;
      }
    }
  }
};

// ---------------------------------------------------------------------------
// step C in FP64: chi[P][Q] -= sum over the unit's slabs of X[P][k] Y[Q][k]
//
// X and Y of two distant auxiliary functions overlap only where both are far
// below their largest magnitudes: digits below one exponent per row would leave
// such an element of chi an error of 2^-61 of the product of the rows' maxima
// (58-atom ribbon: 1.9e-10 of chi between its ends, FP64 sums 4e-14).  So the
// rows have an exponent per sigma-atom, over which they vary little where they
// matter, and the sums over one sigma-atom (a piece of a unit) are shifted to
// the larger of all pieces' scales, 2^(pair - 68) with pair the largest sum of
// the two exponents, before they are added as integers.
// ---------------------------------------------------------------------------
// (hi 2^32 + lo) / 2^s rounded to nearest, s >= 0.
__device__ __forceinline__ void shift_round(long long& hi, uint32_t& lo, int s) {
  if (s <= 0) return;
  if (s > 95) {
    hi = 0;
    lo = 0;
    return;
  }
  const uint32_t sg = static_cast<uint32_t>(static_cast<int32_t>(static_cast<unsigned long long>(hi) >> 32) >> 31);
  uint32_t w2 = static_cast<uint32_t>(static_cast<unsigned long long>(hi) >> 32), w1 = static_cast<uint32_t>(hi),
           w0 = lo;
  // by s - 1, then one is added and the last bit goes
  const int t = s - 1, words = t >> 5, bits = t & 31;
  const uint32_t a = words == 0 ? w0 : (words == 1 ? w1 : w2);
  const uint32_t b = words == 0 ? w1 : (words == 1 ? w2 : sg), c = words == 0 ? w2 : sg;
  w0 = __funnelshift_r(a, b, bits);
  w1 = __funnelshift_r(b, c, bits);
  w2 = __funnelshift_r(c, sg, bits);
  asm("add.cc.u32 %0, %0, 1;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, %2, 0;" : "+r"(w0), "+r"(w1), "+r"(w2));
  lo = __funnelshift_r(w0, w1, 1);
  w1 = __funnelshift_r(w1, w2, 1);
  w2 = static_cast<uint32_t>(static_cast<int32_t>(w2) >> 1);
  hi = static_cast<long long>((static_cast<unsigned long long>(w2) << 32) | w1);
}

struct Chi64Job {
  const int *unit_tile, *unit_first, *unit_count, *n_units;
  const int* tasks;
  const int* counts;
  int nslab, nqt, P0, prow, nri;
  int per;  // slabs of a sigma-atom
  const long long* slab_k0;
  const int* slab_len;
  const int *ex, *ey;  // exponents [sigma-atom][row]
  const int* pair;     // [nri][prow]: exponent of element (P, Q)'s integers
  double* chi;
  unsigned long long* part;
  const double *X, *Y;
  long long ldk;
  __device__ static bool a_blocked() { return true; }
  __device__ static bool b_blocked() { return true; }
  struct Tile {
    int ya, yb, n, id;
    const int* list;  // the piece's entries, and how many the unit has from here on
    int cnt, left, atom;
  };
  __device__ int items() const { return *n_units; }
  __device__ void piece(Tile& T) const {
    T.atom = T.list[0] / per;
    T.n = 0;
    for (T.cnt = 0; T.cnt < T.left && T.list[T.cnt] / per == T.atom; ++T.cnt) T.n += slab_len[T.list[T.cnt]] / kChunk;
  }
  __device__ Tile tile(int u) const {
    Tile T;
    T.id = unit_tile[u];
    T.ya = T.id / nqt * kM;
    T.yb = T.id % nqt * kN2;
    T.left = unit_count[u];
    T.list = tasks + static_cast<long long>(T.id) * nslab + unit_first[u];
    piece(T);
    return T;
  }
  __device__ bool next(Tile& T) const {
    T.left -= T.cnt;
    T.list += T.cnt;
    if (T.left <= 0) return false;
    piece(T);
    return true;
  }
  __device__ void half(Tile& T, int side) const { T.yb += side * kN; }
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
  __device__ int row_exp(const Tile& T, int row) const {
    return T.ya + row < prow ? ex[static_cast<long long>(T.atom) * prow + T.ya + row] : kOut;
  }
  __device__ int col_exp(const Tile& T, int c) const {
    return T.yb + c < nri ? ey[static_cast<long long>(T.atom) * nri + T.yb + c] : kOut;
  }
  __device__ void write(long long (&hi)[kCols], uint32_t (&lo)[kCols], const Tile& T, int row0, int lane, int c0,
                        int er, int ec, unsigned long long* stg) const {
    const int p0 = T.ya + row0, q0 = T.yb + c0;
    const Exps es(er, ec);
    const int* e = pair + static_cast<long long>(q0) * prow + p0 + lane;
    add_partial(part, false, nri, prow, p0, q0, lane,
                [&](int j, long long& h, uint32_t& l) {
                  h = hi[j];
                  l = lo[j];
                  const int scale = es.sum(j) - kUnit;
                  if (es.in(j)) {
                    const int to = e[static_cast<long long>(j) * prow];
                    if (to != kBad) shift_round(h, l, to - scale);
                  }
                },
                stg);
  }
};
// pair[q][p] = the largest sum over the sigma-atoms of ex[s][p] + ey[s][q], kBad
// where one of them is; part = 0.
__global__ void __launch_bounds__(256) k_pair_exps(const int* __restrict__ ex, const int* __restrict__ ey, int ns,
                                                   int prow, int nri, int* __restrict__ pair,
                                                   ulonglong2* __restrict__ part) {
  for (int i = threadIdx.x >> 5; i < 32; i += 8) {
    const int pp = blockIdx.x * 32 + i, qq = blockIdx.y * 32 + (threadIdx.x & 31);
    if (pp < prow && qq < nri) part[static_cast<long long>(pp) * nri + qq] = make_ulonglong2(0, 0);
  }
  const int p = blockIdx.x * 32 + (threadIdx.x & 31);
  const int q0 = blockIdx.y * 32 + (threadIdx.x >> 5) * 4;
  if (p >= prow) return;
  int m[4] = {kOut, kOut, kOut, kOut};
#pragma unroll 4
  for (int s = 0; s < ns; ++s) {
    const int a = ex[static_cast<long long>(s) * prow + p];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (q0 + i < nri) {
        const int b = ey[static_cast<long long>(s) * nri + q0 + i];
        m[i] = max(m[i], a == kBad || b == kBad ? kBad : a + b);
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (q0 + i < nri) pair[static_cast<long long>(q0 + i) * prow + p] = m[i];
}
__global__ void __launch_bounds__(256) k_chi64_finish(const Chi64Job j) {
  __shared__ int t[32][33];
  const int q0 = blockIdx.x * 32, p0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8)
    if (q0 + i < j.nri && p0 + tx < j.prow) t[i][tx] = j.pair[static_cast<long long>(q0 + i) * j.prow + p0 + tx];
  __syncthreads();
  const int q = q0 + tx;
  ulonglong2 v[4];
  double old[4];
  bool on[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int p = p0 + ty + 8 * i;
    on[i] = p < j.prow && q < j.nri && j.counts[p / kM * j.nqt + q / kN2] != 0;
    if (!on[i]) continue;
    v[i] = reinterpret_cast<const ulonglong2*>(j.part)[static_cast<long long>(p) * j.nri + q];
    old[i] = j.chi[static_cast<long long>(j.P0 + p) * j.nri + q];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (!on[i]) continue;
    const int p = p0 + ty + 8 * i, e = t[tx][ty + 8 * i];
    j.chi[static_cast<long long>(j.P0 + p) * j.nri + q] =
        old[i] - (e == kBad ? j.direct(p / kM * j.nqt + q / kN2, p, q)
                            : sums_to_double(static_cast<long long>(v[i].x), static_cast<long long>(v[i].y), e + kUnit));
  }
}

// ---------------------------------------------------------------------------
// the persistent kernel: warp 0 TMA producer, warp 1 MMA issuer, warps 2-17
// epilogue; every wait is bounded (tc_ptx.h)
// ---------------------------------------------------------------------------
// eight columns from each of two addresses, both loads in flight together
__device__ __forceinline__ void tmem_ld8x2(uint32_t a0, uint32_t a1, uint32_t (&r)[8], uint32_t (&s)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(a0));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]), "=r"(s[7])
               : "r"(a1));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(s[0]), "+r"(s[1]), "+r"(s[2]), "+r"(s[3]), "+r"(s[4]), "+r"(s[5]), "+r"(s[6]), "+r"(s[7])
               :
               : "memory");
}
// An accumulator (an integer in FP32) as int.  small: |v| <= 2^22, as for
// diagonals 0-2 (the leading digits are at most 64): adding 1.5 2^23 puts the
// integer in the low bits, on the FP32 pipe at eight times the rate of the
// conversion.
__device__ __forceinline__ int to_int(uint32_t v, bool small) {
  if (small) return __float_as_int(__uint_as_float(v) + 12582912.f) - 0x4B400000;
  return __float2int_rn(__uint_as_float(v));
}

// Adds the accumulators of diagonals 2p and 2p + 1 into this thread's columns:
// pairs 0 and 1, times 2^24, 2^16, 2^8 and 1, into hi; pairs 2 and 3 the same
// into lo, with the carry into hi at once (lo as 64 bits would cost the
// registers that the way out needs).
template <bool kHi>
__device__ __forceinline__ bool add_pair(int p, int q, uint64_t* acc_full, uint64_t* acc_empty, uint32_t parity,
                                         volatile int* abort_flag, uint32_t row_addr, int lane,
                                         long long (&hi)[kCols], uint32_t (&lo)[kCols]) {
  if (!mbar_wait_warp(&acc_full[p], parity, abort_flag)) return false;
  tc_fence_after();
  const int w0 = q ? 1 << 8 : 1 << 24, w1 = q ? 1 : 1 << 16;
#pragma unroll
  for (int h = 0; h < kCols; h += 8) {  // 16 columns at once would spill
    uint32_t r0[8], r1[8];
    tmem_ld8x2(row_addr + static_cast<uint32_t>(2 * p * kN + h),
               row_addr + static_cast<uint32_t>((2 * p + 1) * kN + h), r0, r1);
    if (h + 8 == kCols) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[p]);
    }
    // diagonals 0 to 2 are at most 2^22
    if (kHi && q == 0) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        hi[h + j] += static_cast<long long>(to_int(r0[j], true)) * w0;
        hi[h + j] += static_cast<long long>(to_int(r1[j], true)) * w1;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        long long t = kHi ? hi[h + j] : static_cast<long long>(lo[h + j]);
        t += static_cast<long long>(to_int(r0[j], false)) * w0;
        t += static_cast<long long>(to_int(r1[j], false)) * w1;
        if (kHi) {
          hi[h + j] = t;
        } else {
          hi[h + j] += t >> kLoBits;
          lo[h + j] = static_cast<uint32_t>(t);
        }
      }
    }
  }
  return true;
}

template <class Job>
__global__ void __launch_bounds__(kThreads, 1)
    k_emu(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const Job job,
          int stall, int* __restrict__ err_flag) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* staging = smem + kStages * kStageBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(staging + kEpiWarps * kStgBytes);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;
  uint64_t* acc_empty = acc_full + kPairs;
  uint64_t* drain = acc_empty + kPairs;
  uint64_t* never = drain + 1;  // arrived at by nothing (stall test hook)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = __reduce_max_sync(0xffffffffu, threadIdx.x / 32), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < kPairs; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kEpiWarps);
    }
    mbar_init(drain, 1);
    mbar_init(never, 1);
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
  const int side = blockIdx.x & 1, first = blockIdx.x >> 1, step = gridDim.x >> 1;

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool armed[kStages] = {};
      uint32_t armed_parity[kStages] = {};
      bool ok = true;
      for (int t = first; t < n_items && ok; t += step) {
        typename Job::Tile T = job.tile(t);
        job.half(T, side);
        do {
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
            const int x = it.next(), z = x / kChunk * kS;
            const bool ba = job.a_blocked(), bb = job.b_blocked();
            tma_load_3d(st, &map_a, ba ? 0 : x, T.ya, ba ? z : 0, &full[stage]);
            tma_load_3d(st + kS * kABytes, &map_b, bb ? 0 : x, T.yb, bb ? z : 0, &full[stage]);
            if (++stage == kStages) {
              stage = 0;
              phase ^= 1u;
            }
          }
        } while (ok && job.next(T));
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
    constexpr uint32_t one = idesc_f32(kM, kN, true), two = idesc_f32(kM, 2 * kN, true);
    const uint32_t lead = elect_one();
    const uint32_t tmu = __reduce_max_sync(0xffffffffu, tmem);
    int stage = 0;
    uint32_t phase = 0, aphase = 1;
    bool ok = true, issued = false;
    for (int t = first; t < n_items && ok; t += step) {
      typename Job::Tile T = job.tile(t);
      do {
        const int n = __reduce_max_sync(0xffffffffu, job.nchunks(T));
        for (int i = 0; i < n && ok; ++i) {
          ok = mbar_wait_warp(&full[stage], phase, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const bool first = (i % kGroup) == 0, last = (i % kGroup) == kGroup - 1 || i == n - 1;
          const uint64_t da = desc_sw64(smem_u32(smem + stage * kStageBytes));
          const uint32_t a_lo = static_cast<uint32_t>(da), hi = static_cast<uint32_t>(da >> 32);
          const uint32_t b_lo = a_lo + static_cast<uint32_t>((kS * kABytes) >> 4);
#pragma unroll
          for (int p = 0; p < kPairs; ++p) {
            if (first) {
              ok = mbar_wait_warp(&acc_empty[p], aphase, abort_flag);
              if (!ok) break;
              tc_fence_after();
            }
            if (lead) {
              // digit a of A with digits 2p - a and 2p - a + 1 of B, whose rows
              // follow one another, into the two accumulators side by side; the
              // last digit of A only meets digit 0
              const uint32_t acc = tmu + static_cast<uint32_t>(2 * p * kN);
#pragma unroll
              for (int a = 0; a <= 2 * p + 1; ++a)
#pragma unroll
                for (int k = 0; k < kSub; ++k) {
                  const uint32_t da_lo = a_lo + static_cast<uint32_t>((a * kABytes + k * kMmaK * 2) >> 4);
                  if (a <= 2 * p)
                    mma_f16_lo(acc, da_lo, b_lo + static_cast<uint32_t>(((2 * p - a) * kBBytes + k * kMmaK * 2) >> 4),
                               hi, two, (a | k) ? 1u : (first ? 0u : 1u));
                  else
                    mma_f16_lo(acc + kN, da_lo, b_lo + static_cast<uint32_t>((k * kMmaK * 2) >> 4), hi, one, 1u);
                }
              if (last) mma_commit(&acc_full[p]);
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
      } while (ok && job.next(T));
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
    unsigned long long* stg = reinterpret_cast<unsigned long long*>(staging + (warp - 2) * kStgBytes);
    const uint32_t row_addr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(c0);
    uint32_t aphase = 0;
    // test hook: the bounded wait gives up and the kernel reports a time-out
    bool ok = stall ? mbar_wait_warp(never, 0, abort_flag) : true;
    for (int t = first; t < n_items && ok; t += step) {
      typename Job::Tile T = job.tile(t);
      if (job.nchunks(T) == 0) continue;
      job.half(T, side);
      do {
        const int n = job.nchunks(T);
        // exponents of this lane's row and of column c0 + lane % 16, loaded here:
        // beside the stores they would be fetched one by one
        const int er = job.row_exp(T, quad * 32 + lane), ec = job.col_exp(T, c0 + lane % kCols);
        // value = hi 2^32 + lo: 48 registers for 16 columns
        long long hi[kCols];
        uint32_t lo[kCols];
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
          hi[j] = 0;
          lo[j] = 0;
        }
        for (int i = 0; i < n && ok; i += kGroup, aphase ^= 1u) {
          // pairs 0 and 1 (diagonals 0-3) into hi, 2 and 3 into lo; rolled, for
          // the instruction cache
#pragma unroll 1
          for (int p = 0; p < kPairs / 2 && ok; ++p)
            ok = add_pair<true>(p, p, acc_full, acc_empty, aphase, abort_flag, row_addr, lane, hi, lo);
#pragma unroll 1
          for (int p = 0; p < kPairs / 2 && ok; ++p)
            ok = add_pair<false>(kPairs / 2 + p, p, acc_full, acc_empty, aphase, abort_flag, row_addr, lane, hi, lo);
        }
        if (!ok) break;
        job.write(hi, lo, T, quad * 32, lane, c0, er, ec, stg);
      } while (job.next(T));
      if (!ok) break;
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
  k_emu<Job><<<2 * std::min(n_items, std::max(sms / 2, 1)), kThreads, kSmem, st>>>(ma, mb, job, tc_stall_test(), err_flag);
  return 0;
}

// tensor map of an operand's tiles of box_rows rows x one stage x all digits
int operand_map(CUtensorMap* map, const EmuOp& op, int box_rows) {
  const long long rows = op.s.nz > 1 ? op.stride_rows : op.s.rows;
  if (op.blocked)
    return make_digit_map(map, op.dig, kChunk, rows, op.stride_rows, op.kp / kChunk * kS, kChunk, box_rows, kS);
  return make_digit_map(map, op.dig, op.kp, rows, op.stride_rows, kS, kChunk, box_rows, kS);
}

// K splits of an m x n product: the number of units that makes the last wave
// over the 76 pairs of CTAs short.  Costs in stages (about 1.7 us each): a unit's
// start and end about 3, clearing the partial sums about 3 in all.
int k_splits(long long m, long long n, int K, int nz) {
  const long long tiles = ((m + kM - 1) / kM) * ((n + kN2 - 1) / kN2) * nz;
  const long long stages = (K + kChunk - 1) / kChunk;
  if (m * n * nz > (1ll << 28)) return 1;  // 4 GB of partial sums
  long long best = 1, cost = 0;
  for (long long ks = 1; ks <= 64 && ks * 4 <= std::max(stages, 4ll); ++ks) {
    const long long c = (tiles * ks + 75) / 76 * ((stages + ks - 1) / ks + 3) + (ks > 1 ? 3 : 0);
    if (ks == 1 || c < cost) {
      cost = c;
      best = ks;
    }
  }
  return static_cast<int>(best);
}

}  // namespace emu

void launch_emu_prep_segments(EmuOp& op, const EmuSrc& s, const long long* seg, int n_seg, int max_len,
                              cudaStream_t st) {
  op.s = s;
  op.stride_rows = s.rows;
  op.kp = emu_kp(s.K);
  op.blocked = true;
  if (s.rows <= 0 || n_seg <= 0) return;
  const int pieces = std::max(1, (max_len + emu::kSegPiece - 1) / emu::kSegPiece);
  const dim3 ge(static_cast<unsigned>((s.rows + 7) / 8), static_cast<unsigned>(std::min(n_seg * pieces, 65535)));
  if (pieces > 1) cudaMemsetAsync(op.exps, 0x80, static_cast<size_t>(s.rows) * n_seg * sizeof(int), st);
  const dim3 gd(static_cast<unsigned>((s.rows + emu::kSegRows - 1) / emu::kSegRows),
                static_cast<unsigned>((emu_kp(max_len) + emu::kSegK - 1) / emu::kSegK), n_seg);
  __half* dig = static_cast<__half*>(op.dig);
  if (s.ld % 2 == 0 && s.K % 2 == 0 && reinterpret_cast<uintptr_t>(s.src) % 16 == 0) {
    emu::k_segment_exps<true><<<ge, 256, 0, st>>>(s.src, s.ld, s.rows, s.K, seg, n_seg, pieces, op.exps);
    emu::k_segment_digits<true><<<gd, 256, 0, st>>>(s.src, s.ld, s.rows, s.K, seg, n_seg, op.exps, dig);
  } else {
    emu::k_segment_exps<false><<<ge, 256, 0, st>>>(s.src, s.ld, s.rows, s.K, seg, n_seg, pieces, op.exps);
    emu::k_segment_digits<false><<<gd, 256, 0, st>>>(s.src, s.ld, s.rows, s.K, seg, n_seg, op.exps, dig);
  }
}

void launch_emu_prep(EmuOp& op, const EmuSrc& s, cudaStream_t st) {
  // long rows in blocks (a whole row is the one segment)
  if (!s.trans && s.nz == 1 && s.K >= kEmuBlockedK) return launch_emu_prep_segments(op, s, nullptr, 1, s.K, st);
  op.s = s;
  const long long rows = s.rows * s.nz;
  op.stride_rows = rows;
  op.kp = emu_kp(s.K);
  op.blocked = false;
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

// Sums go out as integers and a second kernel rounds them, also where K is not
// split, as long as they stay in the L2 cache: beside the accumulators there
// are few registers left for the conversion, which takes 20000 cycles per tile
// there (a stage takes 3400), the integers alone 3500.
size_t emu_gemm_ws_bytes(long long m, long long n, int K, int nz) {
  const size_t bytes = static_cast<size_t>(m) * n * 16 * nz;
  return bytes <= (size_t(96) << 20) || emu::k_splits(m, n, K, nz) > 1 ? bytes : 0;
}

int launch_emu_gemm(const EmuOp& A, const EmuOp& B, const EmuGemm& g, void* ws, int* err_flag,
                    cudaStream_t st) {
  const int m = static_cast<int>(A.s.rows), n = static_cast<int>(B.s.rows);
  if (m <= 0 || n <= 0) return 0;
  CUtensorMap ma, mb;
  if (emu::operand_map(&ma, A, emu::kM) || emu::operand_map(&mb, B, emu::kN)) return -2;
  emu::GemmJob j{};
  j.m = m;
  j.n = n;
  j.K = A.s.K;
  j.nt = (n + emu::kN2 - 1) / emu::kN2;
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
  j.a_kind = g.alpha == 1.0 ? 0 : (g.alpha == -1.0 ? 1 : 2);
  j.accumulate = g.beta != 0.0;
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
  j.blocked_a = A.blocked;
  j.blocked_b = B.blocked;
  j.B = B.s.src;
  j.ldb = B.s.ld;
  j.tb = B.s.trans;
  j.part = static_cast<unsigned long long*>(ws);
  if (j.ks > 1) {
    cudaMemsetAsync(ws, 0, static_cast<size_t>(m) * n * 16 * nz, st);
  }
  const int rc = emu::launch(ma, mb, j, j.n_items, err_flag, st);
  if (rc) return rc;
  if (j.part) {
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
                     x ? emu::kM : emu::kN, kEmuSlices) ||
      make_digit_map(&mg, p.g_dig, p.g_kp, p.g_rows, p.g_rows, kEmuSlices, emu::kChunk, x ? emu::kN : emu::kM,
                     kEmuSlices))
    return -2;
  emu::Panel64Job j{p.tiles, p.n_tiles, p.mode, p.R,  p.r0,   p.P0b, p.tasks, p.ldk, p.rowbase,
                    p.rowmul, p.panel_exps, p.g_exps, p.out, p.pool, p.G, p.lam, p.nao};
  return x ? emu::launch(mp, mg, j, p.n_tiles, err_flag, st) : emu::launch(mg, mp, j, p.n_tiles, err_flag, st);
}

int launch_chi64(const EmuOp& x, const EmuOp& y, const Chi64Args& c, int* err_flag, cudaStream_t st) {
  CUtensorMap mx, my;
  if (emu::operand_map(&mx, x, emu::kM) || emu::operand_map(&my, y, emu::kN)) return -2;
  emu::Chi64Job j{c.units.u_tile, c.units.u_first, c.units.u_count, c.units.n_units, c.tasks, c.counts, c.nslab,
                  c.nqt, c.P0, c.prow, c.nri, c.per, c.slab_k0, c.slab_len, x.exps, y.exps, c.pair, c.chi,
                  static_cast<unsigned long long*>(c.part), x.s.src, y.s.src, x.s.ld};
  const unsigned gp = static_cast<unsigned>((c.prow + 31) / 32), gq = static_cast<unsigned>((c.nri + 31) / 32);
  emu::k_pair_exps<<<dim3(gp, gq), 256, 0, st>>>(x.exps, y.exps, c.nslab / c.per, c.prow, c.nri, c.pair,
                                                  static_cast<ulonglong2*>(c.part));
  const int rc = emu::launch(mx, my, j, INT32_MAX, err_flag, st);
  if (rc) return rc;
  emu::k_chi64_finish<<<dim3(gq, gp), 256, 0, st>>>(j);
  return 0;
}

}  // namespace gw
