// FP64 matrix products on the tensor cores from exact integer digits
// (k_emu.cu): operand preparation, the dense product and the FP64 forms of
// steps A, B and C of Eq. 3.
#pragma once

#include <cuda_runtime.h>

#include "gw_internal.h"

namespace gw {

constexpr int kEmuSlices = 8;   // digits per operand element
constexpr int kEmuTileM = 128;  // rows (A operand) and columns (B operand) of a tile
constexpr int kEmuTileN = 64;

// A matrix to be used as an operand: rows x K, element (r, k) at
// src[r * ld + k], or src[k * ld + r] when trans.
struct EmuSrc {
  const double* src = nullptr;
  long long ld = 0, rows = 0;
  int K = 0;
  bool trans = false;
};
// The same as digits: [kEmuSlices][stride_rows][kp] binary16, kp a multiple of
// 64, zero for k >= K, and per row the power of two above its largest
// magnitude.  The FP64 values are read again only for rows that hold an Inf
// or NaN.
struct EmuOp {
  void* dig = nullptr;
  int* exps = nullptr;
  long long stride_rows = 0;
  int kp = 0;
  EmuSrc s;
  EmuOp slice_rows(long long r0, long long n) const;  // rows [r0, r0 + n)
};
inline EmuOp EmuOp::slice_rows(long long r0, long long n) const {
  EmuOp o = *this;
  o.dig = static_cast<char*>(dig) + r0 * kp * 2;
  o.exps = exps + r0;
  o.s.src = s.src + (s.trans ? r0 : r0 * s.ld);
  o.s.rows = n;
  return o;
}
inline int emu_kp(int k) { return (k + 63) / 64 * 64; }
inline size_t emu_dig_bytes(long long rows, int k) {
  return static_cast<size_t>(kEmuSlices) * rows * emu_kp(k) * 2;
}
// Digits and exponents of s into op.dig (emu_dig_bytes) and op.exps (s.rows
// ints; twice that when trans).
void launch_emu_prep(EmuOp& op, const EmuSrc& s, cudaStream_t st);

// C[r * ldc + c] = alpha * sum_k A[r][k] B[c][k] + beta * C, with C's columns
// in blocks of cblk (0: one block) cblk_stride elements apart.
//   tri 1: only the tiles that touch r + tri_off >= c are computed
//   ktri 1: A[r][k] is zero for k < r + tri_off: those stages are left out
struct EmuGemm {
  double alpha = 1.0, beta = 0.0;
  double* C = nullptr;
  long long ldc = 0;
  int tri = 0, ktri = 0;
  long long tri_off = 0;
  int cblk = 0;
  long long cblk_stride = 0, col0 = 0;  // col0: index of B's first row in the blocks
};
// Bytes of the partial-sum workspace of a product (0: not split along K).
size_t emu_gemm_ws_bytes(long long m, long long n, int K);
// Returns 0, or a negative set-up error.  err_flag as for the other
// tensor-core launchers (k_tc.h).
int launch_emu_gemm(const EmuOp& A, const EmuOp& B, const EmuGemm& g, void* ws, int* err_flag,
                    cudaStream_t st);

// The same on the work buffers of a context (gw_fp64.cu).  Between emu_begin
// and emu_end of one call; names tell apart operands in use together.
int emu_begin(gw_ctx* ctx, cudaStream_t st);
int emu_prep(gw_ctx* ctx, const char* name, const EmuSrc& s, EmuOp* op, cudaStream_t st);
int emu_mm(gw_ctx* ctx, const EmuOp& A, const EmuOp& B, const EmuGemm& g, cudaStream_t st);
// Product of two matrices.  Operands beyond 4 GB of digits go in row chunks;
// keep (may be null): on a later call with the same A, its digits are reused
// where they are whole (keep->dig set by the first call).
int emu_product(gw_ctx* ctx, const EmuSrc& A, const EmuSrc& B, const EmuGemm& g, EmuOp* keep,
                cudaStream_t st);
// G^occ(tau), G^virt(tau) of Eq. 2 from the context's orbitals; cso, csv:
// scratch for the scaled orbitals (n_AO x n_occ, n_AO x n_virt).
int greens_fp64(gw_ctx* ctx, double tau, double* cso, double* csv, double* g_occ, double* g_virt, cudaStream_t st);
// Reads the error flag after the stream has been synchronised.
int emu_end(gw_ctx* ctx, const char* call);

}  // namespace gw
