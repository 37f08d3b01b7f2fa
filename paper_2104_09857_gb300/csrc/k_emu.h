// FP64 matrix products on the tensor cores from exact integer digits
// (k_emu.cu): operand preparation, the dense product and the FP64 forms of
// steps A, B and C of Eq. 3.
#pragma once

#include <cuda_runtime.h>

#include "gw_internal.h"
#include "k_tc.h"

namespace gw {

constexpr int kEmuSlices = 8;   // digits per operand element
constexpr int kEmuProducts = 36;  // digit pairs of a product
constexpr int kEmuTileM = 128;  // rows (A operand) and columns (B operand) of a tile
constexpr int kEmuTileN = 128;
constexpr int kEmuBlock = 32;     // reduction elements of a stage
// Rows of this length and more are kept in blocks: a tile's 1024 rows of digits
// would lie 128 KB apart.
constexpr int kEmuBlockedK = 65536;

// A matrix to be used as an operand: rows x K, element (r, k) at
// src[r * ld + k], or src[k * ld + r] when trans.
struct EmuSrc {
  const double* src = nullptr;
  long long ld = 0, rows = 0;
  int K = 0;
  bool trans = false;
  // several matrices of `rows` rows each, z_stride elements apart, one below
  // the other in the digits (not with trans)
  int nz = 1;
  long long z_stride = 0;
};
// The same as digits: [kEmuSlices][stride_rows][kp] binary16, kp a multiple of
// 64, zero for k >= K (blocked: in blocks of kEmuBlock elements of all rows, as
// k_segment_digits says), and per row the power of two above its largest
// magnitude.  The FP64 values are read again only for rows that hold an Inf
// or NaN.
struct EmuOp {
  void* dig = nullptr;
  int* exps = nullptr;
  long long stride_rows = 0;
  int kp = 0;
  bool blocked = false;
  EmuSrc s;
  EmuOp slice_rows(long long r0, long long n) const;  // rows [r0, r0 + n)
};
inline EmuOp EmuOp::slice_rows(long long r0, long long n) const {
  EmuOp o = *this;
  o.dig = static_cast<char*>(dig) + r0 * (blocked ? kEmuBlock : kp) * 2;
  o.exps = exps + r0;
  o.s.src = s.src + (s.trans ? r0 : r0 * s.ld);
  o.s.rows = n;
  return o;
}
inline int emu_kp(int k) { return (k + 63) / 64 * 64; }
inline size_t emu_dig_bytes(long long rows, int k) {
  return static_cast<size_t>(kEmuSlices) * rows * emu_kp(k) * 2;
}
// Digits and exponents of s into op.dig (emu_dig_bytes) and op.exps (s.nz *
// s.rows ints; twice that when trans).
void launch_emu_prep(EmuOp& op, const EmuSrc& s, cudaStream_t st);

// C[r * ldc + c] = alpha * sum_k A[r][k] B[c][k] + beta * C, with C's columns
// in blocks of cblk (0: one block) cblk_stride elements apart.
//   tri 1: only the tiles that touch r + tri_off >= c are computed
//   ktri 1: A[r][k] is zero for k < r + tri_off: those stages are left out
// With A.s.nz > 1 the same for every pair of matrices (B may be one matrix),
// C's c_zstride elements apart.
struct EmuGemm {
  double alpha = 1.0, beta = 0.0;
  double* C = nullptr;
  long long ldc = 0;
  int tri = 0, ktri = 0;
  long long tri_off = 0;
  int cblk = 0;
  long long cblk_stride = 0, col0 = 0;  // col0: index of B's first row in the blocks
  long long c_zstride = 0;
};
// Bytes of the partial-sum workspace of a product (0: not split along K).
size_t emu_gemm_ws_bytes(long long m, long long n, int K, int nz = 1);
// Returns 0, or a negative set-up error.  err_flag as for the other
// tensor-core launchers (k_tc.h).
int launch_emu_gemm(const EmuOp& A, const EmuOp& B, const EmuGemm& g, void* ws, int* err_flag,
                    cudaStream_t st);

// The same with an exponent per segment of a row, for step C: segment i starts at
// element seg[i] of the row (a multiple of 64; in device memory) and is max_len
// long at most (seg null: the row is one segment).  s.nz = 1, not s.trans;
// op.exps holds n_seg * s.rows ints, [segment][row]; the digits lie in blocks.
void launch_emu_prep_segments(EmuOp& op, const EmuSrc& s, const long long* seg, int n_seg, int max_len,
                              cudaStream_t st);

// One panel problem of the FP64 steps A / B: digits of the panel's rows from
// p_row0, of G's rows (gathered on its lambda functions) from g_row0.
struct PanelTask64 {
  long long panel_off, seg;  // seg: K offset of the owner's segment in X (mode 0)
  int p_row0, g_row0, K, N, npw, nsig, p0, aom, lam_off, pad;
};
// Digits of all owner panels ([K][N] each in pool): rows row0[i].., pitch kp;
// be, exps: one int per row.
void launch_panel_digits(const double* pool, const PanelDesc* panels, const long long* row0, int n_panels, int max_n,
                         int max_k, long long rows, int kp, int* be, void* dig, int* exps, cudaStream_t st);
// Digits of G gathered per task: rows rbase .. rbase + R of g to rows g_row0..
void launch_gather_digits(const EmuOp& g, int rbase, int R, const PanelTask64* tasks, int n_tasks, const int* lam,
                          long long out_rows, int kp, void* out, cudaStream_t st);
// Steps A (mode 0, X) and B (mode 1, Y): rows r0 .. r0 + R of G, output as
// k_panel_gemm's (k_simt.cu).
struct Panel64Args {
  const int4* tiles;  // (task, A tile of 128 rows, B tile of 128, 0)
  int n_tiles, mode, R, r0, P0b;
  const PanelTask64* tasks;
  long long ldk;
  const long long* rowbase;
  const int* rowmul;
  const void* panel_dig;
  const int* panel_exps;
  long long panel_rows;
  int kp;
  const void* g_dig;
  const int* g_exps;
  long long g_rows;
  int g_kp;
  double* out;
  const double *pool, *G;
  const int* lam;
  int nao;
};
int launch_panel64(const Panel64Args& p, int* err_flag, cudaStream_t st);
// Step C over work units (k_tc.h, launch_plan_units) of 128 x 128 tiles, operands
// with an exponent per sigma-atom (`per` slabs).  Scratch per (X row, RI
// function): part 16 bytes of partial sums, pair 4 of their exponent.
struct Chi64Args {
  UnitScratch units;
  const int *tasks, *counts;
  int nslab, nqt, P0, prow, nri, per;
  const long long* slab_k0;
  const int* slab_len;
  double* chi;
  void* part;
  int* pair;
};
int launch_chi64(const EmuOp& x, const EmuOp& y, const Chi64Args& c, int* err_flag, cudaStream_t st);

// The same on the work buffers of a context (gw_fp64.cu).  Between emu_begin
// and emu_end of one call; names tell apart operands in use together.
int emu_begin(gw_ctx* ctx, cudaStream_t st);
int emu_flag(gw_ctx* ctx, int** err);  // the error flag of the launchers
int emu_prep(gw_ctx* ctx, const char* name, const EmuSrc& s, EmuOp* op, cudaStream_t st);
int emu_prep_segments(gw_ctx* ctx, const char* name, const EmuSrc& s, const long long* seg, int n_seg, int max_len,
                      EmuOp* op, cudaStream_t st);
int emu_mm(gw_ctx* ctx, const EmuOp& A, const EmuOp& B, const EmuGemm& g, cudaStream_t st);
// Product of two matrices.  Operands beyond 4 GB of digits, or whose digits do
// not fit the device, go in row chunks; one matrix on both sides has one set of
// digits.  keep (may be null): on a later call with the same A, its digits are
// reused where they are whole (keep->dig set by the first call).
int emu_product(gw_ctx* ctx, const EmuSrc& A, const EmuSrc& B, const EmuGemm& g, EmuOp* keep,
                cudaStream_t st);
// G^occ(tau), G^virt(tau) of Eq. 2 from the orbitals of mol (ctx: the context
// whose work buffers serve, often the same); cso, csv: scratch for the scaled
// orbitals (n_AO x n_occ, n_AO x n_virt).
int greens_fp64(gw_ctx* ctx, const gw_ctx& mol, double tau, double* cso, double* csv, double* g_occ, double* g_virt, cudaStream_t st);
// Reads the error flag after the stream has been synchronised.
int emu_end(gw_ctx* ctx, const char* call);

}  // namespace gw
