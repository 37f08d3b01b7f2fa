// FP64 products of a context: operands and workspaces of the digit engine
// (k_emu.cu) on the context's named work buffers.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>

#include "gw_internal.h"
#include "k_emu.h"
#include "k_simt.h"

namespace gw {

namespace {
// digits of one operand held at a time by emu_product
constexpr size_t kMaxDigits = size_t(4) << 30;
}  // namespace

int emu_flag(gw_ctx* ctx, int** err) {
  void* p;
  const int rc = work_buffer(ctx, "w.err", sizeof(int), &p);
  *err = static_cast<int*>(p);
  return rc;
}

int emu_begin(gw_ctx* ctx, cudaStream_t st) {
  int* err;
  int rc;
  if ((rc = emu_flag(ctx, &err))) return rc;
  if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) {
    ctx->err = "FP64 products: clearing the error flag failed";
    return GW_ERR_CUDA;
  }
  return GW_OK;
}

namespace {
// Digits of `rows` rows of length K and n_exps exponents in buffers of this name,
// which go when the call ends (gw::WorkTrim) unless they are chi's ("d64_").
int digit_buffers(gw_ctx* ctx, const char* name, long long rows, int K, long long n_exps, EmuOp* op) {
  void* p;
  int rc;
  const std::string n = std::string(std::strncmp(name, "d64_", 4) ? "w.dig." : "") + name;
  if ((rc = work_buffer(ctx, n.c_str(), std::max<size_t>(emu_dig_bytes(rows, K), 16), &p))) return rc;
  op->dig = p;
  if ((rc = work_buffer(ctx, (n + ".e").c_str(), std::max<size_t>(n_exps, 1) * sizeof(int), &p))) return rc;
  op->exps = static_cast<int*>(p);
  return GW_OK;
}
int prep_launched(gw_ctx* ctx) {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return GW_OK;
  ctx->err = std::string("FP64 operand preparation: ") + cudaGetErrorString(e);
  return GW_ERR_CUDA;
}
}  // namespace

int emu_prep(gw_ctx* ctx, const char* name, const EmuSrc& s, EmuOp* op, cudaStream_t st) {
  const int rc = digit_buffers(ctx, name, s.rows * s.nz, s.K, s.rows * s.nz * 2, op);
  if (rc) return rc;
  launch_emu_prep(*op, s, st);
  return prep_launched(ctx);
}

int emu_prep_segments(gw_ctx* ctx, const char* name, const EmuSrc& s, const long long* seg, int n_seg, int max_len,
                      EmuOp* op, cudaStream_t st) {
  const int rc = digit_buffers(ctx, name, s.rows, s.K, s.rows * n_seg, op);
  if (rc) return rc;
  launch_emu_prep_segments(*op, s, seg, n_seg, max_len, st);
  return prep_launched(ctx);
}

int emu_mm(gw_ctx* ctx, const EmuOp& A, const EmuOp& B, const EmuGemm& g, cudaStream_t st) {
  void* ws = nullptr;
  int* err;
  int rc;
  const size_t bytes = emu_gemm_ws_bytes(A.s.rows, B.s.rows, A.s.K, A.s.nz);
  if (bytes && (rc = work_buffer(ctx, "w.part", bytes, &ws))) return rc;
  if ((rc = emu_flag(ctx, &err))) return rc;
  if (launch_emu_gemm(A, B, g, ws, err, st)) {
    ctx->err = "FP64 product: launch set-up failed";
    return GW_ERR_CUDA;
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    ctx->err = std::string("FP64 product: ") + cudaGetErrorString(e);
    return GW_ERR_CUDA;
  }
  return GW_OK;
}

namespace {
// Rows of s whose digits take up to `most` bytes, in whole tiles and at least one.
long long chunk_rows(const EmuSrc& s, size_t most) {
  return static_cast<long long>(std::max<size_t>(most / emu_dig_bytes(1, s.K) / kEmuTileM, 1)) * kEmuTileM;
}
EmuSrc row_chunk(const EmuSrc& s, long long r0, long long n) {
  EmuSrc p = s;
  p.src = s.src + (s.trans ? r0 : r0 * s.ld);
  p.rows = std::min(n, s.rows - r0);
  return p;
}
// the product with at most `most` bytes of digits of each operand at a time
int product_in_chunks(gw_ctx* ctx, const EmuSrc& A, const EmuSrc& B, const EmuGemm& g, EmuOp* keep, size_t most,
                      cudaStream_t st) {
  const long long ca = chunk_rows(A, most), cb = chunk_rows(B, most);
  const bool square = A.src == B.src && A.ld == B.ld && A.rows == B.rows && A.K == B.K && A.trans == B.trans;
  int rc;
  for (long long r0 = 0; r0 < A.rows; r0 += ca) {
    EmuOp a;
    if (keep && keep->dig && A.rows <= ca) {
      a = *keep;
    } else {
      if ((rc = emu_prep(ctx, keep ? "kept" : "a", row_chunk(A, r0, ca), &a, st))) return rc;
      if (keep && A.rows <= ca) *keep = a;
    }
    for (long long c0 = 0; c0 < B.rows; c0 += cb) {
      EmuOp b = a;
      if (!(square && c0 == r0) && (rc = emu_prep(ctx, "b", row_chunk(B, c0, cb), &b, st))) return rc;
      EmuGemm h = g;
      h.C = g.C + r0 * g.ldc + (g.cblk ? 0 : c0);
      h.col0 = g.col0 + c0;
      // for tri, off the diagonal by both chunks' origins; for ktri by the rows'
      h.tri_off = g.tri_off + r0 - c0;
      if (g.ktri && c0 > 0) h.ktri = 0;
      if ((rc = emu_mm(ctx, a, b, h, st))) return rc;
    }
  }
  return GW_OK;
}
}  // namespace

int emu_product(gw_ctx* ctx, const EmuSrc& A, const EmuSrc& B, const EmuGemm& g, EmuOp* keep, cudaStream_t st) {
  size_t most = ctx->test_digit_bytes > 0.0 ? static_cast<size_t>(ctx->test_digit_bytes) : kMaxDigits;
  for (;;) {
    const int rc = product_in_chunks(ctx, A, B, g, keep, most, st);
    // where the digits do not fit, in half as large chunks (the product does not
    // depend on them); C must not have been added to
    const bool smaller = chunk_rows(A, most) > kEmuTileM || chunk_rows(B, most) > kEmuTileM;
    if (!memory_short(ctx, rc) || g.beta != 0.0 || !smaller) return rc;
    // (only this product's: a caller may hold others, or kept ones of another)
    work_trim(ctx, "w.dig.b", 0);
    work_trim(ctx, keep ? "w.dig.kept" : "w.dig.a", 0);
    if (keep) keep->dig = nullptr;
    ctx->err.clear();
    most = std::min(most, std::max(emu_dig_bytes(A.rows, A.K), emu_dig_bytes(B.rows, B.K))) / 2;
  }
}

// From kGreensDigits primary functions on, the digit products: about 10 us of
// preparation and 30 us per product however small, against (n^3 / 2) / 304
// cycles on the FP64 pipes of all SMs (n = 250: 12 us, 400: 50 us, 602: 175).
constexpr int kGreensDigits = 448;

int greens_fp64(gw_ctx* ctx, const gw_ctx& mol, double tau, double* cso, double* csv, double* g_occ, double* g_virt,
                cudaStream_t st) {
  const int n = mol.nao, occ = mol.n_occ;
  if (n < kGreensDigits || occ == 0 || occ == n) {
    launch_greens(mol.d_C, mol.d_eps, n, occ, mol.mu, tau, cso, csv, g_occ, g_virt, st);
    return GW_OK;
  }
  launch_scale_orbitals(mol.d_C, mol.d_eps, n, occ, mol.mu, tau, cso, csv, st);
  // (where their digits do not fit, on the FP64 pipes after all)
  for (int v = 0; v < 2; ++v) {
    EmuSrc s;
    s.src = v ? csv : cso;
    s.K = v ? n - occ : occ;
    s.ld = s.K;
    s.rows = n;
    EmuOp op;
    int rc = emu_prep(ctx, "orbitals", s, &op, st);
    EmuGemm g;
    g.C = v ? g_virt : g_occ;
    g.ldc = n;
    if (!rc) rc = emu_mm(ctx, op, op, g, st);
    if (memory_short(ctx, rc)) {
      ctx->err.clear();
      launch_greens(mol.d_C, mol.d_eps, n, occ, mol.mu, tau, cso, csv, g_occ, g_virt, st);
      return GW_OK;
    }
    if (rc) return rc;
  }
  return GW_OK;
}

int emu_end(gw_ctx* ctx, const char* call) {
  int* err;
  int rc, h = 0;
  if ((rc = emu_flag(ctx, &err))) return rc;
  if (cudaMemcpy(&h, err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) {
    ctx->err = std::string(call) + ": reading the error flag failed";
    return GW_ERR_CUDA;
  }
  if (h) {
    ctx->err = std::string(call) + ": a bounded wait of the FP64 product kernel gave up";
    return GW_ERR_TIMEOUT;
  }
  return GW_OK;
}

}  // namespace gw
