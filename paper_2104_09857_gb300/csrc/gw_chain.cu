// C ABI of the screening chain: chi(i tau) -> chi(i omega) -> eps(i omega)
// (Eq. 7, with V = L L^T, Eq. 8) -> W^c(i omega) (Eq. 9) -> W^c(i tau).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "gw_internal.h"
#include "k_chain.h"
#include "k_emu.h"

namespace {

struct DevBuf {
  void* p = nullptr;
  ~DevBuf() {
    if (p) cudaFree(p);
  }
};

#define CH_TRY(call)                                                              \
  do {                                                                            \
    cudaError_t e_ = (call);                                                      \
    if (e_ != cudaSuccess) {                                                      \
      ctx->err = std::string("chain: ") + #call + ": " + cudaGetErrorString(e_);      \
      return e_ == cudaErrorMemoryAllocation ? GW_ERR_OOM : GW_ERR_CUDA;          \
    }                                                                             \
  } while (0)

// count doubles (or as many bytes of another type) of a named work buffer
template <typename T>
int chain_buffer(gw_ctx* ctx, const char* name, size_t count, T** out) {
  void* p = nullptr;
  const int rc = gw::work_buffer(ctx, name, count * 8, &p);
  *out = static_cast<T*>(p);
  return rc;
}

// gw_chi_to_w with the frequencies factored together in groups of up to `group`
// bytes of [eps; L] (at least one).
int chi_to_w(gw_ctx* ctx, const double* V, int n_omega, const double* gamma, const double* delta,
             const double* chi_tau, int chi_on_device, double* w_tau_out, int out_on_device, size_t group) {
  ctx->err.clear();
  if (ctx->n_at == 0 || !ctx->have_greens) {
    ctx->err = "gw_chi_to_w: call gw_set_basis and gw_set_greens first (the tau grid)";
    return GW_ERR_ORDER;
  }
  const int n = ctx->nri;
  const int n_tau = (int)ctx->tau.size();
  if (!V || !gamma || !delta || !chi_tau || !w_tau_out || n_omega <= 0 || n_omega > 4096) {
    ctx->err = "gw_chi_to_w: bad arguments";
    return GW_ERR_INVALID_ARG;
  }
  for (long long i = 0; i < (long long)n_omega * n_tau; ++i)
    if (!std::isfinite(gamma[i]) || !std::isfinite(delta[i])) {
      ctx->err = "gw_chi_to_w: non-finite transform weight";
      return GW_ERR_NONFINITE;
    }
  for (long long i = 0; i < (long long)n * n; ++i)
    if (!std::isfinite(V[i])) {
      ctx->err = "gw_chi_to_w: non-finite Coulomb matrix element";
      return GW_ERR_NONFINITE;
    }
  CH_TRY(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  gw::WorkTrim trim{ctx};
  const size_t nn = (size_t)n * n;
  DevBuf b_chi, b_w;
  // V, its factor L, [eps; L] of nb frequencies and one product share the
  // context's work buffers.  nb frequencies are factored together: all of
  // them within 1 GB (the sweep's chain of small kernels is then paid once),
  // one at a time for large matrices, whose sweeps fill the chip by themselves.
  const int nb = (int)std::max<size_t>(1, std::min<size_t>((size_t)n_omega, group / (2 * nn * 8)));
  double *v, *low, *m, *t, *ww, *g, *d;
  int* err;
  int rc;
  if ((rc = chain_buffer(ctx, "w.v", nn, &v)) || (rc = chain_buffer(ctx, "w.low", nn, &low)) ||
      (rc = chain_buffer(ctx, "w.eps_l", 2 * nn * nb, &m)) || (rc = chain_buffer(ctx, "w.t", nn, &t)) ||
      (rc = chain_buffer(ctx, "w.ww", nn, &ww)) ||
      (rc = chain_buffer(ctx, "w.gamma", (size_t)n_omega * n_tau, &g)) ||
      (rc = chain_buffer(ctx, "w.delta", (size_t)n_omega * n_tau, &d)) ||
      (rc = chain_buffer(ctx, "w.not_spd", 1, &err)) || (rc = gw::emu_begin(ctx, st)))
    return rc;
  const double* chi;
  if (chi_on_device) {
    chi = chi_tau;
  } else {
    CH_TRY(gw::device_alloc(ctx, &b_chi.p, (size_t)n_tau * nn * 8));
    CH_TRY(cudaMemcpyAsync(b_chi.p, chi_tau, (size_t)n_tau * nn * 8, cudaMemcpyHostToDevice, st));
    chi = (const double*)b_chi.p;
  }
  double* wout;
  if (out_on_device) {
    wout = w_tau_out;
  } else {
    CH_TRY(gw::device_alloc(ctx, &b_w.p, (size_t)n_tau * nn * 8));
    wout = (double*)b_w.p;
  }
  CH_TRY(cudaMemsetAsync(wout, 0, (size_t)n_tau * nn * 8, st));
  CH_TRY(cudaMemsetAsync(err, 0, sizeof(int), st));
  CH_TRY(cudaMemcpyAsync(v, V, nn * 8, cudaMemcpyHostToDevice, st));
  CH_TRY(cudaMemcpyAsync(g, gamma, (size_t)n_omega * n_tau * 8, cudaMemcpyHostToDevice, st));
  CH_TRY(cudaMemcpyAsync(d, delta, (size_t)n_omega * n_tau * 8, cudaMemcpyHostToDevice, st));
  // V = L L^T (Eq. 8)
  CH_TRY(cudaMemcpyAsync(low, v, nn * 8, cudaMemcpyDeviceToDevice, st));
  if ((rc = gw::chain_cholesky(ctx, low, n, n, 1, 0, err, st))) return rc;
  int h_err = 0;
  CH_TRY(cudaMemcpyAsync(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CH_TRY(cudaStreamSynchronize(st));
  if (h_err) {
    ctx->err = "gw_chi_to_w: the Coulomb matrix is not positive definite";
    return GW_ERR_NOT_SPD;
  }
  gw::EmuSrc s_lt, s_row;  // L^T, and a matrix by its rows
  s_lt.src = low;
  s_lt.ld = s_row.ld = n;
  s_lt.rows = s_row.rows = n;
  s_lt.K = s_row.K = n;
  s_lt.trans = true;
  gw::EmuOp lt;  // digits of L^T, made once
  for (int k0 = 0; k0 < n_omega; k0 += nb) {
    const int nk = std::min(nb, n_omega - k0);
    for (int k = k0; k < k0 + nk; ++k) {
      double* mk = m + (size_t)(k - k0) * 2 * nn;
      // chi(i omega_k) = sum_j gamma_kj chi(i tau_j)
      gw::chain_lincomb(chi, n_tau, g + (size_t)k * n_tau, (long long)nn, t, st);
      // (chi L)^T = L^T chi^T by rows, then eps = 1 - L^T (chi L)  (Eq. 7), its
      // lower triangle; row r of L^T starts at column r
      gw::EmuGemm p;
      p.C = ww;
      p.ldc = n;
      p.ktri = 1;
      s_row.src = t;
      if ((rc = gw::emu_product(ctx, s_lt, s_row, p, &lt, st))) return rc;
      p.alpha = -1.0;
      p.C = mk;
      p.tri = 1;
      s_row.src = ww;
      if ((rc = gw::emu_product(ctx, s_lt, s_row, p, &lt, st))) return rc;
      gw::chain_add_diagonal(mk, n, 1.0, st);
      CH_TRY(cudaMemcpyAsync(mk + nn, low, nn * 8, cudaMemcpyDeviceToDevice, st));
    }
    // eps = R R^T with L below it: its rows become L R^-T = Z, and
    // W^c = Z Z^T - V  (Eq. 9), lower triangle
    if ((rc = gw::chain_cholesky(ctx, m, 2LL * n, n, nk, 2LL * nn, err, st))) return rc;
    for (int k = k0; k < k0 + nk; ++k) {
      gw::EmuGemm q;
      q.C = ww;
      q.ldc = n;
      q.tri = 1;
      s_row.src = m + (size_t)(k - k0) * 2 * nn + nn;
      if ((rc = gw::emu_product(ctx, s_row, s_row, q, nullptr, st))) return rc;
      // W^c(i tau_j) += delta_jk W^c(i omega_k)
      gw::chain_add_symmetric(ww, v, d + k, n_omega, n_tau, n, wout, st);
      CH_TRY(cudaGetLastError());
    }
  }
  CH_TRY(cudaMemcpyAsync(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  if (!out_on_device)
    CH_TRY(cudaMemcpyAsync(w_tau_out, wout, (size_t)n_tau * nn * 8, cudaMemcpyDeviceToHost, st));
  CH_TRY(cudaStreamSynchronize(st));
  if ((rc = gw::emu_end(ctx, "gw_chi_to_w"))) return rc;
  if (h_err) {
    ctx->err = "gw_chi_to_w: eps(i omega) is not positive definite (chi must be negative semidefinite)";
    return GW_ERR_NOT_SPD;
  }
  return GW_OK;
}
}  // namespace

extern "C" int gw_chi_to_w(gw_ctx* ctx, const double* V, int n_omega, const double* gamma,
                           const double* delta, const double* chi_tau, int chi_on_device,
                           double* w_tau_out, int out_on_device) {
  if (!ctx) return GW_ERR_INVALID_ARG;
  gw::TraceRange trace("gw_chi_to_w");
  const auto call = [&](size_t group) {
    return chi_to_w(ctx, V, n_omega, gamma, delta, chi_tau, chi_on_device, w_tau_out, out_on_device, group);
  };
  int rc = call(ctx->test_digit_bytes > 0.0 ? (size_t)ctx->test_digit_bytes : size_t(1) << 30);
  if (gw::memory_short(ctx, rc)) {
    // once more, one frequency at a time
    gw::work_trim(ctx, "w.", 0);
    rc = call(0);
  }
  return rc;
}

// S^-1 M S^-1 for n_mat symmetric matrices M (chi~ of Eq. 5, W~ of Eq. 10,
// V~ of Eq. 11), FP64: S = R R^T (blocked Cholesky), R^-1 by a triangular
// solve on the identity, S^-1 = R^-T R^-1, then two products per matrix.
extern "C" int gw_ri_metric(gw_ctx* ctx, const double* S, int n_mat, const double* M, int m_on_device,
                            double* out, int out_on_device) {
  if (!ctx) return GW_ERR_INVALID_ARG;
  gw::TraceRange trace("gw_ri_metric");
  ctx->err.clear();
  if (ctx->n_at == 0) {
    ctx->err = "gw_ri_metric: call gw_set_basis first (the RI size)";
    return GW_ERR_ORDER;
  }
  if (!S || !M || !out || n_mat <= 0) {
    ctx->err = "gw_ri_metric: bad arguments";
    return GW_ERR_INVALID_ARG;
  }
  const int n = ctx->nri;
  const size_t nn = (size_t)n * n;
  for (size_t i = 0; i < nn; ++i)
    if (!std::isfinite(S[i])) {
      ctx->err = "gw_ri_metric: non-finite metric element";
      return GW_ERR_NONFINITE;
    }
  CH_TRY(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  gw::WorkTrim trim{ctx};
  DevBuf b_m, b_o;
  double *r, *si, *t;
  int* err;
  int rc;
  if ((rc = chain_buffer(ctx, "w.eps_l", 2 * nn, &r)) || (rc = chain_buffer(ctx, "w.low", nn, &si)) ||
      (rc = chain_buffer(ctx, "w.t", nn, &t)) || (rc = chain_buffer(ctx, "w.not_spd", 1, &err)) ||
      (rc = gw::emu_begin(ctx, st)))
    return rc;
  const double* m = M;
  if (!m_on_device) {
    CH_TRY(gw::device_alloc(ctx, &b_m.p, (size_t)n_mat * nn * 8));
    CH_TRY(cudaMemcpyAsync(b_m.p, M, (size_t)n_mat * nn * 8, cudaMemcpyHostToDevice, st));
    m = (const double*)b_m.p;
  }
  double* o = out;
  if (!out_on_device) {
    CH_TRY(gw::device_alloc(ctx, &b_o.p, (size_t)n_mat * nn * 8));
    o = (double*)b_o.p;
  }
  CH_TRY(cudaMemsetAsync(err, 0, sizeof(int), st));
  CH_TRY(cudaMemcpyAsync(r, S, nn * 8, cudaMemcpyHostToDevice, st));
  // [S; 1] -> [R; R^-T]
  gw::chain_set_identity(r + nn, n, st);
  if ((rc = gw::chain_cholesky(ctx, r, 2LL * n, n, 1, 0, err, st))) return rc;
  int h_err = 0;
  CH_TRY(cudaMemcpyAsync(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CH_TRY(cudaStreamSynchronize(st));
  if (h_err) {
    ctx->err = "gw_ri_metric: the metric is not positive definite";
    return GW_ERR_NOT_SPD;
  }
  gw::EmuSrc s_q, s_si, s_m;
  s_q.src = r + nn;
  s_q.ld = s_si.ld = s_m.ld = n;
  s_q.rows = s_si.rows = s_m.rows = n;
  s_q.K = s_si.K = s_m.K = n;
  s_si.src = si;
  // S^-1 = R^-T R^-1; row r of R^-T starts at column r
  gw::EmuGemm p;
  p.C = si;
  p.ldc = n;
  p.ktri = 1;
  if ((rc = gw::emu_product(ctx, s_q, s_q, p, nullptr, st))) return rc;
  gw::EmuOp keep;
  for (int k = 0; k < n_mat; ++k) {
    // t = S^-1 M, then t S^-1 (S^-1 symmetric: its rows are its columns)
    gw::EmuGemm q;
    q.C = t;
    q.ldc = n;
    s_m.src = m + (size_t)k * nn;
    s_m.trans = true;  // columns of M
    if ((rc = gw::emu_product(ctx, s_si, s_m, q, &keep, st))) return rc;
    q.C = o + (size_t)k * nn;
    gw::EmuSrc s_t = s_si;
    s_t.src = t;
    if ((rc = gw::emu_product(ctx, s_t, s_si, q, nullptr, st))) return rc;
  }
  CH_TRY(cudaGetLastError());
  if (!out_on_device)
    CH_TRY(cudaMemcpyAsync(out, o, (size_t)n_mat * nn * 8, cudaMemcpyDeviceToHost, st));
  CH_TRY(cudaStreamSynchronize(st));
  return gw::emu_end(ctx, "gw_ri_metric");
}
