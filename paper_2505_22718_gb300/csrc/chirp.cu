// Chirp transforms of the contraction (chirp.cuh): when they apply, their tables, and how the rows
// are split over CTAs.
#include <algorithm>
#include <cmath>

#include "swcl_internal.h"

namespace swcl {

// ln k_q = x0 + q d to rounding: the line through the end points (their logarithms in extended
// precision), with no point further off than 4 eps max(4, |ln k|), eight times the largest rounding error of
// ln k itself.  A grid as geomspace, logspace or an exponential of a linspace give it, whose points carry the
// roundings of an exponent and of a power, lies within 1.4 of those 4 (ranges from 1e-12 to 1e6, 150 to
// 1024 points); the phases e^{-i eta_n ln k_q} of the line differ from those of such a grid about as much as
// rounding ln k changes them, and by a few times that at the bound: at most 5e-12 at N = 2048, where the results
// are held to 1e-10.  A grid rounded to seven digits, or perturbed by 1e-12, does not pass
// (tests/test_gpu_chirp.py).
void chirp_fit_grid(swcl_ctx* c) {
  c->ck_uniform = false;
  c->ck_off = false;
  for (auto& p : c->ck)
    for (auto& d : p) d.ready = false;
  const int n = c->N_k;
  if (n < 3) return;
  const long double x0 = logl((long double)c->k_h[0]);
  const long double d = (logl((long double)c->k_h[n - 1]) - x0) / (n - 1);
  const double x0d = (double)x0, dd = (double)d;
  const double tol = 4.0 * 2.220446e-16 * std::max({4.0, std::fabs(std::log(c->k_h[0])),
                                                   std::fabs(std::log(c->k_h[n - 1]))});
  for (int q = 0; q < n; ++q)
    if (std::fabs(std::log(c->k_h[q]) - std::fma(dd, (double)q, x0d)) > tol) return;
  const long double cc = d / (2.0L * (long double)c->L), xx = x0 / (long double)c->L;
  c->ck_c[0] = (double)cc;
  c->ck_c[1] = (double)(cc - (long double)c->ck_c[0]);
  c->ck_x[0] = (double)xx;
  c->ck_x[1] = (double)(xx - (long double)c->ck_x[0]);
  c->ck_uniform = true;
}

namespace {

// smallest M = 2^m, m = 9..13, that holds the linear convolution; 0 = none
int log_size(int n_in, int n_out) {
  for (int m = 9; m <= 13; ++m)
    if (n_in + n_out - 1 <= (1 << m)) return m;
  return 0;
}

// First frequency of the forward transform.  FP64: the term n = 0, whose phase is 1, is added beside
// the transform, so that N/2 frequencies remain.  FP32: at least the terms n < 64, which carry most of a
// smooth window's Delta, stay in compensated tensor-core products; the FFT's rounding error, about 2e-7 of what
// passes through it, then falls on the small rest.  Rows with a larger rest keep more (k_head), and zeros
// take their places in the transform.  Simulated C error against the FP64 oracle at N5K shape
// (the GEMM over all frequencies 2.1e-5): 2.4e-5 with 32 terms in the products, 1.8e-5 with 64, 2.1e-5
// with 128; 1.4e-4 with none.
int first_freq(int precision) { return precision == SWCL_FP64 ? 1 : kChirpHead; }
int form(int precision) { return precision == SWCL_FP64 ? 0 : 1; }

// multipoles that one CTA of the FP32 transpose sums in FP32 at most (the CTAs' sums in FP64); the
// GEMM's epilogue sums 48 columns or more
constexpr int kMaxSum32 = 16;

}  // namespace

// Transforms per (walker, tracer, multipole): the profile rows of basis mode, or up to four knots.
int chirp_rank(const swcl_ctx* c) { return c->lr_basis ? c->lr_true_rank : c->N_I <= 4 ? c->N_I : 0; }

bool chirp_use(const swcl_ctx* c, int precision) {
  if (!c->ck_uniform || (c->ck_off && precision == SWCL_FP64)) return false;
  const int r = chirp_rank(c), mf = log_size(c->n_h - first_freq(precision), c->N_k), ma = log_size(c->N_k, c->n_h);
  if (r <= 0 || !mf || !ma) return false;
  // FP64 operations: about 75 per point and pair of FFTs, against 2 per (frequency, k point) of the
  // direct sum (four profile rows cost four transforms but one direct sum).  Both sides are bound by
  // the FP64 pipe: forward + VJP at N = 2048, N_k = 1024, 103 multipoles, 15 tracers 0.95 ms against
  // 12.8 ms; N = N_k = 256, 20 multipoles, 2 tracers (three quarters of the line) 0.24 against 0.79 ms.
  // Just inside the line the transforms are the faster side by far (20 multipoles, N_k = 152, one row: 0.11 against
  // 0.65 ms at N = 256, 0.13 against 4.5 ms at N = 2048; N = 8192, N_k = 80 0.56 against 17.7 ms), since the direct
  // sums also run on too few CTAs there.  The line is where the operations are equal, not where the times are.
  if (precision == SWCL_FP64) return 75.0 * r * (double)(1 << std::max(mf, ma)) < 2.0 * c->n_h * (double)c->N_k;
  // the mixed form: beside the basis-mode GEMMs, unless tiles or products of theirs are asked for
  if (precision != SWCL_SPLIT_BF16 || !c->lr_basis || c->bt_disabled || c->bt_asked) return false;
  // From N = 1024 on: 15 tracers, 103 multipoles, N = 2048, N_k = 1024 forward + VJP 59 us a step
  // against 136 us with the GEMMs over all frequencies, 256 such points with ragged lists 7.5 against
  // 25.1 ms, N = N_k = 4096 with 30 tracers and 2999 multipoles 11.6 against 32.2 ms; at N = 512,
  // N_k = 333, 7 tracers, 37 multipoles, three points both take 62 us.  Few k points do not move the line: 64 of
  // them, 7 tracers, 103 multipoles, one and 16 points 70 and 159 us against 82 and 205 us at N = 1024, 90 and 423
  // against 142 and 564 us at N = 4096, 256 and 902 against 365 and 1025 us at N = 8192.  The GEMMs win, forward
  // alone, where all rows keep 256 frequencies (k_head) and those are half of them: N = 1024 with sigma_z = 0.02
  // above z = 0.6, finer than that grid resolves, 78 against 64 us, and equal at N = 2048.
  return c->N >= 1024;
}

// FP64 only: the direct sums need no tables.  (The mixed form has nothing to gain from giving its
// transforms up: the images of the GEMMs over all frequencies take several times as much memory.)
int chirp_drop(swcl_ctx* c) {
  if (c->capturing) return fail(c, SWCL_ERR_STATE, "chirp tables given up during capture");
  for (auto& d : c->ck[form(SWCL_FP64)]) {
    release(c, d.tab);
    d.ready = false;
  }
  release(c, c->ws_ckpart);
  c->ck_off = true;
  return SWCL_OK;
}

int chirp_prepare(swcl_ctx* c, int precision) {
  if (!chirp_use(c, precision)) return SWCL_OK;
  for (int dir = 0; dir < 2; ++dir) {
    ChirpDir& d = c->ck[form(precision)][dir];
    if (d.ready) continue;
    if (c->capturing) return fail(c, SWCL_ERR_STATE, "chirp tables built during capture");
    d.n0 = dir == 0 ? first_freq(precision) : 0;
    const int n_freq = c->n_h - d.n0;
    d.logm = dir == 0 ? log_size(n_freq, c->N_k) : log_size(c->N_k, n_freq);
    const int M = 1 << d.logm;
    d.half = c->N_k <= M / 2 && n_freq <= M / 2 + (dir == 0 ? 0 : 1);
    const bool fp64 = precision == SWCL_FP64;
    const int st = ensure(c, d.tab, fp64 ? chirp64_table_bytes(d.logm, n_freq, c->N_k)
                                         : chirp32_table_bytes(d.logm, n_freq, c->N_k));
    if (st == SWCL_ERR_OOM_BUDGET && fp64) {
      c->err.clear();
      return chirp_drop(c);
    }
    if (st) return st;
    const int t_lo = dir == 0 ? n_freq - 1 : c->N_k - 1, t_hi = dir == 0 ? c->N_k - 1 : n_freq - 1;
    const cudaError_t e =
        fp64 ? chirp64_build(d.tab.p, d.logm, d.n0, n_freq, c->N_k, t_lo, t_hi, c->ck_c, c->ck_x, c->stream)
             : chirp32_build(d.tab.p, d.logm, d.n0, n_freq, c->N_k, t_lo, t_hi, c->ck_c, c->ck_x, dir == 0, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "chirp tables");
    d.ready = true;
  }
  return SWCL_OK;
}

// CTAs per row; each takes an equal share of the row's multipoles.  FP64, bound by one pipe of the SM
// whatever the number of resident CTAs: enough CTAs for eight turns of what the GPU holds at once, so
// that the last turn is a small part.  FP32, which lives from several resident CTAs: the share of at
// most 16 multipoles with the fewest turns x (multipoles + the load of the row's own data, about 0.4 of
// a multipole); 1545 rows of 2048 points take 22.9 us with one multipole per CTA, 20.9 with three (the
// choice), 26.8 with seven; the sum over the transpose's CTAs 22.6, 12.1 and 8.7 us.
static int row_chunks(const swcl_ctx* c, int precision, long rows, int n_l, int logm) {
  if (precision == SWCL_FP64) {
    const long slots = (long)c->num_sms * chirp64_ctas_per_sm(logm);
    const long per = std::max<long>(1, rows * n_l / (8 * slots));
    return (int)std::min<long>(n_l, (n_l + per - 1) / per);
  }
  const long slots = (long)c->num_sms * chirp32_ctas_per_sm(logm);
  int best = 1;
  double best_cost = 0.0;
  for (int per = 1; per <= std::min(n_l, kMaxSum32); ++per) {
    const long ctas = rows * ((n_l + per - 1) / per);
    const double cost = (double)((ctas + slots - 1) / slots) * (per + 0.4);
    if (per == 1 || cost < best_cost) {
      best = per;
      best_cost = cost;
    }
  }
  return (n_l + best - 1) / best;
}

// Bytes of the adjoint's partial sums over n_l multipoles (whole: with every CTA of a row its own)
size_t chirp_part_bytes(const swcl_ctx* c, int precision, int n_l, bool whole) {
  if (!chirp_use(c, precision)) return 0;
  const long rows = (long)c->n_walk * c->N_tr;
  const int n = whole ? row_chunks(c, precision, rows, n_l, log_size(c->N_k, c->n_h)) : 1;
  return (precision == SWCL_FP64 ? 16 : 8) * (size_t)rows * chirp_rank(c) * c->n_h * n;
}

// the multipoles of one launch: all of [l_lo, l_lo + n_l), or each walker's list where the basis-mode
// GEMMs keep listed multipoles only (Delta's other rows hold zeros)
static ChirpRun run_for(const swcl_ctx* c, int precision, bool adjoint, int l_lo, int n_l) {
  const Stencil sv = stencil(c);
  const bool lists = precision != SWCL_FP64 && c->bt_compact;
  const int n = row_chunks(c, precision, (long)c->n_walk * c->N_tr, n_l, c->ck[form(precision)][adjoint].logm);
  return ChirpRun{c->n_walk, c->N_tr, sv.NI, c->n_h, c->N_k, c->N_ell, l_lo, n_l, chirp_rank(c), n, n, 0,
                  lists ? (const int*)c->d_off.p : nullptr, lists ? (const int*)c->d_idx.p : nullptr};
}

int chirp_forward(swcl_ctx* c, int precision, int l_lo, int n_l) {
  const ChirpDir& d = c->ck[form(precision)][0];
  const Stencil sv = stencil(c);
  const ChirpRun r = run_for(c, precision, false, l_lo, n_l);
  ++c->last_launches;
  prof_begin(c);
  const cudaError_t e =
      precision == SWCL_FP64
          ? chirp64_forward(d, (double*)c->ws_delta.p, (const cplx*)c->ws_coef.p, (const cplx*)c->d_gtab.p,
                            (const int*)c->d_cls_of.p, sv.w, sv.w_ts, (const double*)c->d_kpow.p, r, c->stream)
          : chirp32_forward(d, (float*)c->ws_delta.p, (const float4*)c->ws_coef.p, (const float2*)c->bt_g32.p,
                            (const int*)c->d_cls_of.p, (const float*)c->bt_kmu.p, (const int*)c->ck_head.p, r, c->stream);
  prof_end(c, precision == SWCL_FP64 ? "chirp fwd fp64" : "chirp fwd f32");
  return e == cudaSuccess ? SWCL_OK : cuda_fail(c, e, "chirp transform, forward");
}

int chirp_adjoint(swcl_ctx* c, int precision, int l_lo, int n_l, bool accumulate) {
  const bool fp64 = precision == SWCL_FP64;
  const ChirpDir& d = c->ck[form(precision)][1];
  const Stencil sv = stencil(c);
  ChirpRun r = run_for(c, precision, true, l_lo, n_l);
  // Partial sums of the CTAs of a row: those of all the shares of its multipoles, or as many as the budget
  // has room for.  FP64: then so many larger shares.  FP32, where a share is bounded (kMaxSum32): the
  // shares in turn, group by group, each group added to the sums of those before in FP64.
  const size_t per = chirp_part_bytes(c, precision, n_l, false);
  int fit = r.n_total;
  if (c->budget) {
    const size_t others = c->held - c->ws_ckpart.bytes;
    fit = (int)std::min<size_t>(fit, others < c->budget ? (c->budget - others) / per : 0);
  }
  if (c->capturing) fit = (int)std::min<size_t>(fit, c->ws_ckpart.bytes / per);
  fit = std::max(fit, 1);
  const int st = ensure(c, c->ws_ckpart, per * fit);
  if (st) return st;
  if (fp64) r.n_total = fit;
  for (r.chunk0 = 0; r.chunk0 < r.n_total; r.chunk0 += fit) {
    r.n_chunk = std::min(fit, r.n_total - r.chunk0);
    ++c->last_launches;
    prof_begin(c);
    cudaError_t e =
        fp64 ? chirp64_adjoint(d, c->ws_ckpart.p, (const double*)c->ws_dbar.p, (const cplx*)c->d_gtab.p,
                               (const int*)c->d_cls_of.p, sv.w, sv.w_ts, (const double*)c->d_kpow.p, r, c->stream)
             : chirp32_adjoint(d, c->ws_ckpart.p, (const float*)c->ws_dbar.p, (const float2*)c->bt_g32.p,
                               (const int*)c->d_cls_of.p, (const float*)c->bt_kmu.p, r, c->stream);
    prof_end(c, fp64 ? "chirp adj fp64" : "chirp adj f32");
    if (e != cudaSuccess) return cuda_fail(c, e, "chirp transform, transposed");
    ++c->last_launches;
    prof_begin(c);
    const bool add = accumulate || r.chunk0 > 0;
    e = fp64 ? chirp64_sum((cplx*)c->ws_cbar.p, c->ws_ckpart.p, d, r, add, c->stream)
             : chirp32_sum((cplx*)c->ws_cbar.p, c->ws_ckpart.p, d, r, add, c->stream);
    prof_end(c, "chirp adj sum");
    if (e != cudaSuccess) return cuda_fail(c, e, "chirp transform, sum over multipoles");
  }
  return SWCL_OK;
}

}  // namespace swcl
