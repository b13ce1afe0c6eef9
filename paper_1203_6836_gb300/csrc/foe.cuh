// Device state of one dm_fermi call and the chemical-potential step, shared by
// the launched expansion (fermi.cu) and the single-launch one (foe_run.cu).
#pragma once

#include "common.cuh"

constexpr int kFoeMaxMu = 40;
constexpr int kFoeMaxM = 40;  // doubling steps issued at most
constexpr int kFoeMats = 7;   // E0, A, Z, T, Y, E1, W
// Canonical shift: the last expansion is accepted and shifted by u = beta dmu
// to second order,
//   D(mu + dmu) = D + u D(I - D) + u^2/2 D(I - D)(I - 2D) + R,
// with D(I - D) = W/4 and D(I - D)(I - 2D) = -E W/2, W = (I - 2E)(I + 2E) (two
// products, W and E W, after every expansion), u the root of the trace condition
// Tr D + u Tr[D(I-D)] + u^2/2 Tr[D(I-D)(I-2D)] = N_occ near -(Tr D - N)/Tr[D(I-D)].
// The remainder involves the third derivative beta^3 f(1-f)(1-6f+6f^2), whose
// last factor is at most 1 in magnitude, so ||R||_F <= |u|^3/6 Tr[D(I - D)]
// (D(I - D) is positive semi-definite with eigenvalues <= 1/4).  The shift
// replaces another expansion when that bound is below kCorrFro sqrt(n) and
// |u| <= kCorrMax.
constexpr double kCorrFro = 1e-7;
constexpr double kCorrMax = 0.1;

struct FoeState {
  double mu, lo, hi;
  double emin, emax;
  int done, iters, capped, err;
  int ran;     // 1: the last chemical-potential step evaluated an expansion (it was not skipped)
  int nocorr;  // 0: apply the canonical shift u to the last expansion
  double dmu;  // u / beta
  double u;
  double c;    // start scale beta / 2^{meff+2}
  int meff;    // doubling steps used
  int skipd[kFoeMaxM];  // 1: doubling step k returns at once (k < m_max - meff, or done)
  double tr[kFoeMaxMu + 1], trdd[kFoeMaxMu + 1], mus[kFoeMaxMu + 1];
  unsigned bar;  // arrivals at the grid barriers of the single-launch form
  unsigned left; // its CTAs that have finished
};

// After an expansion, from Tr E, Tr W and Tr E W: Tr D = n/2 + Tr E,
// Tr D(I - D) = Tr W / 4; then the stop test and the next mu (one thread).  The
// expansion index is the device count st->iters.
__device__ __forceinline__ void foe_mu_step(FoeState* st, double tre, double trw, double trew, int n, double nocc,
                                            double beta, double tol, int max_it) {
  const int it = st->iters;
  const double mu = st->mu;
  const double trd = 0.5 * n + tre;
  const double t1 = 0.25 * trw;    // Tr D(I - D)
  const double t2 = -0.5 * trew;   // Tr D(I - D)(I - 2D)
  st->tr[it] = trd;
  st->trdd[it] = t1;
  st->mus[it] = mu;
  st->iters = it + 1;
  st->ran = 1;
  const double dev = trd - nocc;
  const double step = t1 > 1e-12 ? -dev / (beta * t1) : NAN;  // Newton step on mu
  double u = beta * step;
  for (int k = 0; k < 3 && isfinite(u); ++k) {  // root of dev + t1 u + t2 u^2/2 near the Newton step
    const double g = dev + u * (t1 + 0.5 * t2 * u), gp = t1 + t2 * u;
    if (!(gp > 0.0)) break;
    u -= g / gp;
  }
  const bool shift = isfinite(u) && fabs(u) <= kCorrMax &&
                     fabs(u) * u * u / 6.0 * t1 <= kCorrFro * sqrt((double)max(n, 1));
  if (shift) {
    // accept this expansion with the second-order shift to mu + u / beta
    st->done = 1;
    st->nocorr = 0;
    st->u = u;
    st->dmu = u / beta;
    st->tr[it] = trd + u * (t1 + 0.5 * t2 * u);
    st->mus[it] = mu + u / beta;
  } else if (fabs(dev) <= tol) {
    st->done = 1;
  } else if (it + 1 >= max_it) {
    st->done = 1;
    st->capped = 1;
  } else {
    if (dev < 0.0) st->lo = mu;
    else st->hi = mu;
    st->mu = foe_next_mu(mu, dev, t1, beta, tol, st->lo, st->hi);
  }
}

// E + u W/4 - u^2/4 E W (D(I - D) = W/4, D(I - D)(I - 2D) = -E W/2) of one element.
__device__ __forceinline__ float foe_shifted(float x, float w, float ew, float u) {
  const float h = 0.5f * u * u;
  const float first = 0.25f * w, second = -0.5f * ew;
  return fmaf(h, second, fmaf(u, first, x));
}

__device__ __forceinline__ void foe_report(const FoeState* st, int err, int n, double nocc, double tol,
                                           double* mu_out, tb_fermi_report* rep) {
  const int it = st->iters > 0 ? st->iters - 1 : 0;
  const double mu = st->mus[it];
  if (mu_out) *mu_out = mu;
  if (rep) {
    rep->status = err ? err : (fabs(st->tr[it] - nocc) <= tol ? TB_OK : TB_ERR_NOT_CONVERGED);
    rep->mu_iters = st->iters;
    rep->m = st->meff;
    rep->n = n;
    rep->mu = mu;
    rep->trace = st->tr[it];
    rep->trace_dd = st->trdd[it];
    rep->eps_min = st->emin;
    rep->eps_max = st->emax;
  }
}

// The whole expansion loop in one launch (foe_run.cu).
struct FoeRunArgs {
  const double* H;
  double* D;
  double* mu_out;
  tb_fermi_report* rep;
  FoeState* st;
  float* m[kFoeMats];
  void* hi[kFoeMats];
  void* lo[kFoeMats];
  double *parts, *partsw, *parts3;  // Tr E, Tr W, Tr E W: one slot per 16 diagonal elements
  int n, ld, ns, max_it;
  double nocc, beta, tol;
  unsigned long long wait_ns;
};
// Launches it on `s` and sets *ran, or leaves *ran 0 where the launched form
// is to be used (other precisions, a captured call of more tiles than half the SMs).
int foe_run(tb_ctx* ctx, int precision, const FoeRunArgs& a, int captured, int* ran, cudaStream_t s);
