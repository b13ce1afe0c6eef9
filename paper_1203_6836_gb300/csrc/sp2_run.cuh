// Interface of the single-launch SP2 forms: the tensor-core main phase (sp2_run.cu) and
// the FP64 path of small matrices (sp2_run64.cu).
#pragma once

#include "common.cuh"

struct Sp2RunArgs {
  SP2StepArgs a;        // n, ld, nocc, tol, floor, rule, max_iter, st, wait_ns
  const double* H;
  const double* bparts; // Gershgorin partials of k_bounds
  int nbparts;
  float* M[2];          // the iterate's FP32 master and operands, alternating
  void* hi[2];
  void* lo[2];
  double* parts[2];     // (Tr X, ||X||_F^2) of each 128 x 32 chunk of the upper triangle
  unsigned *bar, *bar_tr;  // grid barrier counters (operands stored, traces summed), zero
};
// Launches it on `s` and sets *ran, or leaves *ran 0 where the launched form is to be
// used: other precisions, the CTA-pair form, a large captured call.
int sp2_run(tb_ctx* ctx, int precision, const Sp2RunArgs& g, int captured, int* ran, cudaStream_t s);

constexpr int kSp2Run64Max = 512;
struct Sp2Run64Args {
  SP2StepArgs a;        // n, ld, nocc, tol, rule, max_iter, st
  const double* H;
  const double* bparts; // Gershgorin partials of k_bounds
  int nbparts;
  double* F[2];         // the iterate, alternating, ld x ld
  double* parts[2];     // (Tr X, ||X||_F^2) of each unit
  unsigned* bar;        // grid barrier counter, zero
  double* D;
  tb_sp2_report* rep;   // device or NULL
};
// n <= kSp2Run64Max: the whole FP64 path on `s`.
int sp2_run64(tb_ctx* ctx, const Sp2Run64Args& g, cudaStream_t s);

// The report of a call from its state (one thread); mode 0: FP64 main phase, 1: FP64
// refinement, 2: FP32 master without refinement.
__device__ __forceinline__ void sp2_fill_report(const SP2State* st, int mode, int n, double nocc, tb_sp2_report* rep) {
  double t1, t2;
  if (mode == 1) {
    t1 = st->rt1[st->riters];
    t2 = st->rt2[st->riters];
  } else {
    t1 = st->t1[st->iters];
    t2 = st->t2[st->iters];
  }
  // status: device error; an FP64 phase that hit its cap without reaching
  // |Tr X - Tr X^2| <= 1e-6 max(1, N_occ); a trace that missed N_occ
  // (no gap at the occupation)
  int status = TB_OK;
  const double e = t1 - t2;
  const bool capped = mode == 1 ? st->rcapped : (mode == 0 ? st->capped : 0);
  if (st->err) status = st->err;
  else if (capped && fabs(e) > 1e-6 * fmax(1.0, nocc)) status = TB_ERR_NOT_CONVERGED;
  else if (fabs(t1 - nocc) > 0.25) status = TB_ERR_GAP;
  rep->status = status;
  rep->iters = st->iters;
  rep->refine_iters = mode == 1 ? st->riters : 0;
  rep->n = n;
  rep->eps_min = st->emin;
  rep->eps_max = st->emax;
  rep->trace = t1;
  rep->idem_trace = e;
  rep->idem_fro = mode == 1 && st->riters > 0 ? st->idem_fro : -1.0;
  rep->branch_bits[0] = st->branch[0];
  rep->branch_bits[1] = st->branch[1];
  rep->refine_bits = st->rbranch;
  rep->block_products = 0;
  rep->blocks = 0;
}
