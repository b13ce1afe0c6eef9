// Interface of the single-launch tensor-core SP2 main phase (sp2_run.cu).
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
  unsigned* bar;        // grid barrier counter, zero
};
// Launches it on `s` and sets *ran, or leaves *ran 0 where the launched form is to be
// used: other precisions, the CTA-pair form, a large captured call.
int sp2_run(tb_ctx* ctx, int precision, const Sp2RunArgs& g, int captured, int* ran, cudaStream_t s);
