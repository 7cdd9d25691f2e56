// Interface of the block-expansion applies and the batched MM step (exp_solver.cuh, compiled in
// otlm_exp.cu), used by the FP32 and tensor-core drivers.
#pragma once

#include <cuda_runtime.h>

namespace otlm {

// b = bins per block (a multiple of 8, at least 32), nb = blocks; nb = 0: the grid does not qualify (not
// sorted, too coarse or too long) and runs elsewhere.  q: centres are multiples of q (a power of two at
// least 2^-18 of the largest |xt|), so that differences of centres are exact.
struct ExPlan {
  int b, nb;
  float q;
};

enum { EXA_SOURCE = 0, EXA_TARGET = 1 };
constexpr int EXA_MAX_N = 40960;   // 160 KiB of shared memory for the row beside the scratch

struct ExArgs {
  const int* active;
  const int* n_active;
  const ExPlan* plan;
  const float* xt;
  int n, k, it, max_iter, check, datafit;
  int early;                // launch applies that split a problem over CTAs early, too
  const float* y;
  float *G2, *LA2, *LB2, *S, *mass;
  // stopping decision
  float tol, dw_tol;
  float *err, *dw;
  const float *W, *Wprev;   // tensor-core handles: the weight change is formed here (else dw is given)
  int *done, *iters, *status;
  float* part;              // [P][n] row p holds the problem's partial violations (parts <= n)
  int* count;               // [P] CTAs of the problem that have finished (left at 0)
  // datafit (Table 1)
  float kl_coef, tv_bound, lam_over_eps, log_lam_over_eps;
  // TF32 operand of D^T r by slot
  float *Rhi, *Rlo;
  int ld;
};

struct MMBArgs {
  const int* active;
  const int* n_active;
  int n, k;
  const float *D, *Dt, *xcol, *LA2;
  float *S, *W, *mass, *dw;
  const int* done;
  int penalty, mm_steps;
  float eps, alpha, beta;
};

// Launches (the first error of the launch): the block plan of a grid on the device, one apply over
// the active problems (tc: the tensor-core handle's variant), the log ratios of a later MM step, and
// the batched MM and source step.  with_plan, without (may be null): the numbers of active problems of
// the expansion kernels and of the log-domain kernels, batch and 0 or 0 and batch by the plan.
cudaError_t ex_plan(const float* xt, int n, ExPlan* plan, int batch, int* with_plan, int* without, cudaStream_t stream);
cudaError_t ex_apply_source(const ExArgs& a, int batch, bool tc, int sms, cudaStream_t stream);
cudaError_t ex_apply_target(const ExArgs& a, int batch, bool tc, int sms, cudaStream_t stream);
cudaError_t ex_ratio(const ExArgs& a, int batch, cudaStream_t stream);
cudaError_t mm_batch(const MMBArgs& a, int batch, int sms, cudaStream_t stream);

// A small batch sharing grid, dictionary and eps solved in one launch (ragged.cuh, compiled in
// otlm_api.cu); outputs as otlm_solve, any of g, t_out, iters, err, status, dw may be null.
struct SmallSolve {
  int batch, n, k, datafit, penalty, max_iter, mm_steps;
  double eps, lam, alpha, beta, tol;
  const float *x, *D, *y;
  float *w, *g, *t_out;
  int* iters;
  float* err;
  int* status;
  float* dw;
  int empty_t0 = 0;  // tensor-core handles: t = 0 where the target sum is empty, whatever g is there
};
cudaError_t small_solve(const SmallSolve& c, cudaStream_t stream);

}  // namespace otlm
