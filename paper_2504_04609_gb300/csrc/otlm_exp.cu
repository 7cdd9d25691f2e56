// Block-expansion applies and the batched MM step (exp_solver.cuh) in a translation unit of their own.
#include "exp_solver.cuh"

namespace otlm {

cudaError_t ex_plan(const float* xt, int n, ExPlan* plan, int batch, int* with_plan, int* without, cudaStream_t stream) {
  ex_plan_kernel<<<1, 1024, 0, stream>>>(xt, n, plan, batch, with_plan, without);
  return cudaGetLastError();
}
cudaError_t ex_apply_source(const ExArgs& a, int batch, bool tc, int sms, cudaStream_t stream) {
  return tc ? launch_ex_apply<EXA_SOURCE, true>(a, batch, sms, stream) : launch_ex_apply<EXA_SOURCE, false>(a, batch, sms, stream);
}
cudaError_t ex_apply_target(const ExArgs& a, int batch, bool tc, int sms, cudaStream_t stream) {
  return tc ? launch_ex_apply<EXA_TARGET, true>(a, batch, sms, stream) : launch_ex_apply<EXA_TARGET, false>(a, batch, sms, stream);
}
cudaError_t ex_ratio(const ExArgs& a, int batch, cudaStream_t stream) {
  ex_ratio_kernel<<<batch, 256, 0, stream>>>(a);
  return cudaGetLastError();
}
cudaError_t mm_batch(const MMBArgs& a, int batch, int sms, cudaStream_t stream) {
  return launch_mm_batch(a, batch, sms, stream);
}

}  // namespace otlm
