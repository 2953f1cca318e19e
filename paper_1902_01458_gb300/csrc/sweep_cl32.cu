// The whole-sweep cluster kernels in FP32 (sweep_cl.cuh).
#include "sweep_cl.cuh"

double sweep_cl32_us(const rr_factors* fa, int k, int adjoint) {
  return sweepcl::make_plan<float>(fa->op->d, active_count(fa), k, adjoint).form_us;
}

rr_status launch_sweep_cl32(rr_factors* fa, int k, int adjoint, const void* in, void* x, void* h) {
  const sweepcl::Plan p = sweepcl::make_plan<float>(fa->op->d, active_count(fa), k, adjoint);
  return adjoint ? sweepcl::launch_plan<float, true>(fa, p, k, in, x, h)
                 : sweepcl::launch_plan<float, false>(fa, p, k, in, x, h);
}
