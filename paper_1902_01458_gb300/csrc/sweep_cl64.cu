// The whole-sweep cluster kernels in FP64 (sweep_cl.cuh).
#include "sweep_cl.cuh"

rr_status launch_sweep_cl64(rr_factors* fa, int k, int adjoint, const void* in, void* x, void* h) {
  const sweepcl::Plan p = sweepcl::make_plan<double>(fa->op->d, active_count(fa), k, adjoint);
  return adjoint ? sweepcl::launch_plan<double, true>(fa, p, k, in, x, h)
                 : sweepcl::launch_plan<double, false>(fa, p, k, in, x, h);
}
