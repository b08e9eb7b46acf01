// Dispatch of the Q = 18 steps by storage type and rounding, and the FP32 step
// kernels (see lbm_step_impl.cuh); every other type has a unit of its own, so
// that they compile in parallel.
#include "lbm_step_impl.cuh"

namespace lbm {

LBM_STEP_EXTERN(18, double, false);
LBM_STEP_EXTERN(18, __half, false);
LBM_STEP_EXTERN(18, __half, true);
LBM_STEP_EXTERN(18, __nv_bfloat16, false);
LBM_STEP_EXTERN(18, __nv_bfloat16, true);

cudaError_t launch_step_q18(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                            const SlabPlan& plan, cudaStream_t st, StepProgress* done) {
  return launch_storage<18>(d, n, count, b, plan, st, done);
}

}  // namespace lbm
