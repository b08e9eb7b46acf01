// Step kernels for Q = 26 with BF16 storage (see lbm_step_impl.cuh).
#include "lbm_step_impl.cuh"

namespace lbm {

cudaError_t launch_step_q26_bf16(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                                 const SlabPlan& plan, cudaStream_t st) {
  return launch_typed<26, __nv_bfloat16, float>(d, n, count, b, plan, st);
}

}  // namespace lbm
