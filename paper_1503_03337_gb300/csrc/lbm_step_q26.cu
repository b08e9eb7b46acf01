// Step kernels for Q = 26 with FP64 and FP32 storage (see lbm_step_impl.cuh);
// the 2-byte storage types are in lbm_step_q26h.cu, so the two compile in
// parallel.
#include "lbm_step_impl.cuh"

namespace lbm {

cudaError_t launch_step_q26_half(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                                 const SlabPlan& plan, cudaStream_t st);

cudaError_t launch_step_q26(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                            const SlabPlan& plan, cudaStream_t st) {
  switch (d.storage) {
    case LBM_STORAGE_F64: return launch_typed<26, double, double>(d, n, count, b, plan, st);
    case LBM_STORAGE_F32: return launch_typed<26, float, float>(d, n, count, b, plan, st);
    case LBM_STORAGE_F16:
    case LBM_STORAGE_BF16: return launch_step_q26_half(d, n, count, b, plan, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm
