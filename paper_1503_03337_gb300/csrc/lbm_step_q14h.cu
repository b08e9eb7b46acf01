// Step kernels for Q = 14, FP16 storage, rounding to nearest (see lbm_step_impl.cuh).
#include "lbm_step_impl.cuh"

namespace lbm {

LBM_STEP_UNIT(14, __half, false);

}  // namespace lbm
