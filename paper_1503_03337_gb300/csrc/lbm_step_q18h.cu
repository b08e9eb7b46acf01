// Step kernels for Q = 18, FP16 storage, rounding to nearest (see lbm_step_impl.cuh).
#include "lbm_step_impl.cuh"

namespace lbm {

LBM_STEP_UNIT(18, __half, false);

}  // namespace lbm
