// Step kernels for Q = 18, BF16 storage, rounding to nearest (see lbm_step_impl.cuh).
#include "lbm_step_impl.cuh"

namespace lbm {

LBM_STEP_UNIT(18, __nv_bfloat16, false);

}  // namespace lbm
