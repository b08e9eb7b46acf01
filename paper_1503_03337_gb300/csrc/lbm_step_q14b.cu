// Step kernels for Q = 14, BF16 storage, rounding to nearest (see lbm_step_impl.cuh).
#include "lbm_step_impl.cuh"

namespace lbm {

LBM_STEP_UNIT(14, __nv_bfloat16, false);

}  // namespace lbm
