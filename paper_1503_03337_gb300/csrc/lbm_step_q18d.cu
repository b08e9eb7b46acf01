// Step kernels for Q = 18, FP64 storage (see lbm_step_impl.cuh).
#include "lbm_step_impl.cuh"

namespace lbm {

LBM_STEP_UNIT(18, double, false);

}  // namespace lbm
