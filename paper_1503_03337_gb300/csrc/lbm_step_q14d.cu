// Step kernels for Q = 14, FP64 storage (see lbm_step_impl.cuh).
#include "lbm_step_impl.cuh"

namespace lbm {

LBM_STEP_UNIT(14, double, false);

}  // namespace lbm
