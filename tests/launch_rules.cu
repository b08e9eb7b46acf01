// Host harness: the launch rules of single-domain steps (csrc/lbm_step.cu),
// one answer per line of input.
//   block Q nx ny nz storage   ->  bx by linear
#include <cstdio>

#include "../paper_1503_03337_gb300/csrc/lbm_step.cu"

namespace lbm {
// the rules launch nothing
#define NO_LAUNCH(name)                                                                         \
  cudaError_t name(const DomainDesc&, int64_t, int64_t, BlockShape, const SlabPlan&, cudaStream_t, \
                   StepProgress*) {                                                             \
    return cudaSuccess;                                                                         \
  }
NO_LAUNCH(launch_step_q14)
NO_LAUNCH(launch_step_q18)
NO_LAUNCH(launch_step_q26)
}  // namespace lbm

int main() {
  int Q, nx, ny, nz, storage;
  while (std::scanf(" block %d %d %d %d %d", &Q, &nx, &ny, &nz, &storage) == 5) {
    const int64_t N = (int64_t)nx * ny * nz;
    const lbm::BlockShape b = lbm::default_block(Q, nx, ny, N, storage);
    std::printf("%d %d %d\n", b.bx, b.by, (int)lbm::steps_in_line(Q, nx, ny, N));
  }
  return 0;
}
