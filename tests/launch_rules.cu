// Host harness: the launch rules of single-domain steps (csrc/lbm_step.cu),
// one answer per line of input.
//   block Q nx ny nz storage              ->  bx by linear
//   tune Q nx ny nz storage solid per_z neq trials l2 -> slabs depth steps, candidates
//     of two cells a thread, the tuner's key (9 values)
//   count Q nx ny nz storage updates l2   ->  step launches of a walled box
#include <cstdio>
#include <cstring>

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
  char what[8];
  int Q, nx, ny, nz, storage;
  while (std::scanf(" %7s %d %d %d %d %d", what, &Q, &nx, &ny, &nz, &storage) == 6) {
    const int64_t N = (int64_t)nx * ny * nz;
    if (!std::strcmp(what, "block")) {
      const lbm::BlockShape b = lbm::default_block(Q, nx, ny, N, storage);
      std::printf("%d %d %d\n", b.bx, b.by, (int)lbm::steps_in_line(Q, nx, ny, N));
      continue;
    }
    long long l2;
    lbm::DomainDesc d{};
    d.Q = Q;
    d.nx = nx;
    d.ny = ny;
    d.nz = nz;
    d.N = N;
    d.storage = storage;
    if (!std::strcmp(what, "count")) {
      int updates, launches = 0;
      if (std::scanf("%d %lld", &updates, &l2) != 2) return 2;
      lbm::run_slabs(nz, false, lbm::slab_plan(d, l2), updates, [&](int64_t, int, int) {
        ++launches;
        return cudaSuccess;
      });
      std::printf("%d\n", launches);
      continue;
    }
    int solid, trials;
    if (std::scanf("%d %d %d %d %lld", &solid, &d.per[2], &d.neq_vel, &trials, &l2) != 5) return 2;
    const uint32_t mask = 0;  // any address: the rules only ask whether there is one
    d.solid = solid ? &mask : nullptr;
    const lbm::SlabPlan plan = lbm::slab_plan(d, l2);
    int pairs = 0;
    for (int bx : {32, 64, 128}) pairs += lbm::tune_candidate(d, {bx, 1, 2});
    std::printf("%d %d %d %d", plan.slabs, plan.depth, lbm::tune_steps(trials, plan), pairs);
    for (int v : lbm::tune_key(d, plan)) std::printf(" %d", v);
    std::printf("\n");
  }
  return 0;
}
