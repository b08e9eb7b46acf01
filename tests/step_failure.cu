// Host harness: run_slabs (csrc/lbm_internal.h) when its k-th launch fails, for
// every k.  Arguments: nz periodic slabs depth count.  Prints per k: the
// reported whole steps and torn flag, the fewest and most steps any plane
// has taken, and the error; the last line is the run without a failure.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../paper_1503_03337_gb300/csrc/lbm_internal.h"

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  const int nz = std::atoi(argv[1]);
  lbm::SlabPlan p;
  p.slabs = std::atoi(argv[3]);
  p.depth = std::atoi(argv[4]);
  for (int k = 0;; ++k) {
    int seen = 0;
    std::vector<int> taken(nz, 0);
    lbm::StepProgress done{-1, true};
    const cudaError_t e = lbm::run_slabs(
        nz, std::atoi(argv[2]) != 0, p, std::atoll(argv[5]),
        [&](int64_t, int z0, int planes) {
          if (seen++ == k) return cudaErrorInvalidConfiguration;
          for (int z = z0; z < z0 + planes; ++z) ++taken[z % nz];
          return cudaSuccess;
        },
        &done);
    std::printf("%lld %d %d %d %d\n", (long long)done.steps, (int)done.torn,
                *std::min_element(taken.begin(), taken.end()),
                *std::max_element(taken.begin(), taken.end()), (int)e);
    if (e == cudaSuccess) break;
  }
  return 0;
}
