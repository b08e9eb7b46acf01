// Host harness: prints the launches of run_slabs (csrc/lbm_internal.h), one
// "step plane planes" line each.  Arguments: nz periodic slabs depth count.
#include <cstdio>
#include <cstdlib>

#include "../paper_1503_03337_gb300/csrc/lbm_internal.h"

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  lbm::SlabPlan p;
  p.slabs = std::atoi(argv[3]);
  p.depth = std::atoi(argv[4]);
  lbm::run_slabs(std::atoi(argv[1]), std::atoi(argv[2]) != 0, p, std::atoll(argv[5]),
                 [](int64_t s, int z0, int planes) {
                   std::printf("%lld %d %d\n", (long long)s, z0, planes);
                   return cudaSuccess;
                 });
  return 0;
}
