// Host harness: FastDiv (csrc/lbm_internal.h) against the division, around the
// multiples of every divisor; prints the number of quotients that differ.
#include <cstdio>

#include "../paper_1503_03337_gb300/csrc/lbm_internal.h"

int main() {
  long bad = 0;
  const long top = (1l << 31) - 1;
  for (long n = 1; n <= top; n = n < 5000 ? n + 1 : n * 17 / 16) {
    const lbm::FastDiv q((int)n);
    for (long k = 0; k <= top / n; k = k < 40 ? k + 1 : k * 9 / 8)
      for (long i = k * n - 1; i <= k * n + 1; ++i)
        if (i >= 0 && i <= top && q((int)i) != i / n) ++bad;
    for (long i = top - 2 * (n < 1000 ? n : 1000); i <= top; ++i)
      if (i >= 0 && q((int)i) != i / n) ++bad;
  }
  std::printf("%ld\n", bad);
  return 0;
}
