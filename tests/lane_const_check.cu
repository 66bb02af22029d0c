// Host driver for tests/test_lane_constants.py: prints (hex doubles) the interpolation constants
// of paper_2301_05985_gb300/csrc/lane_ops.cuh: rho, then a^0 .. a^6.
#include <cstdio>

#include "lane_ops.cuh"

int main() {
  std::printf("%a\n", kRho);
  for (int n = 0; n <= 6; ++n) std::printf("%a\n", ipow(kVal, n));
  return 0;
}
