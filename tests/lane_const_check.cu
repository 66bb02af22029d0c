// Host driver for tests/test_lane_constants.py: prints (hex) the interpolation constants of
// paper_2301_05985_gb300/csrc/lane_ops.cuh: rho, then a^0 .. a^6; then per input line "x n e"
// (x a hex float) the FP32 product x a^n 2^e.
#include <cstdio>

#include "lane_ops.cuh"

int main() {
  std::printf("%a\n", kRho);
  for (int n = 0; n <= 6; ++n) std::printf("%a\n", ipow(kVal, n));
  float x;
  int n, e;
  while (std::scanf("%a %d %d", &x, &n, &e) == 3) std::printf("%a\n", times_const_f(x, ipow(kVal, n), e));
  return 0;
}
