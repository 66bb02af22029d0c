// Host driver for tests/test_double_float_split.py: per input line "x a_hi a_lo b_hi b_lo c_hi
// c_lo" (hex floats) prints the split of the double x, the double joined from it, and the
// quick sum a + b, difference a - b and fused a b + c of
// paper_2301_05985_gb300/csrc/df32.cuh.
#include <cstdio>

#include "df32.cuh"

int main() {
  double x;
  float v[6];
  while (std::scanf("%la %a %a %a %a %a %a", &x, &v[0], &v[1], &v[2], &v[3], &v[4], &v[5]) == 7) {
    const df a(v[0], v[1]), b(v[2], v[3]), c(v[4], v[5]);
    const df s = df_split(x), p = add_q(a, b), m = sub_q(a, b), f = fma_q(a, b, c);
    std::printf("%a %a %a %a %a %a %a %a %a\n", s.hi, s.lo, df_to_double(s), p.hi, p.lo, m.hi, m.lo, f.hi, f.lo);
  }
  return 0;
}
