// Host driver for tests/test_inner_sums.py: argv trials, chunks; per trial the FP32 running sum
// of paper_2301_05985_gb300/csrc/dot4.cuh over that many float4 of products in [0.5, 1.5) and
// the exact sum's double (hex), and the sum of squares of the sums on the way.
#include <cstdio>
#include <cstdlib>

#include "dot4.cuh"

static double uniform(unsigned long long& s) {
  s = s * 6364136223846793005ull + 1442695040888963407ull;
  return 0.5 + (double)(s >> 40) / (double)(1 << 24);
}

int main(int, char** argv) {
  const int trials = std::atoi(argv[1]), chunks = std::atoi(argv[2]);
  unsigned long long st = 12345;
  for (int t = 0; t < trials; ++t) {
    float s = 0.f;
    double exact = 0.0, sq = 0.0;
    for (int c = 0; c < chunks; ++c) {
      float v[4];
      for (float& x : v) x = (float)uniform(st);
      s = dot4(make_float4(v[0], v[1], v[2], v[3]), make_float4(1.f, 1.f, 1.f, 1.f), s);
      exact += ((double)v[0] + v[1]) + ((double)v[2] + v[3]);  // 24-bit terms: exact in double
      sq += exact * exact;
    }
    std::printf("%a %a %a\n", s, exact, sq);
  }
  return 0;
}
