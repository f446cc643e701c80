// Largest relative error of em1_series against long double over |x| <= kEm1Small: in FP64
// (the series' own), in FP32, where and at the ends; its values at 0.
#include <cmath>
#include <cstdio>

#include "../paper_1305_2418_gb300/csrc/em1_series.h"

int main() {
  double w64 = 0.0, w32 = 0.0;
  const int n = 200000;
  for (int q = -n; q <= n; ++q) {
    const float x = kEm1Small * (float)q / (float)n;
    if (x == 0.f) continue;
    const long double ref = expm1l((long double)x);
    const double a = (double)std::fabs((em1_series((double)x) - ref) / ref);
    const double b = (double)std::fabs(((long double)em1_series(x) - ref) / ref);
    if (a > w64) w64 = a;
    if (b > w32) w32 = b;
  }
  auto end = [](double x) { return std::fabs(em1_series(x) / std::expm1(x) - 1.0); };
  std::printf("%.4e %.4e %.4e %.4e %d\n", w64, w32, end(-(double)kEm1Small),
              end((double)kEm1Small), em1_series(0.f) == 0.f);
  return 0;
}
