// Largest errors (in ulp of the FP64 result) of lean_exp and lean_rsqrt against
// long double over seeded arguments, and their values at the edges.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_1305_2418_gb300/csrc/lean_fp64.cuh"

static double ulp(double y) {
  int e;
  std::frexp(y, &e);
  return std::ldexp(1.0, e - 53);
}

int main() {
  std::mt19937_64 g(5);
  double we = 0.0, wr = 0.0;
  for (int q = 0; q < 2000000; ++q) {
    const double s = std::uniform_real_distribution<double>(-1, 1)(g);
    const double x = (q & 1) ? 40.0 * s : std::ldexp(s, (int)(g() % 60) - 50);
    const long double ref = expl((long double)x);
    const double e = (double)(std::fabs((long double)lean_exp(x) - ref) / ulp((double)ref));
    if (e > we) we = e;
    const double a = std::exp(60.0 * s);
    const long double rr = 1.0L / sqrtl((long double)a);
    const double r = (double)(std::fabs((long double)lean_rsqrt(a) - rr) / ulp((double)rr));
    if (r > wr) wr = r;
  }
  std::printf("%.4f %.4f %d %d %d\n", we, wr, lean_exp(0.0) == 1.0, lean_exp(-800.0) == 0.0,
              std::isnan(lean_exp(NAN)) && std::isinf(lean_exp(1000.0)));
  return 0;
}
