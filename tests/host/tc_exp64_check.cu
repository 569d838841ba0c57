// Host program that checks exp64 and log64 (csrc/tc_exp64.cuh) against the C library's
// long-double functions (not part of libtc_gb300.so; built and run by tests/test_exp64.py).
// Prints one JSON object: the largest errors in units in the last place over a sweep of
// each function's range, near its special points, and the results at the ends.
#include <cfloat>
#include <cmath>
#include <cstdio>

#include "tc_exp64.cuh"

using namespace tcg;

static double ulps(double got, long double want) {
  int e;
  (void)std::frexp((double)want, &e);
  return (double)(std::fabs((long double)got - want) / std::ldexp(1.0L, e - 53));
}

int main() {
  double e_all = 0, e_small = 0, l_all = 0, l_one = 0, l_ends = 0;
  unsigned long long s = 12345;
  auto rnd = [&]() {  // splitmix64 (Steele, Lea & Flood 2014)
    unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (double)((z ^ (z >> 31)) >> 11) * 0x1p-53;
  };
  for (int i = 0; i < 2000000; ++i) {
    double x = -708.0 + 1417.0 * rnd();
    e_all = std::fmax(e_all, ulps(exp64(x), std::exp((long double)x)));
    x = (rnd() - 0.5) * std::exp2(-60.0 * rnd());
    e_small = std::fmax(e_small, ulps(exp64(x), std::exp((long double)x)));
    x = std::exp2(-1021.0 + 2044.0 * rnd());
    l_all = std::fmax(l_all, ulps(log64(x), std::log((long double)x)));
    x = 1.0 + (rnd() - 0.5) * std::exp2(-50.0 * rnd());
    if (x != 1.0) l_one = std::fmax(l_one, ulps(log64(x), std::log((long double)x)));
  }
  // the edges of the logarithm's bins
  for (int j = 0; j <= 128; ++j)
    for (int d = -1; d <= 1; ++d) {
      double x = from_words(0x3fe69000 + j * 0x2000, 0);
      if (d) x = std::nextafter(x, d > 0 ? 2.0 : 0.0);
      if (x != 1.0) l_ends = std::fmax(l_ends, ulps(log64(x), std::log((long double)x)));
    }
  const double nan = NAN;
  const bool ends = exp64(0.0) == 1.0 && exp64(-0.0) == 1.0 && exp64(-708.5) == std::exp(-708.5) && exp64(-745.0) == std::exp(-745.0) && exp64(-746.0) == 0.0 &&
                    exp64(-1e300) == 0.0 && exp64(709.7) == std::exp(709.7) && exp64(709.8) == INFINITY &&
                    exp64(-INFINITY) == 0.0 && exp64(INFINITY) == INFINITY &&
                    exp64(1e300) == INFINITY && std::isnan(exp64(nan)) && std::isnan(exp64(-nan)) && log64(1.0) == 0.0 &&
                    log64(0.0) == -INFINITY && log64(-0.0) == -INFINITY && std::isnan(log64(-1.0)) &&
                    std::isnan(log64(nan)) && log64(INFINITY) == INFINITY && log64(DBL_MIN / 4) == std::log(DBL_MIN / 4);
  printf("{\"exp\": %.4f, \"exp_small\": %.4f, \"log\": %.4f, \"log_one\": %.4f, \"log_bins\": %.4f, \"ends\": %d}\n",
         e_all, e_small, l_all, l_one, l_ends, (int)ends);
  return 0;
}
