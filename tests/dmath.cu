// Host check of the FP64 functions of fx/dmath.cuh (compiled by
// tests/test_dmath.py with nvcc and run on the CPU): errors in ulps against
// the long double functions, over random arguments and the neighbourhoods
// where the seeds are worst. The host's FP32 seeds are off by two ulps, more
// than the hardware's.
#include <cmath>
#include <cstdio>
#include <random>

#include "fx/dmath.cuh"

using namespace fx::dm;

static double ulps(double got, long double ref) {
  int e;
  frexp(double(ref), &e);
  return double(fabsl((long double)got - ref) / ldexpl(1.0L, e - 53));
}

int main() {
  std::mt19937_64 g(1);
  std::normal_distribution<double> nd;
  std::uniform_real_distribution<double> ud(-1, 1);
  double me = 0, ms = 0, md = 0;
  long refused = 0;
  for (long i = 0; i < 2000000; ++i) {
    double x = i % 3 == 0 ? nd(g) : i % 3 == 1 ? 699.9 * ud(g) : std::ldexp(ud(g), -int(g() % 1000));
    if (exp_fast_ok(x)) me = fmax(me, ulps(exp_fast(x), expl((long double)x)));
    else ++refused;

    double s = std::fabs(nd(g));
    if (i % 4 == 0) s = std::ldexp(s, int(g() % 2000) - 1000);
    if (i % 7 == 0) s = std::nextafter(std::ldexp(1.0, int(g() % 40) - 20), i % 2 ? 0.0 : 1e9);
    if (sqrt_fast_ok(s)) ms = fmax(ms, ulps(sqrt_fast(s), sqrtl((long double)s)));
    else ++refused;

    double a = nd(g), b = 1 + std::exp(nd(g));
    if (i % 4 == 0) {
      a = std::ldexp(a, int(g() % 780) - 390);
      b = std::ldexp(nd(g), int(g() % 780) - 390);
    }
    if (i % 11 == 0) b = std::nextafter(std::ldexp(1.0, int(g() % 40) - 20), i % 2 ? 0.0 : 1e9);
    if (i % 13 == 0) a = b;
    if (i % 17 == 0) a = std::nextafter(b, i % 2 ? 0.0 : 1e300);
    if (div_fast_ok(a, b)) md = fmax(md, ulps(div_fast(a, b), (long double)a / (long double)b));
    else ++refused;
  }
  long bad = 0;
  const double inf = HUGE_VAL, nan = std::nan(""), sub = 0x1p-1060, big = 0x1p1000;
  for (double v : {inf, -inf, nan, 700.0, -700.0, 1e300}) bad += exp_fast_ok(v);
  for (double v : {inf, nan, 0.0, -0.0, -1.0, sub}) bad += sqrt_fast_ok(v);
  for (double v : {inf, -inf, nan, 0.0, -0.0, sub, big}) bad += div_fast_ok(v, 1.0) + div_fast_ok(1.0, v);
  bad += exp_fast(0.0) != 1.0 || exp_fast(-0.0) != 1.0 || sqrt_fast(4.0) != 2.0 || div_fast(-6.0, 3.0) != -2.0;
  printf("exp %.4f sqrt %.4f div %.4f refused %ld bad %ld\n", me, ms, md, refused, bad);
  return 0;
}
