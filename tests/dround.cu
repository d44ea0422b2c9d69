// Host check that FP64 division and square root are correctly rounded wherever
// fx/dmath.cuh is sure of them (compiled by tests/test_dround.py with nvcc and
// run on the CPU, whose own operations are correctly rounded), over random
// arguments, both sides of powers of two, and quotients and roots near a tie.
// The host's FP32 seeds are off by two ulps, more than the hardware's.
#include <cmath>
#include <cstdio>
#include <random>

#include "fx/dmath.cuh"

using namespace fx::dm;

static long bad = 0, unsure = 0, n = 0;  // unsure, of the plain random arguments

static void root(double x, bool plain = false) {
  if (!sqrt_fast_ok(x)) return;
  bool sure;
  const double s = sqrt_fast(x, sure);
  n += plain;
  unsure += plain && !sure;
  bad += sure && s != std::sqrt(x);
}
static void quotient(double a, double b, bool plain = false) {
  if (!div_fast_ok(a, b)) return;
  bool sure;
  const double s = div_fast(a, b, sure);
  n += plain;
  unsure += plain && !sure;
  bad += sure && s != a / b;
}

int main() {
  std::mt19937_64 g(2);
  std::uniform_real_distribution<double> u(1, 2);
  auto scale = [&](double x) { return std::ldexp(x, int(g() % 700) - 350); };
  for (long i = 0; i < 8000000; ++i) {
    const double a = u(g), b = u(g);
    quotient(i % 5 ? a : scale(a), i % 5 ? b : scale(b), true);
    root(i % 2 ? a : 2 * b, true);
    if (i % 8 == 0) {
      const double p = std::ldexp(1.0, int(g() % 9) - 4);
      quotient(std::nextafter(p, i % 16 ? 0.0 : 4.0), b);
      quotient(a, std::nextafter(p, i % 16 ? 0.0 : 4.0));
      root(std::nextafter(p, i % 16 ? 0.0 : 4.0));
      quotient(p, b);
      quotient(b * p, b);
      root(b * b);
    }
    // near a tie: the argument nearest to that of a point midway between two results
    quotient(std::fma(a, b, b * std::ldexp(1.0, -53)), b);
    root(std::fma(a, a, a * std::ldexp(1.0, -52)));
  }
  printf("random %ld unsure %ld bad %ld\n", n, unsure, bad);
  return 0;
}
