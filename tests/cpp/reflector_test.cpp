// The reflector of the on-chip tridiagonalisation (csrc/reflector.h) against the
// formulas in extended precision.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_1611_03189_gb300/csrc/reflector.h"

using namespace hs;

// |x - exact| in units in the last place of T at exact
template <typename T>
static double ulps(T x, long double exact) {
  int e;
  std::frexp((double)exact, &e);
  const long double ulp = std::ldexp(1.0L, e - (sizeof(T) == 4 ? 24 : 53));
  return (double)(std::fabs((long double)x - exact) / ulp);
}

template <typename T>
static int check(double limit) {
  std::mt19937_64 rng(sizeof(T));
  std::uniform_real_distribution<double> mant(1.0, 2.0), ex(-44.0, 6.0);
  double worst_tau = 0, worst_scale = 0, worst_orth = 0;
  for (int i = 0; i < 2000000; ++i) {
    T alpha = (T)(mant(rng) * std::exp2(std::floor(ex(rng)))), tail2 = (T)(mant(rng) * std::exp2(std::floor(2 * ex(rng))));
    if (i % 3 == 0) tail2 = (T)((double)alpha * alpha * std::exp2(-60.0 * (i % 1000) / 1000.0));   // small tails
    if (i % 5 == 0) alpha = -alpha;
    if (i % 1001 == 0) alpha = T(0);
    T scale, tau, xn2;
    reflector(tail2, alpha, scale, tau, xn2);
    if (!(tail2 > (sizeof(T) == 4 ? T(1e-30f) : T(1e-290)))) {
      if (tau != 0 || scale != 0 || beta_of(beta_code(tau, xn2, alpha), false) != (double)alpha) return 1;
      continue;
    }
    const long double a = std::fabs((long double)alpha), s = sqrtl((long double)xn2);
    if (tau == 0 || (scale < 0) != std::signbit((double)alpha)) return 2;
    worst_tau = std::fmax(worst_tau, ulps<T>(tau, (a + s) / s));
    worst_scale = std::fmax(worst_scale, ulps<T>(std::fabs(scale), 1 / (a + s)));
    // H^T H = I: tau |v|^2 = 2
    const long double vv = 1 + (long double)tail2 * scale * scale;
    worst_orth = std::fmax(worst_orth, (double)(std::fabs(tau * vv - 2) / std::ldexp(1.0L, sizeof(T) == 4 ? -24 : -53)));
    const double beta = beta_of(beta_code(tau, xn2, alpha), true);
    if (ulps<double>(std::fabs(beta), s) > 0.5 + 1e-3 || (beta > 0) != std::signbit((double)alpha)) return 3;
  }
  if (worst_tau > limit || worst_scale > limit || worst_orth > 8.0) {
    std::printf("tau %.4f, scale %.4f ulp, |tau v.v - 2| %.2f u\n", worst_tau, worst_scale, worst_orth);
    return 4;
  }
  // a tail of sqrt(u) / 100 beside a large alpha is not lost
  const T alpha = (T)0.7, tail = (T)(0.7 * (sizeof(T) == 4 ? 2e-6 : 1e-10));
  T scale, tau, xn2;
  reflector(tail * tail, alpha, scale, tau, xn2);
  const T v = tail * scale, left = tail - tau * v * (alpha + tail * v);   // H x below its first entry
  if (std::fabs(left) > 4 * (sizeof(T) == 4 ? 6e-8 : 1.1e-16) * tail) return 5;
  return 0;
}

int main() {
  // FP32: FP64 results rounded; FP64: a root, a sum and a quotient, whose roundings
  // are a unit in the last place each at most
  const int f = check<float>(0.51), d = f ? f : check<double>(3.0);
  if (f || d) {
    std::printf("failed: %d %d\n", f, d);
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
