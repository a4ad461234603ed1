// The Householder reflector of a column in the on-chip tridiagonalisation
// (kernels_cluster.cu); compiles for the host too.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define HS_REFL_FN __device__ __forceinline__
#else
#define HS_REFL_FN inline
#endif

namespace hs {

// H = I - tau v v^T, v = (1, tail scale), takes x = (alpha, tail) to (beta, 0),
// beta = -sign(alpha) sqrt(xn2): tau = (|alpha| + s) / s and scale = sign(alpha) /
// (|alpha| + s) with s = sqrt(xn2), xn2 = alpha^2 + tail2.  tail2 = |tail|^2 is
// summed without alpha: the difference |x|^2 - alpha^2 of rounded sums loses tails
// below sqrt(u) |alpha|, a backward error of sqrt(u) ||J||.
// A tail whose square leaves the range (J's largest diagonal entry is about 1) is
// no tail: tau = 0, beta = alpha.
//
// FP32: the root and both quotients carry their rounding errors along as a second
// word (fused multiply-adds make the residuals exact; T. J. Dekker, "A
// floating-point technique for extending the available precision", Numer. Math.
// 18, 1971), so tau and scale are the FP32 roundings of FP64 results without an
// FP64 instruction on a step's chain: they are within 0.51 units in the last place.
HS_REFL_FN void reflector(float tail2, float alpha, float &scale, float &tau, float &xn2) {
  if (!(tail2 > 1e-30f)) {
    scale = tau = xn2 = 0.f;
    return;
  }
  xn2 = fmaf(alpha, alpha, tail2);
  const float a = fabsf(alpha);
  const float s = sqrtf(xn2), inv = 1.f / s;
  const float sl = 0.5f * fmaf(-s, s, xn2) * inv;         // s + sl = sqrt(xn2)
  const float sum = a + s, suml = (a - (sum - s)) + sl;   // sum + suml = |alpha| + sqrt(xn2); a <= s
  const float r = 1.f / sum;
  scale = copysignf(fmaf(r, fmaf(-sum, r, 1.f) - r * suml, r), alpha);
  const float q = a * inv, t = 1.f + q;
  tau = t + fmaf(inv, fmaf(-q, s, a) - q * sl, q - (t - 1.f));
}

HS_REFL_FN void reflector(double tail2, double alpha, double &scale, double &tau, double &xn2) {
  if (!(tail2 > 1e-290)) {
    scale = tau = xn2 = 0.0;
    return;
  }
  xn2 = fma(alpha, alpha, tail2);
  const double a = fabs(alpha), s = sqrt(xn2);
  scale = copysign(1.0 / (a + s), alpha);
  tau = 1.0 + a / s;
}

// The off-diagonal entry of a step as the kernels keep it until the end (a square
// root in FP64 is taken off the steps' chain): xn2 with beta's sign, or alpha
// itself without a tail
template <typename T>
HS_REFL_FN double beta_code(T tau, T xn2, T alpha) {
  return tau == T(0) ? (double)alpha : -copysign((double)xn2, (double)alpha);
}
HS_REFL_FN double beta_of(double code, bool tail) { return tail ? copysign(sqrt(fabs(code)), code) : code; }

}  // namespace hs
