// The barrier and dual step of one column (Eqs. Simple-Update:Barrier-X and Simple-Update:Dual) in
// FP64 from two FP32 estimates, for the device and, with estimates of its own, for a host test.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define ABIP_HD __host__ __device__ __forceinline__
#else
#define ABIP_HD inline
#endif

namespace abip {

// x and s, the roots of t^2 - omega t - c = 0 in absolute value: the larger, L = (|omega| + D) / 2 with D
// the root of the discriminant, and c / L.
//   D: Goldschmidt's coupled iteration (R. E. Goldschmidt, 1964; in the fused form of P. Markstein,
//      "Software division and square root using Goldschmidt's algorithms", 2004): g -> sqrt(disc) and
//      h -> 1 / (2 sqrt(disc)) from one estimate r of 1 / sqrt(disc), one step, then Newton's correction
//      of g by its residual.  An estimate off by d leaves 1.5 d^2 after the step and its square after
//      the correction: d = 2^-22 is far more than enough.
//   c / L: Newton's iteration for 1 / L from an estimate of it, one step, the quotient corrected by its
//      residual.
// Every multiply-add is spelled out, so the bits are the same wherever it is compiled.  With u = 2^-53
// the error is the roundings': disc (u, of which D has half), D (u), the sum (u), and for c / L one
// more: at most 2.5 u for the larger root and 3.5 u for the smaller.  Measured over omega in
// +-[1e-15, 1e15] and c in [1e-30, 1e2], estimates off by 2^-22: 2.3 u and 2.5 u.
// rsqrt32, rcp32: FP32 estimates.  Where disc lies outside what they take, the closed form.
template <typename Rsqrt, typename Rcp>
ABIP_HD void barrier_step_refined(double omega, double c, Rsqrt rsqrt32, Rcp rcp32, double& x, double& s) {
  const double aw = fabs(omega), disc = fma(omega, omega, 4.0 * c);
  double L, small;
  if (disc > 1e-30 && disc < 1e30) {
    const double r = (double)rsqrt32((float)disc);
    double g = disc * r, h = 0.5 * r;
    const double e = fma(-g, h, 0.5);
    g = fma(g, e, g);
    h = fma(h, e, h);
    L = 0.5 * (aw + fma(fma(-g, g, disc), h, g));
    double q = (double)rcp32((float)L);
    q = fma(q, fma(-L, q, 1.0), q);
    const double t = c * q;
    small = fma(q, fma(-L, t, c), t);
  } else {
    L = 0.5 * (aw + sqrt(disc));
    small = c / L;
  }
  x = omega >= 0.0 ? L : small;
  s = omega >= 0.0 ? small : L;
}

}  // namespace abip
