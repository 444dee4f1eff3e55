// barrier_step_refined on the host against the closed form in long double, from FP32 estimates that are
// off by 2^-22 either way (more than the hardware's: 2^-22.9 and one unit in the last place).  Built and
// run by tests/test_barrier_refined_cpu.py; prints "ok <errors in u = 2^-53>" and exits 0, or the worst case and 1.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "../paper_1805_12344_gb300/csrc/barrier_refined.h"

static uint64_t g_state = 1805;
static double uniform() {   // splitmix64
  uint64_t z = (g_state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return (double)((z ^ (z >> 31)) >> 11) * 0x1p-53;
}

static long double g_worst[2] = {0, 0};
static bool check(double omega, double c) {
  const long double aw = fabsl((long double)omega);
  const long double L = 0.5L * (aw + sqrtl((long double)omega * omega + 4.0L * c)), small = (long double)c / L;
  bool ok = true;
  for (int a = -1; a <= 1; ++a)
    for (int b = -1; b <= 1; ++b) {
      double x, s;
      abip::barrier_step_refined(omega, c, [a](float v) { return (float)((1.0 + a * 0x1p-22) / sqrt((double)v)); },
                                 [b](float v) { return (float)((1.0 + b * 0x1p-22) / (double)v); }, x, s);
      const double big = omega >= 0.0 ? x : s, less = omega >= 0.0 ? s : x;
      const long double e[2] = {fabsl(big - L) / L * 0x1p53L, fabsl(less - small) / small * 0x1p53L};
      for (int k = 0; k < 2; ++k)
        if (e[k] > g_worst[k]) g_worst[k] = e[k];
      // the roundings' 2.5 u and 3.5 u, and their second order
      if (!(e[0] <= 2.51L && e[1] <= 3.51L)) {
        if (ok) std::printf("FAIL omega %.17g c %.17g: %.3Lf u, %.3Lf u\n", omega, c, e[0], e[1]);
        ok = false;
      }
    }
  return ok;
}

int main() {
  bool ok = true;
  // zero, omega far above and below sqrt(c), both ends of the estimates' range and just outside it
  const std::vector<double> ws = {0.0, 1e-15, 9.99e-16, 1.01e-15, 1e-7, 1.0, 3.0, 1e12, 0.999e15, 1e15, 1.001e15, 1e100};
  const std::vector<double> cs = {1e-31, 2.4e-31, 2.5e-31, 2.6e-31, 1e-30, 1e-15, 1e-6, 1e-2, 1.0, 1e2, 2.4e29, 2.6e29};
  for (double w : ws)
    for (double c : cs) ok = check(w, c) && check(-w, c) && ok;
  for (int k = 0; k < 200000; ++k) {
    const double w = exp(log(1e-15) + uniform() * log(1e30)), c = exp(log(1e-30) + uniform() * log(1e32));
    ok = check(uniform() < 0.5 ? w : -w, c) && ok;
    const double near = 2.0 * sqrt(c) * (0.5 + uniform());   // omega^2 and 4 c alike: every rounding counts
    ok = check(uniform() < 0.5 ? near : -near, c) && ok;
  }
  if (ok) std::printf("ok %.3Lf %.3Lf\n", g_worst[0], g_worst[1]);
  return ok ? 0 : 1;
}
