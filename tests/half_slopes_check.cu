// Host-only check (compiled by tests/test_fp64_half_slopes.py): the slope functions
// that the FP64 kernels and the adjoint call, against the limiter's definition in
// plain IEEE operations, on random differences and every pair of special ones
// (signed zeros, subnormals, extremes, infinities), and the adjoint's multipliers
// for every derivative code.  Prints the disagreements.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_2510_24175_gb300/csrc/mhd_adjoint.cuh"

using namespace mhd;

// half the limited slope: min(|dm|, |dp|, (|dm| + |dp|) / 4) or min(|dm|, |dp|) / 2,
// a NaN difference (infinity times zero below) ordered as an infinite one
static double ref(double dm, double dp, bool mc) {
  if (dm != dm) dm = std::copysign(HUGE_VAL, dm);
  if (dp != dp) dp = std::copysign(HUGE_VAL, dp);
  if (dm == 0.0 || dp == 0.0 || (dm > 0.0) != (dp > 0.0)) return 0.0;
  const double am = fabs(dm), ap = fabs(dp);
  double h = am < ap ? am : ap;
  if (mc) {
    const double q = 0.5 * (0.5 * (am + ap));
    h = q < h ? q : h;
  } else {
    h = 0.5 * h;
  }
  return dm > 0.0 ? h : -h;
}

int main() {
  std::mt19937_64 g(5);
  Phys<double> ph{};
  long long bad = 0;
  auto check = [&](double dm, double dp) {
    bad += half_slope_mc(dm, dp, ph) != ref(dm, dp, true);
    bad += half_slope_minmod(dm, dp) != ref(dm, dp, false);
  };
  auto draw = [&](int range) {
    const double m = 1.0 + (double)(g() >> 12) / 4503599627370496.0;
    return std::ldexp((g() & 1) ? m : -m, (int)(g() % (2 * range)) - range);
  };
  for (int i = 0; i < 1000000; ++i) {
    const double a = draw(i & 1 ? 40 : 1070);  // (the wide range reaches subnormals)
    check(a, draw(40));
    check(a, a * (1.0 + (double)(g() % 9) - 4.0));
    check(a, a * std::ldexp((double)(g() >> 12), -51));
  }
  const double s[] = {0.0, -0.0, 4.9e-324, -4.9e-324, 1.5e-323, 2.2250738585072014e-308,
                      -2.2250738585072014e-308, 1.1125369292536007e-308, 1.0, -1.0, 3.5,
                      1.7976931348623157e308, -1.7976931348623157e308, 8.98846567431158e307,
                      HUGE_VAL, -HUGE_VAL};
  for (double a : s)
    for (double b : s) check(a, b);
  // codes: piece 0 .. 3, one-sided difference dp or dm
  for (unsigned code = 0; code < 8; ++code)
    for (int k = 0; k < 4; ++k) {
      const bool ok = k & 1, b = k & 2, m = code >> 2;
      const double one[4] = {0.0, 1.0, 2.0, 0.5}, v = ok ? one[code & 3] : 0.0;
      const bool central = (code & 3) == 3;
      const double dm = central || m ? v : 0.0, dp = central || !m ? v : 0.0;
      double hm, hp, c1;
      slope_code_half(code, ok, b, hm, hp, c1);
      bad += hm != 0.5 * dm || hp != 0.5 * dp || c1 != (b ? 1.0 - hm + hp : 1.0 + hm - hp);
    }
  std::printf("%lld disagreements\n", bad);
  return bad != 0;
}
