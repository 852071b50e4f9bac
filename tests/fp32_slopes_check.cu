// Host-only check (compiled by tests/test_fp32_slopes.py): the FP32 half slopes
// against half of the limiter's definition, on random one-sided differences
// and every pair of special ones (zeros, infinities, NaN).
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_2510_24175_gb300/csrc/mhd_physics.cuh"

using namespace mhd;

int main() {
  std::mt19937_64 g(3);
  Phys<float> ph{};
  long long bad = 0;
  auto check = [&](float dm, float dp) {
    const float mc = half_slope_mc(dm, dp, ph), mm = half_slope_minmod(dm, dp);
    bad += mc != 0.5f * limited_slope<float>(dm, dp, kLimMC);
    bad += mm != 0.5f * limited_slope<float>(dm, dp, kLimMinmod);
  };
  auto draw = [&] {
    const float m = 1.0f + (float)(g() & 0x7fffff) / 8388608.0f;
    return std::ldexp((g() & 1) ? m : -m, (int)(g() % 80) - 40);
  };
  for (int i = 0; i < 2000000; ++i) {
    const float a = draw();
    check(a, draw());
    check(a, a * (1.0f + (float)(g() % 9) - 4.0f));
  }
  const float s[] = {0.0f, -0.0f, 1.0f, -1.0f, 3.5f, INFINITY, -INFINITY, NAN, -NAN};
  for (float a : s)
    for (float b : s) check(a, b);
  std::printf("%lld differences\n", bad);
  return bad != 0;
}
