// Host-only check (compiled by tests/test_fp64_fixed_point.py): the FP64
// reciprocal and square root that the kernels evaluate in 64-bit fixed point,
// against long double, on random and structured significands over the whole
// exponent range they accept.  Prints the largest errors in ulp.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_2510_24175_gb300/csrc/mhd_physics.cuh"

using namespace mhd;

static double ulps(double got, long double want) {
  const double w = (double)want;
  return (double)(fabsl((long double)got - want) / (long double)(std::nextafter(w, HUGE_VAL) - w));
}

int main() {
  std::mt19937_64 g(7);
  double er = 0.0, es = 0.0;
  long long range = 0;
  for (long long i = 0; i < 3000000; ++i) {
    unsigned long long m = g() & 0xfffffffffffffull;
    if (i % 4 == 1) m &= ~0ull << (g() % 52);       // few leading bits
    if (i % 4 == 2) m |= 0xfffffffffffffull >> (g() % 52);  // trailing ones
    if (i % 4 == 3) m = (i & 8) ? g() % 64 : 0xfffffffffffffull - g() % 64;  // next to 1 and 2
    const unsigned long long ex = i % 16 == 0 ? (i & 16 ? 64 : 1982) : 64 + g() % 1919;
    const double x = bits2d((long long)((ex << 52) | m));
    range += !in_fixed_range((uint32_t)(dbits(x) >> 32));
    er = fmax(er, ulps(rcp_fixed(x), 1.0L / (long double)x));
    er = fmax(er, ulps(-rcp_fixed(-x), 1.0L / (long double)x));
    es = fmax(es, ulps(sqrt_fixed(x), sqrtl((long double)x)));
  }
  const double out[] = {0.0, 4.9e-324, bits2d((63ll << 52) | 0xfffffffffffffll),
                        bits2d(1983ll << 52), HUGE_VAL, NAN};
  for (double x : out) range += in_fixed_range((uint32_t)(dbits(x) >> 32));
  printf("reciprocal %.4f ulp, square root %.4f ulp, %lld range errors\n", er, es, range);
  return er <= 0.51 && es <= 0.51 && range == 0 ? 0 : 1;
}
