// The fixed-point FP64 reciprocal and square root (compiled by
// tests/test_fixed_point_seeds.py) against long double, without arguments on the
// host with seeds moved by every -4..4 units of 2^-24 (a relative error up to
// 2^-21, the bound that their derivation assumes), with an argument on the GPU
// with the seeds the kernels use, whose own errors are checked too.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2510_24175_gb300/csrc/mhd_physics.cuh"

using namespace mhd;

static double ulps(double got, long double want) {
  const double w = (double)want;
  return (double)(fabsl((long double)got - want) / (long double)(std::nextafter(w, HUGE_VAL) - w));
}

static double operand(std::mt19937_64& g, long long i) {
  unsigned long long m = g() & 0xfffffffffffffull;
  if (i % 4 == 1) m &= ~0ull << (g() % 52);       // few leading bits
  if (i % 4 == 2) m |= 0xfffffffffffffull >> (g() % 52);  // trailing ones
  if (i % 4 == 3) m = (i & 8) ? g() % 64 : 0xfffffffffffffull - g() % 64;  // next to 1 and 2
  const unsigned long long ex = i % 16 == 0 ? (i & 16 ? 64 : 1982) : 64 + g() % 1919;
  return bits2d((long long)((ex << 52) | m));
}

struct Moved {  // a seed function moved by u
  float u;
  bool root;
  MHD_HD float operator()(float f) const { return (root ? seed_rsqrt(f) : seed_rcp(f)) + u; }
};
MHD_HD float seed_arg(double x) {  // in [1, 2)
  return bits_f32(0x3f800000u | (((uint32_t)(dbits(x) >> 32) & 0xfffffu) << 3));
}

__global__ void eval(const double* x, double* r, double* s, float* er, float* es, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = rcp(x[i]);
  s[i] = tsqrt(x[i]);
  const float f = seed_arg(x[i]);
  er[i] = seed_rcp(f);
  es[i] = seed_rsqrt((i & 1) ? f + f : f);
}

int main(int argc, char**) {
  std::mt19937_64 g(7);
  double er = 0.0, es = 0.0, sr = 0.0, ss = 0.0;
  if (argc == 1) {
    for (long long i = 0; i < 400000; ++i) {
      const double x = operand(g, i);
      for (int d = -4; d <= 4; ++d) {
        const float u = d * 5.9604645e-8f;
        er = fmax(er, ulps(rcp_fixed(x, Moved{u, false}), 1.0L / (long double)x));
        es = fmax(es, ulps(sqrt_fixed(x, Moved{u, true}), sqrtl((long double)x)));
      }
    }
  } else {
    const int n = 1 << 22;
    std::vector<double> x(n), r(n), s(n);
    std::vector<float> fr(n), fs(n);
    for (int i = 0; i < n; ++i) x[i] = operand(g, i);
    double *dx, *dr, *ds;
    float *dfr, *dfs;
    if (cudaMalloc(&dx, n * 8) || cudaMalloc(&dr, n * 8) || cudaMalloc(&ds, n * 8) ||
        cudaMalloc(&dfr, n * 4) || cudaMalloc(&dfs, n * 4) ||
        cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice))
      return 2;
    eval<<<n / 256, 256>>>(dx, dr, ds, dfr, dfs, n);
    if (cudaMemcpy(r.data(), dr, n * 8, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(s.data(), ds, n * 8, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(fr.data(), dfr, n * 4, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(fs.data(), dfs, n * 4, cudaMemcpyDeviceToHost))
      return 3;
    for (int i = 0; i < n; ++i) {
      er = fmax(er, ulps(r[i], 1.0L / (long double)x[i]));
      es = fmax(es, ulps(s[i], sqrtl((long double)x[i])));
      const double f = seed_arg(x[i]);
      sr = fmax(sr, fabs(fr[i] * f - 1.0));
      ss = fmax(ss, fabs(fs[i] * std::sqrt((i & 1) ? f + f : f) - 1.0));
    }
  }
  printf("reciprocal %.4f ulp, square root %.4f ulp, seeds 2^%.1f, 2^%.1f\n", er, es,
         sr > 0 ? std::log2(sr) : 0.0, ss > 0 ? std::log2(ss) : 0.0);
  return er <= 0.51 && es <= 0.51 && sr < 0x1p-21 && ss < 0x1p-21 ? 0 : 1;
}
