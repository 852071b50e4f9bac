// Device-side pointwise physics of the GLM-MHD hot path, templated on the
// arithmetic type T (double for MHD_FP64, float for MHD_FP32).
//
// The stage structure is Section 3.2's (boundary calculation, cons->prim,
// reconstruction, Riemann solver, right-hand side); HLLD is named in
// Section 4.2 and divergence cleaning (GLM) in Section 4.2's strong-scaling
// paragraph.  The formulas are the published methods:
//   - HLLD: Miyoshi & Kusano (2005), J. Comput. Phys. 208: wave speeds
//     (Eq. 67), S_M and p_t* (Eqs. 38, 41), single-star states (Eqs. 43-48),
//     Alfven speeds S*_{L,R} (Eq. 51), double-star states (Eqs. 59-63),
//     fan-region fluxes (Eqs. 64-66).
//   - GLM interface values: Dedner et al. (2002), J. Comput. Phys. 175,
//     Eq. 41 (exact solution of the 2x2 (B_n, psi) Riemann problem).
//   - PLM slopes: minmod / monotonised-central limiters of van Leer (1977),
//     applied to primitive variables, with a zero-slope fallback for a cell
//     whose face density or pressure would be non-positive.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#define MHD_HD __host__ __device__ __forceinline__

namespace mhd {

enum { kRHO = 0, kVX = 1, kVY = 2, kVZ = 3, kBX = 4, kBY = 5, kBZ = 6, kPRS = 7, kPSI = 8,
       kNV = 9 };
enum { kLimFlat = 0, kLimMinmod = 1, kLimMC = 2, kLimWenoz = 3 };
// kBcHalo: the ghost cells of that side come from a caller-supplied halo buffer
// (a subdomain boundary of a decomposed grid)
enum { kBcPeriodic = 0, kBcOutflow = 1, kBcHalo = 2 };
// cons->prim flags: density floor, pressure floor, and (FP32 only) the
// pressure recomputed in FP64 because the FP32 value fell in the
// cancellation-dominated range
enum { kFloorRho = 1u, kFloorP = 2u, kPressF64 = 4u };

template <class T>
struct Phys {
  T gamma;      // adiabatic index
  T gm1;        // gamma - 1
  T gm1i;       // 1 / (gamma - 1)
  T gm1im1;     // 1 / (gamma - 1) - 1
  T rho_floor;
  T p_floor;
  double gm1_d, rho_floor_d, p_floor_d;  // FP64 gamma - 1 and floors for the floor branch
  T one = T(1), nzero = T(-0.0);  // operands of add_f / sub_f / mul_f
};

// Single-precision seeds of the FP64 reciprocal and square root below (the
// host build, used only by host-side unit harnesses, divides).
MHD_HD float seed_rcp(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / x;
#endif
}
MHD_HD float seed_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / sqrtf(x);
#endif
}
MHD_HD uint32_t f32_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  memcpy(&b, &x, sizeof(b));
  return b;
#endif
}
MHD_HD float bits_f32(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  memcpy(&x, &b, sizeof(x));
  return x;
#endif
}
MHD_HD uint32_t mulhi_u(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
MHD_HD int32_t mulhi_s(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }

// FP32 mode: hardware-approximate reciprocal and square root (a few ulp;
// the FP32 bulk path's error budget is ~1e-5 relative).
MHD_HD float rcp(float x) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.0f, x);
#else
  return 1.0f / x;
#endif
}
// A product and a fused multiply-add whose rounding the source fixes.  In a
// sum of two products the compiler may fuse either product into the add, and
// copies of the same code inlined at different sites (or kernels that differ
// only elsewhere) may then round differently; the sums whose results must
// not depend on where the code runs are written with these (the same number
// of instructions as the contracted form).
MHD_HD double mul_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
MHD_HD float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
MHD_HD double fma_rn(double a, double b, double c) { return fma(a, b, c); }
MHD_HD float fma_rn(float a, float b, float c) { return fmaf(a, b, c); }
// Sums, differences and products as fused multiply-adds with the constants 1
// and -0 (exact, so each rounds once, as the plain operation does).  The FP64
// unit takes a fused multiply-add of a warp with three register operands every
// 16.1 clocks, but an addition, a multiplication or a fused multiply-add with
// a constant operand only every 19.1.  The kernels therefore hold ph.one and
// ph.nzero in registers whose values the compiler cannot see (fp64_registers);
// elsewhere they are plain constants.  FP32 uses the plain operations.
MHD_HD double add_f(double a, double b, const Phys<double>& ph) { return fma(a, ph.one, b); }
MHD_HD double sub_f(double a, double b, const Phys<double>& ph) { return fma(-b, ph.one, a); }
MHD_HD double mul_f(double a, double b, const Phys<double>& ph) { return fma(a, b, ph.nzero); }
MHD_HD float add_f(float a, float b, const Phys<float>&) { return a + b; }
MHD_HD float sub_f(float a, float b, const Phys<float>&) { return a - b; }
MHD_HD float mul_f(float a, float b, const Phys<float>&) { return mul_rn(a, b); }
// a0 b0 + a1 b1 + a2 b2, rounded as fma(a2, b2, fma(a1, b1, a0 b0))
template <class T>
MHD_HD T dot3_f(T a0, T b0, T a1, T b1, T a2, T b2, const Phys<T>& ph) {
  return fma_rn(a2, b2, fma_rn(a1, b1, mul_f(a0, b0, ph)));
}

MHD_HD double tabs(double x) { return fabs(x); }
MHD_HD float tabs(float x) { return fabsf(x); }
MHD_HD double tmin(double a, double b) { return fmin(a, b); }
MHD_HD float tmin(float a, float b) { return fminf(a, b); }

// Bit-pattern helpers (the host build, used only by host-side harnesses,
// goes through memcpy).
MHD_HD long long dbits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long b;
  memcpy(&b, &x, sizeof(b));
  return b;
#endif
}
MHD_HD double bits2d(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  memcpy(&x, &b, sizeof(x));
  return x;
#endif
}

// FP64 reciprocal and square root without FP64 instructions.  The SM's FP64
// unit issues 2 lanes per clock against 128 for the integer and FP32 pipes, which
// idle beside it.  Time per warp and SM with the pipes full, in fused
// multiply-adds: CUDA's correctly rounded reciprocal 5.4, this one 1.4; CUDA's
// square root 9.0, this one 1.7.  A single-precision seed of the significand
// (relative error < 2^-21) is corrected in 64-bit fixed point: the residual against the
// full significand is exact to 2^-62, and the first- and second-order terms of
// the correction leave less than 2^-61, so the rounded result is within 0.51
// ulp.  Both need a biased exponent in [64, 1982] (in_fixed_range); other
// operands (zero, subnormal, extreme, infinite, NaN, negative for the root)
// take the CUDA function behind a branch.
MHD_HD bool in_fixed_range(uint32_t hi) { return ((hi >> 20) & 0x7ffu) - 64u < 1919u; }

// seed: the single-precision reciprocal (square root: reciprocal root) function.
template <class Seed>
MHD_HD double rcp_fixed(double x, Seed seed) {
  const uint64_t b = (uint64_t)dbits(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  // significand in [1, 2): xh 2^-31 + xl 2^-63
  const uint32_t xh = 0x80000000u | (hi << 11) | (lo >> 21), xl = lo << 11;
  const float r0 = seed(bits_f32(0x3f800000u | ((xh >> 8) & 0x7fffffu)));
  const float r = fminf(fmaxf(r0, 0.5f), 0.99999994f);
  const uint32_t y = (f32_bits(r) << 8) | 0x80000000u;  // seed, units 2^-32
  const int32_t yh = (int32_t)(y >> 1);                 // the same, units 2^-31
  // e = 1 - x y and the corrections y e, y e^2, units 2^-62
  const int64_t e = (int64_t)(0x4000000000000000ull -
                              ((uint64_t)xh * (uint32_t)yh + mulhi_u(xl, (uint32_t)yh)));
  const int64_t c = (((int64_t)(int32_t)(e >> 32) * yh) << 1) + mulhi_u((uint32_t)e, y);
  const int32_t c2 = mulhi_s((int32_t)(c >> 11), (int32_t)(e >> 11)) >> 8;
  const uint64_t q = ((uint64_t)(uint32_t)yh << 31) + (uint64_t)c + (uint64_t)(int64_t)c2;
  const uint64_t m = (q + 0x100u) >> 9;  // [2^52, 2^53]
  const uint64_t ex = (uint64_t)(2044u - ((hi >> 20) & 0x7ffu)) << 52;
  return bits2d((int64_t)((m + ex) | (b & 0x8000000000000000ull)));
}

template <class Seed>
MHD_HD double sqrt_fixed(double x, Seed seed) {
  const uint64_t b = (uint64_t)dbits(x);
  const uint32_t hi = (uint32_t)(b >> 32);
  const uint32_t odd = ((hi >> 20) & 1u) ^ 1u;  // odd exponent: significand in [2, 4)
  // m in [1, 4), units 2^-62
  const uint64_t m = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << (10 + odd);
  const float f = bits_f32((0x3f800000u + (odd << 23)) | (uint32_t)((b >> 29) & 0x7fffffu));
  const float y0 = fminf(fmaxf(seed(f), 0.5f), 0.99999994f);
  const float s0 = fminf(fmaxf(f * y0, 1.0f), 1.9999999f);
  const uint32_t t = (f32_bits(s0) << 8) | 0x80000000u;                  // units 2^-31
  const int32_t yh = (int32_t)(((f32_bits(y0) << 8) | 0x80000000u) >> 1);  // units 2^-31
  // sqrt(m) = t + d + d (e - d y / 2) with r = m - t^2, d = r y / 2, e = 1 - t y
  const int64_t r = (int64_t)(m - (uint64_t)t * t);
  const int64_t d = (int64_t)(int32_t)(r >> 32) * yh + mulhi_u((uint32_t)r, (uint32_t)yh);
  const int64_t e = (int64_t)(0x4000000000000000ull - (uint64_t)t * (uint32_t)yh);
  const int32_t ds = (int32_t)(d >> 12);  // units 2^-50
  const int32_t g = (int32_t)(e >> 12) - mulhi_s(ds, yh);
  const uint64_t q = ((uint64_t)t << 31) + (uint64_t)d + (uint64_t)(int64_t)(mulhi_s(ds, g) >> 6);
  const uint64_t s = (q + 0x200u) >> 10;  // [2^52, 2^53]
  const uint64_t ex = (uint64_t)((((hi >> 20) + 1023u) >> 1) - 1u) << 52;
  return bits2d((int64_t)(s + ex));
}

MHD_HD double rcp_fixed(double x) {
  return rcp_fixed(x, [](float f) { return seed_rcp(f); });
}
MHD_HD double sqrt_fixed(double x) {
  return sqrt_fixed(x, [](float f) { return seed_rsqrt(f); });
}

// (The CUDA functions as volatile asm: otherwise the compiler evaluates them
// for every operand and selects afterwards.)
MHD_HD double rcp(double x) {
#ifdef __CUDA_ARCH__
  double r = rcp_fixed(x);
  if (!in_fixed_range((uint32_t)__double2hiint(x)))
    asm volatile("rcp.rn.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
#else
  return 1.0 / x;
#endif
}
MHD_HD double tsqrt(double x) {
#ifdef __CUDA_ARCH__
  const uint32_t hi = (uint32_t)__double2hiint(x);
  double s = sqrt_fixed(x);
  if (!in_fixed_range(hi) || (int)hi < 0)
    asm volatile("sqrt.rn.f64 %0, %1;" : "=d"(s) : "d"(x));
  return s;
#else
  return sqrt(x);
#endif
}

// max that keeps a NaN once either operand has one (fmax drops NaNs).  Its
// operands are wave speeds or magnitudes: +0, positive, +inf or NaN.  For
// those, the unsigned order of the FP64 bit patterns is the numeric order
// with every NaN above +inf, so the device takes the FP64 max on the
// integer pipe (the FP64 pipe is the bound of the FP64 kernels).
MHD_HD double nan_max(double a, double b) {
#ifdef __CUDA_ARCH__
  const unsigned long long x = (unsigned long long)dbits(a), y = (unsigned long long)dbits(b);
  return bits2d((long long)(x > y ? x : y));
#else
  return (a != a || b > a || b != b) ? (a != a ? a : b) : a;
#endif
}
MHD_HD float nan_max(float a, float b) { return (a != a || b > a || b != b) ? (a != a ? a : b) : a; }
MHD_HD bool is_nan(double x) {
  return ((unsigned long long)dbits(x) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
}
MHD_HD bool is_nan(float x) { return x != x; }

// Sign tests and min / max with IEEE results (-0, subnormals, infinities and
// NaN included: a NaN compares false, and tmin2 / tmax2 return the other
// operand like fmin / fmax).  FP64 takes them on the integer pipe from the
// bit patterns: x > 0 exactly when the pattern lies in [1, +inf], x < 0 when
// it lies in [-0 + 1 ulp, -inf] (sign-magnitude order), and two doubles order
// like their patterns once the magnitude bits of negative ones are flipped.
MHD_HD bool gt0(double x) {
  return (unsigned long long)dbits(x) - 1ull < 0x7ff0000000000000ull;
}
MHD_HD bool lt0(double x) {
  return (unsigned long long)dbits(x) - 0x8000000000000001ull < 0x7ff0000000000000ull;
}
MHD_HD bool ge0(double x) {
  const unsigned long long b = (unsigned long long)dbits(x);
  return b <= 0x7ff0000000000000ull || b == 0x8000000000000000ull;
}
MHD_HD bool gt0(float x) { return x > 0.0f; }
MHD_HD bool lt0(float x) { return x < 0.0f; }
MHD_HD bool ge0(float x) { return x >= 0.0f; }
MHD_HD long long order_key(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffll); }
MHD_HD double tmin2(double a, double b) {
  const long long x = dbits(a), y = dbits(b);
  const bool pick_a = is_nan(b) || (!is_nan(a) && order_key(x) <= order_key(y));
  return pick_a ? a : b;
}
MHD_HD double tmax2(double a, double b) {
  const long long x = dbits(a), y = dbits(b);
  const bool pick_a = is_nan(b) || (!is_nan(a) && order_key(x) >= order_key(y));
  return pick_a ? a : b;
}
MHD_HD float tmin2(float a, float b) { return fminf(a, b); }
MHD_HD float tmax2(float a, float b) { return fmaxf(a, b); }
// a < b with IEEE semantics (NaN unordered, -0 == +0): a double's pattern,
// with negative ones mapped to minus their magnitude, is a signed integer in
// the numeric order.
MHD_HD long long num_key(long long b) { return b < 0 ? -(b & 0x7fffffffffffffffll) : b; }
MHD_HD bool lt_ieee(double a, double b) {
  return !is_nan(a) && !is_nan(b) && num_key(dbits(a)) < num_key(dbits(b));
}
MHD_HD bool lt_ieee(float a, float b) { return a < b; }
// x != 0 (true for NaN, as the IEEE comparison)
MHD_HD bool nonzero(double x) { return (dbits(x) << 1) != 0; }
MHD_HD bool nonzero(float x) { return x != 0.0f; }
// |a| < t, IEEE (false when either is NaN)
MHD_HD bool abs_lt(double a, double t) {
  const long long x = dbits(a) & 0x7fffffffffffffffll, y = dbits(t);
  return x < y && y <= 0x7ff0000000000000ll;
}
MHD_HD bool abs_lt(float a, float t) { return fabsf(a) < t; }
// |a| >= |b|, FP64 by the leading 32 bits alone (equal ones count as greater)
MHD_HD bool mag_ge(double a, double b) {
  return ((uint32_t)(dbits(a) >> 32) & 0x7fffffffu) >= ((uint32_t)(dbits(b) >> 32) & 0x7fffffffu);
}
MHD_HD bool mag_ge(float a, float b) { return fabsf(a) >= fabsf(b); }
// max(x, 0) for the square-root discriminant (fmax(NaN, 0) = 0 as well)
MHD_HD double pos_part(double x) { return gt0(x) ? x : 0.0; }
MHD_HD float pos_part(float x) { return fmaxf(x, 0.0f); }

// Exact 2x and x/2 of a non-negative double (or +inf / NaN, which are kept)
// from its bit pattern: a power-of-two scaling moves the exponent field; a
// subnormal doubles by a shift, and halving into the subnormal range
// shifts the significand right with the dropped bit rounded to nearest even
// (the IEEE results of x + x and 0.5 * x, overflow to +inf included).
MHD_HD long long twice_bits(long long b) {
  const long long e = b >> 52;
  if (e == 0) return b << 1;
  if (e < 2046) return b + (1ll << 52);
  return e == 2047 ? b : 0x7ff0000000000000ll;
}
MHD_HD long long half_bits(long long b) {
  const long long e = b >> 52;
  if (e >= 2) return e == 2047 ? b : b - (1ll << 52);
  return (b >> 1) + ((b & 1) & ((b >> 1) & 1));
}

// -4x and x/2 with IEEE results; FP64 moves the exponent field on the
// integer pipe (twice_bits / half_bits, exact including subnormals and
// overflow).
MHD_HD double neg4(double x) {
  const long long b = dbits(x), sign = b & (long long)0x8000000000000000ull;
  return bits2d(twice_bits(twice_bits(b ^ sign)) | (sign ^ (long long)0x8000000000000000ull));
}
MHD_HD float neg4(float x) { return -4.0f * x; }
MHD_HD double half_of(double x) {
  const long long b = dbits(x), sign = b & (long long)0x8000000000000000ull;
  return bits2d(half_bits(b ^ sign) | sign);
}
MHD_HD float half_of(float x) { return 0.5f * x; }

// x * s for a sign factor s = +1 / -1 given by its sign bit (0, or the top
// bit of a 64-bit pattern): FP64 flips the sign bit of x on the integer pipe
// (the product by +-1 is exact, so the result is the same, NaN payloads
// aside); FP32 negates.
MHD_HD long long sign_bit_of(bool negative) {
  return negative ? (long long)0x8000000000000000ull : 0ll;
}
MHD_HD double sign_mul(double x, long long sbit) { return bits2d(dbits(x) ^ sbit); }

// Two FP32 values in one register pair.  The packed instructions (FFMA2 / FMUL2
// / FADD2) do two values' arithmetic in one issue slot, each rounded as the
// scalar instruction rounds it.
struct f2 {
  float2 v;
  MHD_HD f2() {}
  MHD_HD f2(float a) : v(make_float2(a, a)) {}
  MHD_HD f2(float a, float b) : v(make_float2(a, b)) {}
  MHD_HD explicit f2(float2 a) : v(a) {}
};
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
MHD_HD f2 fma_rn(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }
MHD_HD f2 mul_rn(f2 a, f2 b) { return f2(__fmul2_rn(a.v, b.v)); }
MHD_HD f2 operator+(f2 a, f2 b) { return f2(__fadd2_rn(a.v, b.v)); }
#else
MHD_HD f2 fma_rn(f2 a, f2 b, f2 c) { return f2(fmaf(a.v.x, b.v.x, c.v.x), fmaf(a.v.y, b.v.y, c.v.y)); }
MHD_HD f2 mul_rn(f2 a, f2 b) { return f2(mul_rn(a.v.x, b.v.x), mul_rn(a.v.y, b.v.y)); }
MHD_HD f2 operator+(f2 a, f2 b) { return f2(a.v.x + b.v.x, a.v.y + b.v.y); }
#endif
// (a - b is fma(b, -1, a): the product is exact, so it rounds once)
MHD_HD f2 operator-(f2 a, f2 b) { return fma_rn(b, f2(-1.0f), a); }
MHD_HD f2 tabs(f2 a) { return f2(fabsf(a.v.x), fabsf(a.v.y)); }
MHD_HD f2 rcp(f2 a) { return f2(rcp(a.v.x), rcp(a.v.y)); }

// x * (+1 or -1): sign_of(m) is the factor -1 where m holds.  FP64: the sign
// bit (sign_mul); FP32: a product.
MHD_HD long long sign_of(bool m, double) { return sign_bit_of(m); }
MHD_HD float sign_of(bool m, float) { return m ? -1.0f : 1.0f; }
MHD_HD float sign_mul(float x, float s) { return mul_rn(x, s); }

// Reciprocal and square root inside the Riemann solver.  FP32: the hardware
// approximations (one instruction each; subnormal operands count as zero).
MHD_HD double rcp_h(double x) { return rcp(x); }
MHD_HD double sqrt_h(double x) { return tsqrt(x); }
MHD_HD float rcp_h(float x) { return seed_rcp(x); }
MHD_HD float sqrt_h(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return sqrtf(x);
#endif
}

// Square root of the fast speed's discriminant.  FP32: subnormal ones count: a^2 is
// subnormal for speeds below 3e-10, and taking it as 0 gives speeds wrong by up
// to a factor of 1.4.  The same bits as sqrt_h for normal values (512^3, a step of
// two stages 25.0 ms, 24.8 with subnormals as 0).
MHD_HD double sqrt_disc(double x) { return tsqrt(x); }
MHD_HD float sqrt_disc(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return sqrtf(x);
#endif
}

// x / 2 + y: FP64 halves by half_of, FP32 in one fused multiply-add.
MHD_HD double half_plus(double x, double y, const Phys<double>& ph) { return add_f(half_of(x), y, ph); }
MHD_HD float half_plus(float x, float y, const Phys<float>&) { return fma_rn(0.5f, x, y); }

// Pressure floor.  FP64: plain comparison.  FP32: when the FP32 pressure is
// within the cancellation-dominated range (internal energy below 1e-3 of the
// total, or below the floor) p is recomputed in FP64 from the promoted
// conservative inputs and the floor decision is taken in FP64.
MHD_HD double pressure_floor(double p, const double u[kNV], double rho,
                                                 const Phys<double>& ph, unsigned& flags) {
  if (lt_ieee(p, ph.p_floor)) {
    flags |= kFloorP;
    return ph.p_floor;
  }
  return p;
}
MHD_HD float pressure_floor(float p, const float u[kNV], float rho,
                                                const Phys<float>& ph, unsigned& flags) {
  if (p < ph.p_floor || p < 1e-3f * ph.gm1 * u[kPRS]) {
    flags |= kPressF64;
    // (volatile, so that no part of the branch is evaluated for every cell: one
    // FP64 instruction holds the SM's FP64 unit for 16 clocks)
    double e;
#ifdef __CUDA_ARCH__
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(e) : "f"(u[kPRS]));
#else
    e = u[kPRS];
#endif
    const double r = rho;
    const double m2 = (double)u[kVX] * u[kVX] + (double)u[kVY] * u[kVY] + (double)u[kVZ] * u[kVZ];
    const double b2 = (double)u[kBX] * u[kBX] + (double)u[kBY] * u[kBY] + (double)u[kBZ] * u[kBZ];
    const double pd = ph.gm1_d * (e - 0.5 * m2 / r - 0.5 * b2);
    if (pd < ph.p_floor_d) {
      flags |= kFloorP;
      return ph.p_floor;
    }
    return (float)pd;
  }
  return p;
}

// Conservative -> primitive (step 2 of the stage).  Floors by replacement,
// density first, then pressure; activations are flagged.
template <class T>
MHD_HD void cons_to_prim(const T u[kNV], T v[kNV], const Phys<T>& ph, unsigned& flags) {
  T rho = u[kRHO];
  if (lt_ieee(rho, ph.rho_floor)) {
    rho = ph.rho_floor;
    flags |= kFloorRho;
  }
  const T ri = rcp(rho);
  const T vx = mul_f(u[kVX], ri, ph), vy = mul_f(u[kVY], ri, ph), vz = mul_f(u[kVZ], ri, ph);
  const T k2 = dot3_f(u[kVX], vx, u[kVY], vy, u[kVZ], vz, ph);
  const T b2 = dot3_f(u[kBX], u[kBX], u[kBY], u[kBY], u[kBZ], u[kBZ], ph);
  // gm1 (E - (k2 + b2) / 2)
  T p = mul_f(ph.gm1, half_plus(-b2, half_plus(-k2, u[kPRS], ph), ph), ph);
  p = pressure_floor(p, u, rho, ph, flags);
  v[kRHO] = rho;
  v[kVX] = vx;
  v[kVY] = vy;
  v[kVZ] = vz;
  v[kBX] = u[kBX];
  v[kBY] = u[kBY];
  v[kBZ] = u[kBZ];
  v[kPRS] = p;
  v[kPSI] = u[kPSI];
}

// Primitive -> conservative.
template <class T>
MHD_HD void prim_to_cons(const T v[kNV], T u[kNV], const Phys<T>& ph) {
  const T rho = v[kRHO];
  const T v2 = v[kVX] * v[kVX] + v[kVY] * v[kVY] + v[kVZ] * v[kVZ];
  const T b2 = v[kBX] * v[kBX] + v[kBY] * v[kBY] + v[kBZ] * v[kBZ];
  u[kRHO] = rho;
  u[kVX] = rho * v[kVX];
  u[kVY] = rho * v[kVY];
  u[kVZ] = rho * v[kVZ];
  u[kBX] = v[kBX];
  u[kBY] = v[kBY];
  u[kBZ] = v[kBZ];
  u[kPRS] = v[kPRS] * ph.gm1i + T(0.5) * rho * v2 + T(0.5) * b2;
  u[kPSI] = v[kPSI];
}

// Twice the fast magnetosonic speed squared from 1/rho, gamma p, |B|^2 and
// B_n^2: with g = gamma p / rho, a = g + |B|^2 / rho and c_an^2 = B_n^2 / rho,
// 2 c_f^2 = a + sqrt(a^2 - 4 g c_an^2).
template <class T>
MHD_HD T fast_speed2x(T rho_i, T gp, T b2, T bn2, const Phys<T>& ph) {
  const T g = mul_f(gp, rho_i, ph);
  const T a = fma_rn(b2, rho_i, g);
  const T x = neg4(mul_f(g, mul_f(bn2, rho_i, ph), ph));
  return add_f(a, sqrt_disc(pos_part(fma_rn(a, a, x))), ph);
}

// Fast magnetosonic speed (see fast_speed2x).
template <class T>
MHD_HD T fast_speed(T rho_i, T gp, T b2, T bn2, const Phys<T>& ph) {
  return sqrt_h(half_of(fast_speed2x(rho_i, gp, b2, bn2, ph)));
}

// max over active directions of |v_d| + c_f,d for one conservative cell.
template <class T>
MHD_HD T cell_max_speed(const T u[kNV], const Phys<T>& ph, int ndim, unsigned& flags) {
  T v[kNV];
  cons_to_prim(u, v, ph, flags);
  const T ri = rcp(v[kRHO]);
  const T gp = mul_rn(ph.gamma, v[kPRS]);
  const T b2 = dot3_f(v[kBX], v[kBX], v[kBY], v[kBY], v[kBZ], v[kBZ], ph);
  T lam = tabs(v[kVX]) + fast_speed(ri, gp, b2, mul_rn(v[kBX], v[kBX]), ph);
  if (ndim > 1)
    lam = nan_max(lam, tabs(v[kVY]) + fast_speed(ri, gp, b2, mul_rn(v[kBY], v[kBY]), ph));
  if (ndim > 2)
    lam = nan_max(lam, tabs(v[kVZ]) + fast_speed(ri, gp, b2, mul_rn(v[kBZ], v[kBZ]), ph));
  // NaN anywhere in the cell (psi included) makes the speed NaN, and so does an
  // overflow of a^2 (see fast_speed2x): the discriminant is then minus infinity or
  // NaN, which the positive part turns into a finite, wrong speed
  const T a = mul_rn(gp + b2, ri);
  if (is_nan(v[kPSI]) || is_nan(lam) || !(mul_rn(a, a) < T(INFINITY))) lam = T(NAN);
  return lam;
}

#ifdef __CUDACC__
// ph.one, ph.nzero, ph.gamma and ph.gm1im1 in registers of unknown value (see
// add_f): through shared memory, slot[4].  Every thread of the CTA calls it.
__device__ __forceinline__ void fp64_registers(Phys<double>& ph, double* slot) {
  if (threadIdx.x == 0) {
    slot[0] = 1.0;
    slot[1] = -0.0;
    slot[2] = ph.gamma;
    slot[3] = ph.gm1im1;
  }
  __syncthreads();
  const volatile double* v = slot;
  ph.one = v[0];
  ph.nzero = v[1];
  ph.gamma = v[2];
  ph.gm1im1 = v[3];
}
__device__ __forceinline__ void fp64_registers(Phys<float>&, double*) {}

// ---------------------------------------------------------------------------
// Maximum wave speed of a state (cell_max_speed over all cells): the
// last-stage epilogue and the wave-speed kernels.  FP32 evaluates every cell.
// FP64 works in two passes.  Pass 1 (the epilogue, or a kernel over a state)
// takes an FP32 estimate of each cell's speed from FP32 images of its
// conservative variables (integer-pipe truncation, error < 2^-23 each)
// computed on the FP32 pipe, and the maximum M of the reliable estimates goes
// to one word (FP32 bits, atomicMax).  Reliable means: every input is 0 or
// within 2^-100 <= |x| < 2^100, rho and p are at least twice their floors (no
// floor acts), the internal energy is at least 1/50 of E and each
// direction's discriminant a^2 - 4 g c_an^2 at least 1e-4 a^2 (bounded
// cancellation: the FP32 errors of E - kin - |B|^2/2 and of the discriminant,
// a few 2^-24 of E and of a^2, are amplified at most 50-fold and, through the
// square root, to at most ~3e-5 of c_f^2); the estimate's relative error is
// then below 1e-4 (largest seen on 8 M random states pushed to the guard
// edges: 3.3e-6).  Pass 2
// (speed_exact_kernel) evaluates the FP64 speed of every cell whose estimate
// reaches 0.999 M or is not reliable.  The cell holding the exact maximum
// Lambda has an estimate >= Lambda (1 - 1e-4) when reliable, and
// M <= Lambda (1 + 1e-4), so it is always evaluated: the result is the exact
// FP64 maximum (floors and NaNs included, which are never screened out).
// Pass 2's FP64 evaluation sits behind a warp-uniform branch, so warps
// without a candidate issue no FP64 work for it.

// FP32 image of a double on the integer pipe: sign, rebiased exponent, top 23
// mantissa bits.  Clears ok unless x is 0 or 2^-100 <= |x| < 2^100.
__device__ __forceinline__ float f32_image(double x, bool& ok) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned mag = hi & 0x7fffffffu;
  const bool zero = (mag | lo) == 0u;
  ok = ok && (zero || ((mag >> 20) - 923u) < 200u);
  const unsigned fb = (hi & 0x80000000u) | (((mag - (896u << 20)) << 3) | (lo >> 29));
  return zero ? 0.0f : __uint_as_float(fb);
}

// FP32 estimate of cell_max_speed for an FP64 conservative cell (see above).
struct SpeedEstimator {
  float gm1, gamma, rho2, p2;  // FP32 images of the physics constants
  __device__ explicit SpeedEstimator(const Phys<double>& ph) {
    bool ok = true;
    gm1 = f32_image(ph.gm1, ok);
    gamma = f32_image(ph.gamma, ok);
    rho2 = 2.0f * f32_image(ph.rho_floor, ok);
    p2 = 2.0f * f32_image(ph.p_floor, ok);
    if (!ok) rho2 = __int_as_float(0x7f800000);  // never reliable
  }
  __device__ __forceinline__ float operator()(const double u[kNV], int ndim, bool& ok) const {
    float f[kNV];
#pragma unroll
    for (int k = 0; k < kNV; ++k) f[k] = f32_image(u[k], ok);
    const float r = f[kRHO];
    ok = ok && r >= rho2;
    const float ri = __frcp_rn(r);
    const float v[3] = {f[kVX] * ri, f[kVY] * ri, f[kVZ] * ri};
    const float kin = 0.5f * (f[kVX] * v[0] + f[kVY] * v[1] + f[kVZ] * v[2]);
    const float b2 = f[kBX] * f[kBX] + f[kBY] * f[kBY] + f[kBZ] * f[kBZ];
    const float eint = f[kPRS] - kin - 0.5f * b2;
    ok = ok && eint >= 0.02f * f[kPRS];
    const float pr = gm1 * eint;
    ok = ok && pr >= p2;
    const float g = gamma * pr * ri;
    const float a = b2 * ri + g;
    float lam = 0.0f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (d < ndim) {
        const float bd = f[kBX + d];
        const float disc = a * a - 4.0f * g * (bd * bd * ri);
        ok = ok && disc >= 1e-4f * a * a;
        lam = fmaxf(lam, fabsf(v[d]) + sqrtf(0.5f * (a + sqrtf(fmaxf(disc, 0.0f)))));
      }
    }
    return lam;
  }
};

// Per-thread accumulator of the epilogue and the wave-speed kernels: the
// exact FP32 maximum, or (FP64) the maximum of the reliable estimates.
template <class T>
struct SpeedMax;

template <>
struct SpeedMax<float> {
  float lam = 0.0f;
  __device__ explicit SpeedMax(const Phys<float>&) {}
  __device__ __forceinline__ void update(const float u[kNV], bool valid, const Phys<float>& ph,
                                         int ndim, unsigned& flags) {
    if (valid) lam = nan_max(lam, cell_max_speed(u, ph, ndim, flags));
  }
  __device__ __forceinline__ double value() const { return (double)lam; }
  // one thread per CTA: the CTA's maximum m into the state's wave-speed word
  __device__ __forceinline__ static void publish(double m, unsigned long long* lam_bits,
                                                 unsigned int*) {
    unsigned long long bits = (unsigned long long)__double_as_longlong(m);
    if (is_nan(m)) bits = 0x7ff8000000000000ull;
    atomicMax(lam_bits, bits);
  }
};

template <>
struct SpeedMax<double> {
  float est = 0.0f;
  SpeedEstimator estimate;
  __device__ explicit SpeedMax(const Phys<double>& ph) : estimate(ph) {}
  __device__ __forceinline__ void update(const double u[kNV], bool valid, const Phys<double>&,
                                         int ndim, unsigned&) {
    bool ok = true;
    const float e = estimate(u, ndim, ok);
    if (valid && ok) est = fmaxf(est, e);
  }
  __device__ __forceinline__ double value() const { return (double)est; }
  // the CTA's maximum estimate (a non-negative FP32 value) into the estimate
  // word: non-negative floats order like their bit patterns
  __device__ __forceinline__ static void publish(double m, unsigned long long*,
                                                 unsigned int* est_bits) {
    atomicMax(est_bits, __float_as_uint((float)m));
  }
};
#endif

// Limited slope (van Leer 1977): 0 when the one-sided differences disagree in
// sign; minmod = smaller magnitude; MC = min(2|dm|, 2|dp|, |dm+dp|/2).  The kernels
// take half of it (half_slope_mc, half_slope_minmod) or it with a derivative code
// (limited_slope_c); the host tests compare with this one.
template <class T>
MHD_HD T limited_slope(T dm, T dp, int lim) {
  if (lim == kLimFlat || !(dm * dp > T(0))) return T(0);
  const T am = tabs(dm), ap = tabs(dp);
  T mag = tmin(am, ap);
  if (lim == kLimMC) mag = tmin(T(2) * mag, T(0.5) * tabs(dm + dp));
  return dm > T(0) ? mag : -mag;
}

// FP64 specialisation with the same result: the sign and zero tests, |.|,
// the magnitude comparisons (non-negative doubles order like their bit
// patterns), the doubling and halving of the MC limiter and the sign
// transfer run on the integer pipe; only |dm| + |dp| uses the (scarce) FP64
// pipe.  For equal signs |dm + dp| = |dm| + |dp| exactly, so the central
// slope is (|dm|+|dp|)/2.
template <>
MHD_HD double limited_slope<double>(double dm, double dp, int lim) {
  const long long a = dbits(dm), b = dbits(dp);
  const long long mask = 0x7fffffffffffffffll;
  const long long am = a & mask, bm = b & mask;
  if (lim == kLimFlat || (a ^ b) < 0 || am == 0 || bm == 0) return 0.0;
  long long mb = am < bm ? am : bm;
  if (lim == kLimMC) {
    const long long two = twice_bits(mb);
    const long long cen = half_bits(dbits(bits2d(am) + bits2d(bm)));
    mb = cen < two ? cen : two;
  }
  return bits2d(mb | (a & ~mask));
}

// Half the limited slope, the step from the cell value to its faces: MC
// min(|dm|, |dp|, |dm+dp|/4), minmod min(|dm|, |dp|)/2, with the common sign, 0
// when the signs differ.  FP32: with the central value c between dm and dp, the
// smallest of the three where it is positive, the largest where it is negative
// (a NaN among them passes through these and the comparison with 0 drops it: 0).
MHD_HD float min3(float a, float b, float c) {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
  float d;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
#else
  return a != a || b != b || c != c ? a + b + c : fminf(fminf(a, b), c);
#endif
}
MHD_HD float max3(float a, float b, float c) {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
#else
  return a != a || b != b || c != c ? a + b + c : fmaxf(fmaxf(a, b), c);
#endif
}
MHD_HD float half_slope_mc(float dm, float dp, const Phys<float>&) {
  const float c = mul_rn(0.25f, dm + dp);
  return fmaxf(min3(dm, dp, c), 0.0f) + fminf(max3(dm, dp, c), 0.0f);
}
MHD_HD float half_slope_minmod(float dm, float dp) {
  return mul_rn(0.5f, fmaxf(min3(dm, dp, dp), 0.0f) + fminf(max3(dm, dp, dp), 0.0f));
}
// FP64: decided and scaled on the integer pipe; |dm| + |dp| is the only FP64
// operation.  (A NaN difference orders above infinity there: the slope is then the
// other difference's.)
MHD_HD double half_slope_mc(double dm, double dp, const Phys<double>& ph) {
  const long long a = dbits(dm), b = dbits(dp);
  const long long mask = 0x7fffffffffffffffll;
  const long long am = a & mask, bm = b & mask;
  const long long mb = am < bm ? am : bm;
  const long long qr = half_bits(half_bits(dbits(add_f(bits2d(am), bits2d(bm), ph))));
  const long long h = (qr < mb ? qr : mb) | (a & ~mask);
  return (a ^ b) < 0 || am == 0 || bm == 0 ? 0.0 : bits2d(h);
}
MHD_HD double half_slope_minmod(double dm, double dp) {
  const long long a = dbits(dm), b = dbits(dp);
  const long long mask = 0x7fffffffffffffffll;
  const long long am = a & mask, bm = b & mask;
  const long long h = half_bits(am < bm ? am : bm) | (a & ~mask);
  return (a ^ b) < 0 || am == 0 || bm == 0 ? 0.0 : bits2d(h);
}

// Picks component (dir + j) % 3 of a 3-vector given as scalars (dir is a
// compile-time constant in the flux kernels, so this folds away).
template <class T>
MHD_HD T rot3(int dir, int j, T a, T b, T c) {
  const int m = (dir + j) % 3;
  return m == 0 ? a : (m == 1 ? b : c);
}

// GLM interface step + HLLD along direction dir (0, 1, 2; template
// argument) for primitive face states vl, vr.  ch: cleaning speed;
// half_chi = 0.5 / ch.  F in conservative ordering.  Every sum of products
// is written with mul_rn / fma_rn / dot3_rn, so the flux rounds the same in
// every kernel and at every call site it is inlined into (the results of
// decomposed and undecomposed runs must agree bit for bit).
// FP64 is bound by the SM's FP64 unit, so the solver is arranged for few FP64
// operations: about 96 per face, 131 where a lane of the warp is inside the
// Alfven fan (the form that builds both sides' star and double-star states and
// adds up the wave jumps took about 280 with CUDA's divisions and roots).
// Orszag-Tang 256^3 FP64: 76.4 -> 47.4 ms per step (45.0 with what came after), of
// which the fixed-point reciprocals and roots 11.  Against a quadruple-precision
// evaluation its error is at most that of the longer form (2e-16 to 3e-15 rms of
// the flux, random, smooth, Mach-20, low- and high-beta and degenerate face states;
// for density contrasts see du below).
template <int dir, class T>
MHD_HD void glm_hlld_flux(const T vl[kNV], const T vr[kNV], T ch, T half_chi,
                          const Phys<T>& ph, T F[kNV]) {
  auto add = [&](T a, T b) { return add_f(a, b, ph); };
  auto sub = [&](T a, T b) { return sub_f(a, b, ph); };
  auto mul = [&](T a, T b) { return mul_f(a, b, ph); };
  // rotate: u normal, (v, w) tangential in cyclic order; by, bz likewise
  const T uL = rot3(dir, 0, vl[kVX], vl[kVY], vl[kVZ]);
  const T vL = rot3(dir, 1, vl[kVX], vl[kVY], vl[kVZ]);
  const T wL = rot3(dir, 2, vl[kVX], vl[kVY], vl[kVZ]);
  const T bnL = rot3(dir, 0, vl[kBX], vl[kBY], vl[kBZ]);
  const T byL = rot3(dir, 1, vl[kBX], vl[kBY], vl[kBZ]);
  const T bzL = rot3(dir, 2, vl[kBX], vl[kBY], vl[kBZ]);
  const T uR = rot3(dir, 0, vr[kVX], vr[kVY], vr[kVZ]);
  const T vR = rot3(dir, 1, vr[kVX], vr[kVY], vr[kVZ]);
  const T wR = rot3(dir, 2, vr[kVX], vr[kVY], vr[kVZ]);
  const T bnR = rot3(dir, 0, vr[kBX], vr[kBY], vr[kBZ]);
  const T byR = rot3(dir, 1, vr[kBX], vr[kBY], vr[kBZ]);
  const T bzR = rot3(dir, 2, vr[kBX], vr[kBY], vr[kBZ]);
  const T rL = vl[kRHO], pL = vl[kPRS], rR = vr[kRHO], pR = vr[kPRS];

  // GLM: exact solution of the linear (B_n, psi) interface problem
  const T chi = half_chi + half_chi;  // 1 / c_h
  const T bx = half_of(fma_rn(-chi, sub(vr[kPSI], vl[kPSI]), add(bnL, bnR)));
  const T psis = half_of(fma_rn(-ch, sub(bnR, bnL), add(vl[kPSI], vr[kPSI])));
  const T bx2 = mul(bx, bx);
  const T nbx = -bx, nbx2 = -bx2;

  // total pressures; c_max, the larger fast speed: one square root of the
  // larger c_f^2 (sqrt is monotone)
  const T b2L = fma_rn(bzL, bzL, fma_rn(byL, byL, bx2));
  const T b2R = fma_rn(bzR, bzR, fma_rn(byR, byR, bx2));
  const T ptL = half_plus(b2L, pL, ph), ptR = half_plus(b2R, pR, ph);
  const T cf2L = fast_speed2x(rcp_h(rL), mul(ph.gamma, pL), b2L, bx2, ph);
  const T cf2R = fast_speed2x(rcp_h(rR), mul(ph.gamma, pR), b2R, bx2, ph);
  const T cmax = sqrt_h(half_of(tmax2(cf2L, cf2R)));

  // wave-speed estimates (MK05 Eq. 67) and contact speed (Eq. 38, written as the
  // velocity of the side h with the larger rho |S - u| plus a correction nh)
  const T SL = sub(tmin2(uL, uR), cmax);
  const T SR = add(tmax2(uL, uR), cmax);
  const T SuL = sub(SL, uL), SuR = sub(SR, uR);
  const T dL = mul(SuL, rL), dR = mul(SuR, rR);
  const bool hL = mag_ge(dL, dR);
  const T nh = mul(fma_rn(hL ? dR : dL, sub(uR, uL), sub(ptL, ptR)), rcp_h(sub(dR, dL)));
  const T SM0 = add(hL ? uL : uR, nh);

  // The upwind side a: L if (S_L > 0) or (S_R >= 0 and S_M >= 0), else R
  // (sign tests on the integer pipe in FP64: gt0 / lt0 / ge0); o: the other
  // side, which enters only through the double-star states.  Where the flow is
  // supersonic the interface takes side a's outer state: S_M = u there makes
  // the star state below the outer one (rho and E are selected: their
  // quotients round).
  const bool sup = gt0(SL) || lt0(SR);
  const bool useL = gt0(SL) || (!lt0(SR) && ge0(SM0));
  const T r = useL ? rL : rR, u = useL ? uL : uR;
  const T v = useL ? vL : vR, w = useL ? wL : wR;
  const T by = useL ? byL : byR, bz = useL ? bzL : bzR;
  const T p = useL ? pL : pR, pt = useL ? ptL : ptR;
  const T S = useL ? SL : SR, Su = useL ? SuL : SuR, d = useL ? dL : dR;
  const T SM = sup ? u : SM0;

  // single-star state of side a (MK05 Eqs. 43-48), degenerate (v*, B* equal to
  // the outer state) when |den| < 1e-8 p_t*, den = rho (S-u)(S-S_M) - Bx^2;
  // p_t* = p_t + rho (S-u)(S_M-u), B* = B (1 + rho (S-u)(S_M-u) / den); one
  // reciprocal for the two divisors.  S_M - u of side h is nh itself: the rounding of
  // S_M times its rho (S-u) can exceed p_t* by the ratio of the two sides' densities
  // (as S_M - u_L + u_L - u: momentum flux wrong by 5 % in FP32 at 10^6)
  const T du = useL == hL && !sup ? nh : sub(SM, u);
  const T pts = fma_rn(d, du, pt);
  const T sm = sub(S, SM);
  const T den = fma_rn(d, sm, nbx2);
  const T thr = mul(T(1e-8), pts);
  const bool deg = abs_lt(den, thr);
  const T dn = deg ? T(1) : den;
  const T q = rcp_h(mul(sm, dn));
  const T smi = mul(dn, q);
  const T rs = sup ? r : mul(d, smi);
  const T k0 = deg ? T(0) : mul(du, mul(sm, q));
  const T fv = mul(nbx, k0), fb = mul(d, k0);
  const T vs = fma_rn(by, fv, v), ws = fma_rn(bz, fv, w);
  const T bys = fma_rn(by, fb, by), bzs = fma_rn(bz, fb, bz);
  const T vb = dot3_f(u, bx, v, by, w, bz, ph);
  const T vbs = dot3_f(SM, bx, vs, bys, ws, bzs, ph);
  // E = rho v^2 / 2 + p / (gamma-1) + B^2 / 2, the last two from p_t; E* (S-S_M)
  // = (S-u) E + (p_t* S_M - p_t u) + Bx (v.B - v*.B*).  (rho / 2 by half_of: an
  // exponent move in FP64, the same value as 0.5 * rho)
  const T e = fma_rn(half_of(r), dot3_f(u, u, v, v, w, w, ph), fma_rn(p, ph.gm1im1, pt));
  const T ns = fma_rn(bx, sub(vb, vbs), fma_rn(Su, e, mul(du, fma_rn(d, SM, pt))));
  const T es = sup ? e : mul(ns, smi);

  // Inside the Alfven fan (S*_L <= 0 <= S*_R, Eq. 51: rho* S_M^2 <= B_x^2) the
  // double-star states (Eqs. 59-63).  With s = sign(B_x) on side L and
  // -sign(B_x) on side R, Eqs. 59-62 are a step X from the single-star state
  // of side a: v** = v* + X, B** = B* + s sqrt(rho*) X, X = (sqrt(rho*_o)
  // (v*_o - v*) + s (B*_o - B*)) / (sqrt(rho*) + sqrt(rho*_o)).  Skipped where
  // no lane of the warp is inside the fan.
  const T ru = mul(rs, SM);
  T vF = vs, wF = ws, byF = bys, bzF = bzs, eF = es, vbF = vbs;
  if (!sup && !lt_ieee(bx2, mul(ru, SM))) {
    const T uo = useL ? uR : uL, vo = useL ? vR : vL, wo = useL ? wR : wL;
    const T byo = useL ? byR : byL, bzo = useL ? bzR : bzL;
    const T So = useL ? SR : SL, dO = useL ? dR : dL;
    const T smo = sub(So, SM);
    const T deno = fma_rn(dO, smo, nbx2);
    const bool dego = abs_lt(deno, thr);
    const T dno = dego ? T(1) : deno;
    const T qo = rcp_h(mul(smo, dno));
    const T rso = mul(dO, mul(dno, qo));
    const T k0o = dego ? T(0) : mul(sub(SM, uo), mul(smo, qo));
    const T fvo = mul(nbx, k0o), fbo = mul(dO, k0o);
    const T vso = fma_rn(byo, fvo, vo), wso = fma_rn(bzo, fvo, wo);
    const T byso = fma_rn(byo, fbo, byo), bzso = fma_rn(bzo, fbo, bzo);
    const T sqa = sqrt_h(rs), sqo = sqrt_h(rso);
    const T isum = rcp_h(add(sqa, sqo));
    const auto sg = sign_of(ge0(bx) != useL, T(0));
    const T Xv = mul(fma_rn(sqo, sub(vso, vs), sign_mul(sub(byso, bys), sg)), isum);
    const T Xw = mul(fma_rn(sqo, sub(wso, ws), sign_mul(sub(bzso, bzs), sg)), isum);
    const T sqs = sign_mul(sqa, sg);
    vF = add(vs, Xv);
    wF = add(ws, Xw);
    byF = fma_rn(sqs, Xv, bys);
    bzF = fma_rn(sqs, Xw, bzs);
    vbF = dot3_f(SM, bx, vF, byF, wF, bzF, ph);
    eF = fma_rn(sqs, sub(vbF, vbs), es);
  }

  // HLLD's fan fluxes F_a + S_a (U*_a - U_a) + S*_a (U**_a - U*_a) (Eqs.
  // 64-66) are, by the jump relations that define the star states, the physical
  // flux of the state on the interface with normal velocity S_M and total
  // pressure p_t* -- except the induction terms of a degenerate star state,
  // which keeps B* = B: there B (u - S_M) is left over.
  const T f1 = fma_rn(ru, SM, add(pts, nbx2));
  const T f2 = fma_rn(ru, vF, mul(nbx, byF));
  const T f3 = fma_rn(ru, wF, mul(nbx, bzF));
  T f4 = fma_rn(byF, SM, mul(nbx, vF));
  T f5 = fma_rn(bzF, SM, mul(nbx, wF));
  if (deg) {
    f4 = fma_rn(-by, du, f4);
    f5 = fma_rn(-bz, du, f5);
  }

  F[kRHO] = ru;
  F[kPRS] = fma_rn(add(eF, pts), SM, mul(nbx, vbF));
  F[kPSI] = mul(ch, mul(ch, bx));
  // un-rotate: component m of a vector gets rotated slot j = (m - dir) mod 3
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const int j = (m - dir + 3) % 3;
    F[kVX + m] = j == 0 ? f1 : (j == 1 ? f2 : f3);
    F[kBX + m] = j == 0 ? psis : (j == 1 ? f4 : f5);
  }
}

}  // namespace mhd

namespace mhd {
// Runtime-direction entry (batched unit kernel): dispatches to the
// compile-time direction.
template <class T>
MHD_HD void glm_hlld_flux_dir(const T vl[kNV], const T vr[kNV], int dir, T ch, T half_chi,
                              const Phys<T>& ph, T F[kNV]) {
  if (dir == 0)
    glm_hlld_flux<0>(vl, vr, ch, half_chi, ph, F);
  else if (dir == 1)
    glm_hlld_flux<1>(vl, vr, ch, half_chi, ph, F);
  else
    glm_hlld_flux<2>(vl, vr, ch, half_chi, ph, F);
}
}  // namespace mhd
