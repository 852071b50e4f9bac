// WENO-Z face values (Borges, Carmona, Costa & Don 2008; candidate stencils and
// smoothness indicators of Jiang & Shu 1996) of one cell, shared by the stage
// kernels with WENO-Z reconstruction.
#pragma once

#include "mhd_physics.cuh"

namespace mhd {

// epsilon of the WENO-Z weights (FP32 uses a larger one so that tau / e_k
// below stays finite).  FP64's form below holds while |primitive| < ~1e25
// (the product of both faces' denominators, ~beta^6, stays finite).
template <class T> struct WenoEps;
template <> struct WenoEps<double> { static constexpr double v = 1e-40; };
template <> struct WenoEps<float> { static constexpr float v = 1e-18f; };

// WENO-Z values of one variable at the cell's faces i-1/2 (minus) and i+1/2
// (plus) from f[0..4] = cells i-2 .. i+2.  With the second differences a_k
// and the one-sided first-difference combinations g_k of the three candidate
// stencils:
//   * 12 x (candidate value - cell value) is a_k +- 3 g_k (the plus face takes
//     a0+3g0, a1+3g1, a2-3g2; the minus face, whose stencils are the mirrored
//     ones, a2+3g2, a1-3g1, a0-3g0, with g1 = d1 + d2);
//   * the Jiang-Shu smoothness indicator is beta_k = (13/3 a_k^2 + g_k^2) / 4;
//     the weights are invariant under a common scale of beta, tau and epsilon,
//     so FP64 works with 4 beta and 4 epsilon;
//   * the smoothness indicators are shared by both faces (the reversed
//     stencils' are the same three in reverse order), and so is tau;
//   * the normalised weights w_k = d_k (1 + tau / e_k) / sum_j (...),
//     e_k = beta_k + eps, ideal weights (1, 6, 3)/10 (plus face; reversed on
//     the minus face).
// FP64 multiplies the unnormalised weights by e0 e1 e2 (no reciprocal per
// stencil): P_k = e0 e1 e2 + tau prod_{j != k} e_j, and one reciprocal of the
// product of the two faces' denominators serves both faces: 51 FP64 operations
// (61 from scaled second and first differences formed separately: one SSP-RK3
// step of a 256^3 box 277 -> 223 ms; with the register operands of add_f 205,
// on 32 x 8 tiles 189).  In FP32 these
// products of epsilons underflow (a uniform variable has beta = 0), so FP32
// takes the reciprocals 1 / e_k and one per face, with D_k = a_k / 12 and
// G_k = g_k / 4.
// Constants of the FP64 form; the kernel holds them in registers (see add_f).
template <class T>
struct WenoConst {
  __device__ explicit WenoConst(const double*) {}
};
template <>
struct WenoConst<double> {
  double three, c, eps, i12;
  __device__ explicit WenoConst(const volatile double* v)
      : three(v[0]), c(v[1]), eps(v[2]), i12(v[3]) {}
  __device__ static void fill(double* v) {
    v[0] = 3.0;
    v[1] = 13.0 / 3.0;
    v[2] = 4.0 * WenoEps<double>::v;
    v[3] = 1.0 / 12.0;
  }
};
__device__ __forceinline__ void wenoz_pair(const double f[5], const Phys<double>& ph,
                                           const WenoConst<double>& w, double& minus,
                                           double& plus) {
  auto add = [&](double a, double b) { return add_f(a, b, ph); };
  auto sub = [&](double a, double b) { return sub_f(a, b, ph); };
  auto mul = [&](double a, double b) { return mul_f(a, b, ph); };
  const double d0 = sub(f[1], f[0]), d1 = sub(f[2], f[1]), d2 = sub(f[3], f[2]);
  const double d3 = sub(f[4], f[3]);
  const double a0 = sub(d1, d0), a1 = sub(d2, d1), a2 = sub(d3, d2);
  const double g0 = fma(w.three, d1, -d0), g1 = add(d1, d2), g2 = fma(w.three, -d2, d3);
  const double e0 = fma(g0, g0, fma(mul(w.c, a0), a0, w.eps));
  const double e1 = fma(g1, g1, fma(mul(w.c, a1), a1, w.eps));
  const double e2 = fma(g2, g2, fma(mul(w.c, a2), a2, w.eps));
  const double tau = tabs(sub(e0, e2));
  const double E0 = mul(e1, e2), E2 = mul(e0, e1);
  const double pi = mul(e0, E0);
  // P0, 2 P1, P2: the ideal weights are 1, 3 x 2, 3
  const double P0 = fma(tau, E0, pi), P2 = fma(tau, E2, pi);
  const double P1 = bits2d(twice_bits(dbits(fma(tau, mul(e0, e2), pi))));
  const double den_p = fma(w.three, add(P1, P2), P0), den_m = fma(w.three, add(P1, P0), P2);
  const double num_p = fma(w.three, fma(P1, fma(w.three, g1, a1), mul(P2, fma(-w.three, g2, a2))),
                           mul(P0, fma(w.three, g0, a0)));
  const double num_m = fma(w.three, fma(P1, fma(-w.three, g1, a1), mul(P0, fma(-w.three, g0, a0))),
                           mul(P2, fma(w.three, g2, a2)));
  const double r = mul(rcp(mul(den_p, den_m)), w.i12);
  plus = fma(num_p, mul(den_m, r), f[2]);
  minus = fma(num_m, mul(den_p, r), f[2]);
}

// FP32: two variables at once, the same steps with every operation written out.
__device__ __forceinline__ void wenoz_pair(const f2 f[5], f2& minus, f2& plus) {
  using V = f2;
  const V C12(1.0f / 12.0f), Q4(0.25f), C39(39.0f), M2(-2.0f), M4(-4.0f), T3(3.0f), ONE(1.0f);
  const V D0 = mul_rn(C12, fma_rn(M2, f[1], f[0] + f[2]));
  const V D1 = mul_rn(C12, fma_rn(M2, f[2], f[1] + f[3]));
  const V D2 = mul_rn(C12, fma_rn(M2, f[3], f[2] + f[4]));
  const V G0 = mul_rn(Q4, fma_rn(T3, f[2], fma_rn(M4, f[1], f[0])));
  const V G1 = mul_rn(Q4, f[1] - f[3]);
  const V G2 = mul_rn(Q4, fma_rn(M4, f[3], mul_rn(T3, f[2])) + f[4]);
  const V b0 = fma_rn(G0, G0, mul_rn(mul_rn(C39, D0), D0));
  const V b1 = fma_rn(G1, G1, mul_rn(mul_rn(C39, D1), D1));
  const V b2 = fma_rn(G2, G2, mul_rn(mul_rn(C39, D2), D2));
  const V EPS(0.25f * WenoEps<float>::v);
  const V tau = tabs(b0 - b2);
  const V P0 = fma_rn(tau, rcp(b0 + EPS), ONE);
  const V P1 = fma_rn(tau, rcp(b1 + EPS), ONE);
  const V P2 = fma_rn(tau, rcp(b2 + EPS), ONE);
  const V S1 = mul_rn(V(6.0f), P1), T0 = mul_rn(T3, P0), T2 = mul_rn(T3, P2);
  const V den_p = P0 + S1 + T2, den_m = P2 + S1 + T0;
  const V num_p = fma_rn(T2, D2 - G2, fma_rn(S1, D1 - G1, mul_rn(P0, D0 + G0)));
  const V num_m = fma_rn(T0, D0 - G0, fma_rn(S1, D1 + G1, mul_rn(P2, D2 + G2)));
  plus = fma_rn(num_p, rcp(den_p), f[2]);
  minus = fma_rn(num_m, rcp(den_m), f[2]);
}
}  // namespace mhd
