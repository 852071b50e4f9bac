// Reverse-mode derivatives (vector-Jacobian products) of the pointwise
// pieces of the stage: the GLM + HLLD interface flux, the limited PLM slope
// and the conservative->primitive map.  Written by hand, statement by
// statement in reverse order of the forward code in mhd_physics.cuh, with
// the same branch decisions (HLLD fan region, degenerate star state, limiter
// selection, positivity fallback), which are piecewise constant and carry no
// derivative.  dt and c_h are frozen constants.
#pragma once

#include "mhd_physics.cuh"

namespace mhd {

// Vector-Jacobian product of glm_hlld_flux: given the flux adjoint Fb (9,
// conservative ordering) returns the adjoints of the primitive face states
// vlb, vrb (9 each, overwritten).  The forward statements are glm_hlld_flux's
// (side a: upwind, o: the other one; x_ is the adjoint of x); each block of the
// reverse follows the forward block it belongs to, last block first.  The other
// side's star state and everything of the double-star states run only where a
// lane of the warp is inside the Alfven fan, the fast speed's reverse only for
// the faster side, and the reciprocals and roots on the integer pipe: about
// 330 FP64 operations (430 inside the fan).  Reversing the longer form (both
// sides' star states, wave jumps added up) took about 700.
template <class T>
MHD_HD void glm_hlld_flux_vjp(const T vl[kNV], const T vr[kNV], int dir, T ch, T half_chi,
                              const Phys<T>& ph, const T Fb[kNV], T vlb[kNV], T vrb[kNV]) {
  const T half = T(0.5);
  const T uL = rot3(dir, 0, vl[kVX], vl[kVY], vl[kVZ]), uR = rot3(dir, 0, vr[kVX], vr[kVY], vr[kVZ]);
  const T vL = rot3(dir, 1, vl[kVX], vl[kVY], vl[kVZ]), vR = rot3(dir, 1, vr[kVX], vr[kVY], vr[kVZ]);
  const T wL = rot3(dir, 2, vl[kVX], vl[kVY], vl[kVZ]), wR = rot3(dir, 2, vr[kVX], vr[kVY], vr[kVZ]);
  const T bnL = rot3(dir, 0, vl[kBX], vl[kBY], vl[kBZ]), bnR = rot3(dir, 0, vr[kBX], vr[kBY], vr[kBZ]);
  const T byL = rot3(dir, 1, vl[kBX], vl[kBY], vl[kBZ]), byR = rot3(dir, 1, vr[kBX], vr[kBY], vr[kBZ]);
  const T bzL = rot3(dir, 2, vl[kBX], vl[kBY], vl[kBZ]), bzR = rot3(dir, 2, vr[kBX], vr[kBY], vr[kBZ]);
  const T rL = vl[kRHO], pL = vl[kPRS], rR = vr[kRHO], pR = vr[kPRS];

  // ---------------------------------------------------------- forward --
  const T bx = half * (bnL + bnR) - half_chi * (vr[kPSI] - vl[kPSI]);
  const T bx2 = bx * bx;
  const T b2L = bx2 + byL * byL + bzL * bzL, b2R = bx2 + byR * byR + bzR * bzR;
  const T ptL = pL + half * b2L, ptR = pR + half * b2R;
  const T riL = rcp(rL), riR = rcp(rR);
  T aL, aR, dscL, dscR;  // a and the discriminant of the fast speed
  {
    const T g = ph.gamma * pL * riL;
    aL = g + b2L * riL;
    dscL = pos_part(aL * aL + neg4(g * (bx2 * riL)));
  }
  {
    const T g = ph.gamma * pR * riR;
    aR = g + b2R * riR;
    dscR = pos_part(aR * aR + neg4(g * (bx2 * riR)));
  }
  const T sdL = tsqrt(dscL), sdR = tsqrt(dscR);
  const T c2L = aL + sdL, c2R = aR + sdR;  // 2 c_f^2
  // (comparisons on the integer pipe in FP64; ties pick the left side)
  const bool fastL = !lt_ieee(c2L, c2R);
  const T cmax = tsqrt(half_of(fastL ? c2L : c2R));
  const bool uL_min = !lt_ieee(uR, uL), uL_max = !lt_ieee(uL, uR);
  const T SL = (uL_min ? uL : uR) - cmax, SR = (uL_max ? uL : uR) + cmax;
  const T SuL = SL - uL, SuR = SR - uR;
  const T dL = SuL * rL, dR = SuR * rR;
  const T Di = rcp(dR - dL);
  const bool hL = mag_ge(dL, dR);
  const T nh = ((hL ? dR : dL) * (uR - uL) + (ptL - ptR)) * Di;
  const T SM0 = (hL ? uL : uR) + nh;

  const bool sup = gt0(SL) || lt0(SR);
  const bool useL = gt0(SL) || (!lt0(SR) && ge0(SM0));
  const T r = useL ? rL : rR, u = useL ? uL : uR, v = useL ? vL : vR, w = useL ? wL : wR;
  const T by = useL ? byL : byR, bz = useL ? bzL : bzR, p = useL ? pL : pR;
  const T pt = useL ? ptL : ptR, S = useL ? SL : SR, Su = useL ? SuL : SuR;
  const T d = useL ? dL : dR;
  const T SM = sup ? u : SM0;
  const T du = useL == hL && !sup ? nh : SM - u;
  const T pts = d * du + pt;
  const T sm = S - SM;
  const T den = d * sm - bx2;
  const T thr = T(1e-8) * pts;
  const bool deg = abs_lt(den, thr);
  const T dn = deg ? T(1) : den;
  const T q = rcp(sm * dn);
  const T smi = dn * q, deni = sm * q;
  const T rs = sup ? r : d * smi;
  const T k0 = deg ? T(0) : du * deni;
  const T fv = -(bx * k0), fb1 = d * k0 + T(1);
  const T vs = by * fv + v, ws = bz * fv + w;
  const T bys = by * fb1, bzs = bz * fb1;
  const T vb = u * bx + v * by + w * bz;
  const T vbs = SM * bx + vs * bys + ws * bzs;
  const T vv = u * u + v * v + w * w;
  const T e = half_of(r) * vv + (p * ph.gm1im1 + pt);
  const T hh = d * SM + pt;
  const T ns = bx * (vb - vbs) + (Su * e + du * hh);
  const T es = sup ? e : ns * smi;
  const T ru = rs * SM;
  const bool inner = !sup && !lt_ieee(bx2, ru * SM);

  // rotated flux adjoint: mass, momenta, induction, energy
  const T f0 = Fb[kRHO], f6 = Fb[kPRS];
  const T f1 = rot3(dir, 0, Fb[kVX], Fb[kVY], Fb[kVZ]);
  const T f2 = rot3(dir, 1, Fb[kVX], Fb[kVY], Fb[kVZ]);
  const T f3 = rot3(dir, 2, Fb[kVX], Fb[kVY], Fb[kVZ]);
  const T psis_ = rot3(dir, 0, Fb[kBX], Fb[kBY], Fb[kBZ]);
  const T f4 = rot3(dir, 1, Fb[kBX], Fb[kBY], Fb[kBZ]);
  const T f5 = rot3(dir, 2, Fb[kBX], Fb[kBY], Fb[kBZ]);

  // adjoints: shared ones, the star state of side a, the other side
  T bx_ = ch * ch * Fb[kPSI] - f6 * (sup ? vb : vbs);
  T bx2_ = -f1, SM_ = T(0);
  const T e_F = f6 * SM, vb_F = -(f6 * bx);
  T rs_, vs_, ws_, bys_, bzs_, es_ = e_F, vbs_;
  T uo_ = T(0), vo_ = T(0), wo_ = T(0), byo_ = T(0), bzo_ = T(0), So_ = T(0), do_ = T(0);
  if (!inner) {
    // the physical flux of the star (or outer) state
    const T ru_ = f0 + f1 * SM + f2 * vs + f3 * ws;
    rs_ = ru_ * SM;
    SM_ = ru_ * rs + f1 * ru + f4 * bys + f5 * bzs + f6 * (es + pts);
    vs_ = f2 * ru - f4 * bx;
    ws_ = f3 * ru - f5 * bx;
    bys_ = f4 * SM - f2 * bx;
    bzs_ = f5 * SM - f3 * bx;
    bx_ -= f2 * bys + f3 * bzs + f4 * vs + f5 * ws;
    vbs_ = vb_F;
  } else {
    const T uo = useL ? uR : uL, vo = useL ? vR : vL, wo = useL ? wR : wL;
    const T byo = useL ? byR : byL, bzo = useL ? bzR : bzL;
    const T So = useL ? SR : SL, dO = useL ? dR : dL;
    const T smo = So - SM;
    const T deno = dO * smo - bx2;
    const bool dego = abs_lt(deno, thr);
    const T dno = dego ? T(1) : deno;
    const T qo = rcp(smo * dno);
    const T smio = dno * qo, denio = smo * qo;
    const T rso = dO * smio;
    const T duo = SM - uo;
    const T k0o = dego ? T(0) : duo * denio;
    const T fvo = -(bx * k0o), fbo1 = dO * k0o + T(1);
    const T vso = byo * fvo + vo, wso = bzo * fvo + wo;
    const T byso = byo * fbo1, bzso = bzo * fbo1;
    const T sqa = tsqrt(rs), sqo = tsqrt(rso);
    const T isum = rcp(sqa + sqo);
    const auto sg = sign_of(ge0(bx) != useL, T(0));
    const T dv = vso - vs, dw = wso - ws;
    const T Xv = (sqo * dv + sign_mul(byso - bys, sg)) * isum;
    const T Xw = (sqo * dw + sign_mul(bzso - bzs, sg)) * isum;
    const T sqs = sign_mul(sqa, sg);
    const T vF = vs + Xv, wF = ws + Xw;
    const T byF = sqs * Xv + bys, bzF = sqs * Xw + bzs;
    const T vbF = SM * bx + vF * byF + wF * bzF;
    const T eF = sqs * (vbF - vbs) + es;
    // reverse: flux of the double-star state
    const T ru_ = f0 + f1 * SM + f2 * vF + f3 * wF;
    rs_ = ru_ * SM;
    SM_ = ru_ * rs + f1 * ru + f4 * byF + f5 * bzF + f6 * (eF + pts);
    bx_ += f6 * (vbs - vbF) - (f2 * byF + f3 * bzF + f4 * vF + f5 * wF);
    // eF = es + sqs (vbF - vbs); vbF = SM bx + vF byF + wF bzF
    const T es_sq = e_F * sqs;
    const T vbF_ = vb_F + es_sq;
    vbs_ = -es_sq;
    T sqs_ = e_F * (vbF - vbs);
    SM_ += vbF_ * bx;
    bx_ += vbF_ * SM;
    const T vF_ = f2 * ru - f4 * bx + vbF_ * byF, wF_ = f3 * ru - f5 * bx + vbF_ * bzF;
    const T byF_ = f4 * SM - f2 * bx + vbF_ * vF, bzF_ = f5 * SM - f3 * bx + vbF_ * wF;
    // v** = v* + X, B** = B* + sqs X
    sqs_ += byF_ * Xv + bzF_ * Xw;
    const T Xv_ = vF_ + byF_ * sqs, Xw_ = wF_ + bzF_ * sqs;
    // X = (sqo (v*_o - v*) + s (B*_o - B*)) / (sqa + sqo)
    const T Mv_ = Xv_ * isum, Mw_ = Xw_ * isum;
    const T sum_ = -(Mv_ * Xv + Mw_ * Xw);
    const T sqo_ = Mv_ * dv + Mw_ * dw + sum_;
    const T sqa_ = sum_ + sign_mul(sqs_, sg);
    const T vso_ = Mv_ * sqo, wso_ = Mw_ * sqo;
    const T byso_ = sign_mul(Mv_, sg), bzso_ = sign_mul(Mw_, sg);
    vs_ = vF_ - vso_;
    ws_ = wF_ - wso_;
    bys_ = byF_ - byso_;
    bzs_ = bzF_ - bzso_;
    // sq = sqrt(rho*)
    rs_ += sqa_ * half_of(rcp(sqa));
    const T rso_ = sqo_ * half_of(rcp(sqo));
    // star state of side o
    do_ = rso_ * smio;
    T smo_ = -(rso_ * rso * smio);
    vo_ = vso_;
    wo_ = wso_;
    byo_ = vso_ * fvo + byso_ * fbo1;
    bzo_ = wso_ * fvo + bzso_ * fbo1;
    const T fvo_ = vso_ * byo + wso_ * bzo, fbo_ = byso_ * byo + bzso_ * bzo;
    bx_ -= fvo_ * k0o;
    do_ += fbo_ * k0o;
    const T k0o_ = dego ? T(0) : fbo_ * dO - fvo_ * bx;
    const T duo_ = k0o_ * denio;
    const T deno_ = -(duo_ * k0o);
    do_ += deno_ * smo;
    smo_ += deno_ * dO;
    bx2_ -= deno_;
    SM_ += duo_ - smo_;
    uo_ = -duo_;
    So_ = smo_;
  }

  // side a.  Supersonic: the interface state is the outer state (S_M = u, v* = v
  // ...), so its adjoints are the outer state's own.
  T pt_ = f1 + f6 * SM;  // of p_t*
  T r_ = T(0), u_ = T(0), v_ = vs_, w_ = ws_, by_, bz_, e_, vb_, d_ = T(0), S_ = T(0), Su_ = T(0);
  if (sup) {
    r_ = rs_;
    u_ = SM_;
    SM_ = T(0);
    by_ = bys_;
    bz_ = bzs_;
    e_ = es_;
    vb_ = vbs_;
  } else {
    // E* = ns / (S - S_M), ns = bx (vb - vbs) + Su e + du (pt + d SM)
    const T ns_ = es_ * smi;
    const T nbx = ns_ * bx;
    bx_ += ns_ * (vb - vbs);
    vb_ = nbx;
    vbs_ -= nbx;
    Su_ = ns_ * e;
    e_ = ns_ * Su;
    const T hh_ = ns_ * du;
    T du_ = ns_ * hh + pt_ * d;
    d_ = hh_ * SM + pt_ * du;  // (with p_t* = pt + d du)
    pt_ += hh_;
    SM_ += hh_ * d;
    // vbs = SM bx + vs bys + ws bzs
    SM_ += vbs_ * bx;
    bx_ += vbs_ * SM;
    vs_ += vbs_ * bys;
    ws_ += vbs_ * bzs;
    bys_ += vbs_ * vs;
    bzs_ += vbs_ * ws;
    // v* = v + by fv, B* = by fb1, fv = -bx k0, fb1 = 1 + d k0, k0 = du / den
    v_ = vs_;
    w_ = ws_;
    by_ = vs_ * fv + bys_ * fb1;
    bz_ = ws_ * fv + bzs_ * fb1;
    const T fv_ = vs_ * by + ws_ * bz, fb_ = bys_ * by + bzs_ * bz;
    bx_ -= fv_ * k0;
    d_ += fb_ * k0;
    const T k0_ = deg ? T(0) : fb_ * d - fv_ * bx;
    const T dk = k0_ * deni;
    du_ += dk;
    const T den_ = -(dk * k0);
    // rho* = d / (S - S_M) and E*'s divisor
    const T smi_ = es_ * ns + rs_ * d;
    d_ += rs_ * smi + den_ * sm;
    const T sm_ = den_ * d - smi_ * (smi * smi);
    bx2_ -= den_;
    if (deg) {  // the degenerate star state's induction terms, -B du
      by_ -= f4 * du;
      bz_ -= f5 * du;
      du_ -= f4 * by + f5 * bz;
    }
    SM_ += du_ - sm_;
    u_ = -du_;
    S_ = sm_;
  }
  // vb = u bx + v by + w bz; e = r vv / 2 + p gm1im1 + pt
  u_ += vb_ * bx;
  bx_ += vb_ * u;
  v_ += vb_ * by;
  by_ += vb_ * v;
  w_ += vb_ * bz;
  bz_ += vb_ * w;
  const T er = e_ * r;
  r_ += e_ * half_of(vv);
  u_ += er * u;
  v_ += er * v;
  w_ += er * w;
  const T p_ = e_ * ph.gm1im1;
  pt_ += e_;

  // sides a, o -> L, R
  T rL_ = useL ? r_ : T(0), rR_ = useL ? T(0) : r_;
  T uL_ = useL ? u_ : uo_, uR_ = useL ? uo_ : u_;
  T pL_ = useL ? p_ : T(0), pR_ = useL ? T(0) : p_;
  T ptL_ = useL ? pt_ : T(0), ptR_ = useL ? T(0) : pt_;
  T byL_ = useL ? by_ : byo_, byR_ = useL ? byo_ : by_;
  T bzL_ = useL ? bz_ : bzo_, bzR_ = useL ? bzo_ : bz_;
  T dL_ = useL ? d_ : do_, dR_ = useL ? do_ : d_;
  T SL_ = useL ? S_ : So_, SR_ = useL ? So_ : S_;
  T SuL_ = useL ? Su_ : T(0), SuR_ = useL ? T(0) : Su_;
  // S_M = (d_R u_R - d_L u_L + pt_L - pt_R) / (d_R - d_L); S_M - u_L and u_R - S_M from nh
  {
    const T n_ = SM_ * Di;
    const T dw = uR - uL;
    uL_ -= n_ * dL;
    uR_ += n_ * dR;
    dR_ += n_ * (hL ? dw - nh : -nh);
    dL_ += n_ * (hL ? nh : dw + nh);
    ptL_ += n_;
    ptR_ -= n_;
  }
  // d = Su r, Su = S - u
  SuL_ += dL_ * rL;
  rL_ += dL_ * SuL;
  SuR_ += dR_ * rR;
  rR_ += dR_ * SuR;
  SL_ += SuL_;
  uL_ -= SuL_;
  SR_ += SuR_;
  uR_ -= SuR_;
  // S_L = min(u) - c, S_R = max(u) + c
  const T c_ = SR_ - SL_;
  uL_ += (uL_min ? SL_ : T(0)) + (uL_max ? SR_ : T(0));
  uR_ += (uL_min ? T(0) : SL_) + (uL_max ? T(0) : SR_);
  // c = sqrt(c2 / 2), c2 = a + sd of the faster side m
  T b2L_ = half * ptL_, b2R_ = half * ptR_;
  {
    const T rim = fastL ? riL : riR, am = fastL ? aL : aR, sdm = fastL ? sdL : sdR;
    const T pm = fastL ? pL : pR, b2m = fastL ? b2L : b2R;
    const T gpm = ph.gamma * pm, xm = bx2 * rim, gm = gpm * rim;
    const T c2_ = c_ * (T(0.25) * rcp(cmax));
    // sd = sqrt(disc) (no derivative where the discriminant is clamped at 0)
    const T dsc_ = gt0(sdm) ? half_of(c2_) * rcp(sdm) : T(0);
    const T a_ = c2_ + T(2) * am * dsc_;
    const T d4 = neg4(dsc_);
    const T x_ = d4 * gm, g_ = d4 * xm + a_;
    const T ri_ = a_ * b2m + x_ * bx2 + g_ * gpm;
    const T pm_ = ph.gamma * (g_ * rim), b2m_ = a_ * rim, rm_ = -(ri_ * (rim * rim));
    bx2_ += x_ * rim;
    pL_ += fastL ? pm_ : T(0);
    pR_ += fastL ? T(0) : pm_;
    b2L_ += fastL ? b2m_ : T(0);
    b2R_ += fastL ? T(0) : b2m_;
    rL_ += fastL ? rm_ : T(0);
    rR_ += fastL ? T(0) : rm_;
  }
  // pt = p + b2 / 2, b2 = bx2 + by^2 + bz^2
  pL_ += ptL_;
  pR_ += ptR_;
  bx2_ += b2L_ + b2R_;
  byL_ += byL * (b2L_ + b2L_);
  bzL_ += bzL * (b2L_ + b2L_);
  byR_ += byR * (b2R_ + b2R_);
  bzR_ += bzR * (b2R_ + b2R_);
  // bx = (bnL + bnR)/2 - half_chi (psR - psL); psis = (psL + psR)/2 - ch (bnR - bnL)/2
  bx_ += (bx2_ + bx2_) * bx;
  const T hb = half * bx_, hp = half * psis_;
  const T cb = half_chi * bx_, cp = ch * hp;
  vlb[kPSI] = hp + cb;
  vrb[kPSI] = hp - cb;
  const T bnL_ = hb + cp, bnR_ = hb - cp;
  vlb[kRHO] = rL_;
  vrb[kRHO] = rR_;
  vlb[kPRS] = pL_;
  vrb[kPRS] = pR_;
  const T vL_ = useL ? v_ : vo_, vR_ = useL ? vo_ : v_;
  const T wL_ = useL ? w_ : wo_, wR_ = useL ? wo_ : w_;
  // un-rotate velocity and field adjoints: component m gets rotated slot (m - dir) mod 3
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const int j = (m - dir + 3) % 3;
    vlb[kVX + m] = j == 0 ? uL_ : (j == 1 ? vL_ : wL_);
    vrb[kVX + m] = j == 0 ? uR_ : (j == 1 ? vR_ : wR_);
    vlb[kBX + m] = j == 0 ? bnL_ : (j == 1 ? byL_ : bzL_);
    vrb[kBX + m] = j == 0 ? bnR_ : (j == 1 ? byR_ : bzR_);
  }
}

// Limited slope and its (piecewise constant) partial derivatives with
// respect to the one-sided differences dm, dp (what limited_slope_c encodes; for
// the host tests, as slope_code_d).
template <class T>
MHD_HD T limited_slope_d(T dm, T dp, int lim, T& ddm, T& ddp) {
  ddm = T(0);
  ddp = T(0);
  // the zero branch is decided exactly as in the forward limiter
  const T s = limited_slope(dm, dp, lim);
  if (s == T(0)) return s;
  const T am = tabs(dm), ap = tabs(dp);
  // minmod: the smaller magnitude (dm on ties, as min(a, b) picks a)
  const bool m_is_dm = !(ap < am);
  T gdm = m_is_dm ? T(1) : T(0), gdp = m_is_dm ? T(0) : T(1);
  if (lim == kLimMC) {
    const T two = T(2) * (m_is_dm ? am : ap);
    const T cen = T(0.5) * (am + ap);  // = |dm + dp| / 2 for equal signs
    if (cen < two) {  // central slope selected
      gdm = T(0.5);
      gdp = T(0.5);
    } else {
      gdm *= T(2);
      gdp *= T(2);
    }
  }
  // sign(s) = sign(dm) = sign(dp), so d s / d dm = gdm (signs cancel)
  ddm = gdm;
  ddp = gdp;
  return s;
}

// Derivative code of a limited slope, which is piecewise linear in the
// one-sided differences dm, dp: bits 0-1 the piece -- 0 zero slope, 1 the
// smaller-magnitude difference (minmod), 2 twice it (MC), 3 the central slope
// (dm + dp) / 2 (MC) -- and bit 2 set when the one-sided difference is dm.
// Three bits instead of two doubles keep the 18 derivatives of a face's two
// slopes in one register pair through the flux reverse.
MHD_HD void slope_code_d(unsigned code, double& ddm, double& ddp) {
  const unsigned piece = code & 3u;
  const bool m = (code >> 2) & 1u;
  const double f = piece == 1u ? 1.0 : 2.0;
  ddm = piece == 0u ? 0.0 : (piece == 3u ? 0.5 : (m ? f : 0.0));
  ddp = piece == 0u ? 0.0 : (piece == 3u ? 0.5 : (m ? 0.0 : f));
}

// Half of those derivatives (0 unless ok), and 1 + hm - hp (b = false: the cell
// below a face, v + s / 2) or 1 - hm + hp (b = true: above, v - s / 2): the
// multipliers of the face states' reverse, all 0, small powers of two or 3/2, so
// they are selected, not computed.
MHD_HD double hi_word(unsigned hi) { return bits2d((long long)((unsigned long long)hi << 32)); }
MHD_HD void slope_code_half(unsigned code, bool ok, bool b, double& hm, double& hp,
                            double& c1) {
  const unsigned piece = ok ? code & 3u : 0u;
  const bool m = (code >> 2) & 1u;
  const unsigned f = piece == 1u ? 0x3fe00000u : (piece == 2u ? 0x3ff00000u : 0u);  // 1/2, 1
  const unsigned c = piece == 3u ? 0x3fd00000u : 0u;                               // 1/4
  hm = hi_word(m ? f | c : c);
  hp = hi_word(m ? c : f | c);
  c1 = hi_word(piece == 1u ? (m != b ? 0x3ff80000u : 0x3fe00000u)
                           : (piece == 2u ? (m != b ? 0x40000000u : 0u) : 0x3ff00000u));
}

// FP64: the limited slope from the bit patterns, as limited_slope<double>,
// with its derivative code: the zero test, the minmod choice, the MC doubling
// / halving and the MC decision on the integer pipe; |dm| + |dp| is the only
// FP64 operation.
MHD_HD double limited_slope_c(double dm, double dp, int lim, unsigned& code) {
  code = 0u;
  const long long a = dbits(dm), b = dbits(dp);
  const long long mask = 0x7fffffffffffffffll;
  const long long am = a & mask, bm = b & mask;
  if (lim == kLimFlat || (a ^ b) < 0 || am == 0 || bm == 0) return 0.0;
  const bool m_is_dm = !(bm < am);  // the smaller magnitude; dm on ties
  long long mb = m_is_dm ? am : bm;
  unsigned piece = 1u;
  if (lim == kLimMC) {
    const long long two = twice_bits(mb);
    const long long cen = half_bits(dbits(bits2d(am) + bits2d(bm)));
    if (cen < two) {  // central slope selected
      mb = cen;
      piece = 3u;
    } else {
      mb = two;
      piece = 2u;
    }
  }
  code = piece | (m_is_dm ? 4u : 0u);
  return bits2d(mb | (a & ~mask));
}

template <>
MHD_HD double limited_slope_d<double>(double dm, double dp, int lim, double& ddm, double& ddp) {
  unsigned code;
  const double s = limited_slope_c(dm, dp, lim, code);
  slope_code_d(code, ddm, ddp);
  return s;
}

// Reverse of cons_to_prim (floors inactive: a floored value has zero
// derivative).  vb: adjoint of the primitives; ub: adjoint of the
// conservatives (overwritten).
template <class T>
MHD_HD void cons_to_prim_vjp(const T u[kNV], const T vb[kNV], const Phys<T>& ph,
                             T ub[kNV]) {
  const T rho = u[kRHO];
  const T ri = rcp(rho);
  const T vx = u[kVX] * ri, vy = u[kVY] * ri, vz = u[kVZ] * ri;
  const T kin = T(0.5) * (u[kVX] * vx + u[kVY] * vy + u[kVZ] * vz);
  const T b2 = u[kBX] * u[kBX] + u[kBY] * u[kBY] + u[kBZ] * u[kBZ];
  const T p = ph.gm1 * (u[kPRS] - kin - T(0.5) * b2);
  const bool rfl = lt_ieee(rho, ph.rho_floor);
  const bool pfl = lt_ieee(p, ph.p_floor);
  const T pb = pfl ? T(0) : vb[kPRS];
  // p = gm1 (E - |m|^2/(2 rho) - |B|^2/2)
  T rhob = rfl ? T(0) : vb[kRHO];
  rhob += pb * ph.gm1 * (vx * vx + vy * vy + vz * vz) * T(0.5);
  // v_k = m_k / rho
  rhob -= (vb[kVX] * vx + vb[kVY] * vy + vb[kVZ] * vz) * ri;
  ub[kRHO] = rfl ? T(0) : rhob;
  ub[kVX] = vb[kVX] * ri - pb * ph.gm1 * vx;
  ub[kVY] = vb[kVY] * ri - pb * ph.gm1 * vy;
  ub[kVZ] = vb[kVZ] * ri - pb * ph.gm1 * vz;
  ub[kBX] = vb[kBX] - pb * ph.gm1 * u[kBX];
  ub[kBY] = vb[kBY] - pb * ph.gm1 * u[kBY];
  ub[kBZ] = vb[kBZ] - pb * ph.gm1 * u[kBZ];
  ub[kPRS] = pb * ph.gm1;
  ub[kPSI] = vb[kPSI];
}

}  // namespace mhd
