// Hand-written reverse mode of the per-interface PPM flux (the adjoint of
// the hydro Method of Sec. II.C with dt held fixed).  Each *_bwd function
// recomputes what it needs of its forward counterpart in ppm.cuh and
// accumulates the adjoints of its inputs (+=).  At a kink (min, max, a
// branch) the derivative of the branch the forward pass took is used: every
// value that decides a branch is the forward expression, in its order.  What
// only scales an adjoint is written for GB300's float64 pipe, which bounds the
// float64 adjoint and takes ~10 instructions for a division: one reciprocal per
// divisor, fused multiply-adds.
#pragma once

#include <type_traits>

#include "ppm.cuh"
#include "ppm64.cuh"

namespace cello {

CELLO_HD float vfma(float a, float b, float c) { return fmaf(a, b, c); }
CELLO_HD double vfma(double a, double b, double c) { return fma(a, b, c); }

// Reciprocal of what only scales an adjoint.
CELLO_HD float inverse(float a) { return 1.0f / a; }
CELLO_HD double inverse(double a) { return q64::inverse(a); }

// W = to_primitive(U); rho = max(U_0, floor) and p = max(p of U, floor).
template <typename T>
CELLO_HD void to_primitive_bwd(const T W[5], const Gas<T>& gs, const T Wb[5], T Ub[5]) {
  const T rho = W[0], un = W[1], ut1 = W[2], ut2 = W[3];
  const T ir = inverse(rho);
  const T s = vfma(un, un, vfma(ut1, ut1, ut2 * ut2));
  const T prawb = (W[4] > T(kPFloor)) ? Wb[4] : T(0);
  const T keb = -gs.gm1 * prawb;
  Ub[4] -= keb;
  const T sb2 = keb * rho;   // twice the adjoint of s
  const T unb = vfma(un, sb2, Wb[1]), t1b = vfma(ut1, sb2, Wb[2]), t2b = vfma(ut2, sb2, Wb[3]);
  Ub[1] = vfma(unb, ir, Ub[1]);
  Ub[2] = vfma(t1b, ir, Ub[2]);
  Ub[3] = vfma(t2b, ir, Ub[3]);
  if (rho > T(kRhoFloor)) {
    const T rhob = vfma(T(0.5) * keb, s, Wb[0]);
    Ub[0] += vfma(-vfma(unb, un, vfma(t1b, ut1, t2b * ut2)), ir, rhob);
  }
}

// The slope is 1/2 (ap - am), 2 (a0 - am) or 2 (ap - a0), the smallest of the three,
// where the last two have one sign.
template <typename T>
CELLO_HD void limited_slope_bwd(T am, T a0, T ap, T ob, T& amb, T& a0b, T& apb) {
  const T dl = a0 - am, dr = ap - a0;
  bool centred, left;
  if (std::is_same<T, double>::value && q64::within<-500, 500>(q64::mag(dl)) &&
      q64::within<-500, 500>(q64::mag(dr))) {   // on their bits: see q64::slope
    if ((int)(q64::high(dl) ^ q64::high(dr)) < 0) return;
    constexpr long long kTwo = 0x0010000000000000ll;
    const long long l = q64::bits(q64::absval(dl)), r = q64::bits(q64::absval(dr));
    const long long d = q64::bits(q64::absval(ap - am)) - kTwo;
    centred = d < (l < r ? l : r) + kTwo;
    left = l < r;
  } else {
    if (!(dl * dr > T(0))) return;
    const T adl = T(2) * vabs(dl), adr = T(2) * vabs(dr);
    centred = vabs(T(0.5) * (ap - am)) < vmin(adl, adr);
    left = adl < adr;
  }
  if (centred) {
    apb = vfma(T(0.5), ob, apb);
    amb = vfma(T(-0.5), ob, amb);
  } else if (left) {
    a0b = vfma(T(2), ob, a0b);
    amb = vfma(T(-2), ob, amb);
  } else {
    apb = vfma(T(2), ob, apb);
    a0b = vfma(T(-2), ob, a0b);
  }
}

template <typename T>
CELLO_HD void interface_value_bwd(T ob, T& a0b, T& a1b, T& dm0b, T& dm1b) {
  a0b += T(0.5) * ob;
  a1b += T(0.5) * ob;
  dm1b -= ob * T(1.0 / 6.0);
  dm0b += ob * T(1.0 / 6.0);
}

template <typename T>
CELLO_HD void flatten_tilde_bwd(T pm2, T pm1, T pp1, T pp2, T um1, T up1, T ob, T& pm2b, T& pm1b, T& pp1b,
                                T& pp2b) {
  if (!(um1 - up1 > T(0))) return;
  const T dp1 = pp1 - pm1, dp2 = pp2 - pm2;
  if (!(vabs(dp1) > T(kEpsShock) * vmin(pp1, pm1)) || !(dp2 != T(0))) return;
  const T ratio = dp1 / dp2;
  const T x = T(kOmega2) * (ratio - T(kOmega1));
  if (!(x < T(1)) || !(x > T(0))) return;
  const T rb = T(kOmega2) * ob;
  const T dp1b = rb / dp2, dp2b = -(rb * ratio) / dp2;
  pp1b += dp1b;
  pm1b -= dp1b;
  pp2b += dp2b;
  pm2b -= dp2b;
}

// Where f is 0 the detector it came from is 0 and passes nothing on: fb is left
// out there, as are the products with f.
template <typename T>
CELLO_HD void flatten_monotone_bwd(T a, T f, T aL, T aR, T oLb, T oRb, T& ab, T& fb, T& aLb, T& aRb) {
  const bool flat = f != T(0);
  T l = aL, r = aR;
  if (flat) {
    l = f * a + (T(1) - f) * aL;
    r = f * a + (T(1) - f) * aR;
  }
  const T d1 = r - a, d2 = a - l;
  bool ext;
  if (std::is_same<T, double>::value && q64::within<-500, 500>(q64::mag(d1)) &&
      q64::within<-500, 500>(q64::mag(d2)))
    ext = (int)(q64::high(d1) ^ q64::high(d2)) < 0;
  else
    ext = d1 * d2 <= T(0);
  if (ext) {
    ab += oLb + oRb;
    return;
  }
  T lb = oLb, rb = oRb;
  const T da = r - l, dm = a - T(0.5) * (l + r);
  const T t1 = da * dm, t2 = (da * da) * T(1.0 / 6.0);
  if (t1 > t2) {
    ab = vfma(T(3), oLb, ab);
    rb = vfma(T(-2), oLb, rb);
    lb = T(0);
  }
  if (-t2 > t1) {   // not both
    ab = vfma(T(3), oRb, ab);
    lb = vfma(T(-2), oRb, lb);
    rb = T(0);
  }
  if (flat) {
    fb += lb * (a - aL) + rb * (a - aR);
    ab += (lb + rb) * f;
    lb *= T(1) - f;
    rb *= T(1) - f;
  }
  aLb += lb;
  aRb += rb;
}

template <typename T>
CELLO_HD void avg_right_bwd(T aL, T aR, T a6, T s, T ob, T& aLb, T& aRb, T& a6b, T& sb) {
  const T h = T(0.5) * s, g = T(1) - T(2.0 / 3.0) * s;
  const T oh = ob * h;
  aRb += ob - oh;
  aLb += oh;
  a6b = vfma(oh, g, a6b);
  sb = vfma(-ob, vfma(T(2.0 / 3.0) * s - T(0.5), a6, T(0.5) * (aR - aL)), sb);   // h 2/3 - g/2 = 2/3 s - 1/2
}

template <typename T>
CELLO_HD void avg_left_bwd(T aL, T aR, T a6, T s, T ob, T& aLb, T& aRb, T& a6b, T& sb) {
  const T h = T(0.5) * s, g = T(1) - T(2.0 / 3.0) * s;
  const T oh = ob * h;
  aLb += ob - oh;
  aRb += oh;
  a6b = vfma(oh, g, a6b);
  sb = vfma(ob, vfma(T(0.5) - T(2.0 / 3.0) * s, a6, T(0.5) * (aR - aL)), sb);
}

// Reverse of trace(): adjoints of the two edge states -> adjoints of the
// cell-centre primitives and of the monotone edge values.
template <typename T>
CELLO_HD void trace_bwd(const T W[5], const T aL[5], const T aR[5], T dtdx, const Gas<T>& gs, const T Wmb[5],
                        const T Wpb[5], T Wb[5], T aLb[5], T aRb[5]) {
  const T rho = W[0], un = W[1], p = W[4];
  T csq, c, ic, ir;
  bool fast = false;
  if constexpr (std::is_same<T, double>::value) {   // the ranges of q64::edge_states
    fast = q64::within<-34, 50>(q64::high(rho)) && q64::within<-68, 50>(q64::high(p)) && gs.gamma < 16.0;
    if (fast) {
      ir = q64::rcp(rho);
      csq = q64::quot(gs.gamma * p, rho, ir);
      c = q64::root(csq, ic);
    }
  }
  if (!fast) {
    csq = (gs.gamma * p) / rho;
    c = vsqrt(csq);
    ic = inverse(c);
    ir = inverse(rho);
  }
  T a6[5], a6b[5];
  for (int q = 0; q < 5; ++q) {
    a6[q] = T(6) * vfma(T(-0.5), aL[q] + aR[q], W[q]);
    a6b[q] = T(0);
  }
  const T lm = un - c, l0 = un, lp = un + c;
  const T icsq = ic * ic;
  const T hrc = (T(0.5) * rho) * ic;
  const T hic = T(0.5) * icsq;
  const T cr = c * ir;
  T lmb = 0, l0b = 0, lpb = 0, csqb = 0, cb = 0, rhob = 0, hrcb = 0, hicb = 0, crb = 0;

  {  // right edge
    const T sp = lp * dtdx, s0 = l0 * dtdx, sm = lm * dtdx;
    T ref[5], refb[5];
    for (int q = 0; q < 5; ++q) {
      ref[q] = (lp > T(0)) ? avg_right(aL[q], aR[q], a6[q], sp) : aR[q];
      refb[q] = T(0);
    }
    T bm = T(0), b0 = T(0), B1 = T(0), B4 = T(0), A0 = T(0), A4 = T(0);
    if (lm > T(0)) {
      B4 = avg_right(aL[4], aR[4], a6[4], sm);
      B1 = avg_right(aL[1], aR[1], a6[1], sm);
      bm = (ref[4] - B4) * hic - (ref[1] - B1) * hrc;
    }
    if (l0 > T(0)) {
      A0 = avg_right(aL[0], aR[0], a6[0], s0);
      A4 = avg_right(aL[4], aR[4], a6[4], s0);
      b0 = (ref[0] - A0) - (ref[4] - A4) * icsq;
    }
    T bmb = 0, b0b = 0, spb = 0, s0b = 0, smb = 0;
    // transverse components
    for (int q = 2; q < 4; ++q) {
      if (l0 > T(0)) avg_right_bwd(aL[q], aR[q], a6[q], s0, Wpb[q], aLb[q], aRb[q], a6b[q], s0b);
      else refb[q] += Wpb[q];
    }
    {  // Wp[4] = max(ref4 - csq*bm, floor)
      const T x4 = ref[4] - csq * bm;
      if (x4 > T(kPFloor)) {
        refb[4] += Wpb[4];
        csqb -= Wpb[4] * bm;
        bmb -= Wpb[4] * csq;
      }
    }
    refb[1] += Wpb[1];  // Wp[1] = ref1 + cr*bm
    crb += Wpb[1] * bm;
    bmb += Wpb[1] * cr;
    {  // Wp[0] = max(ref0 - (b0 + bm), floor)
      const T x0 = ref[0] - (b0 + bm);
      if (x0 > T(kRhoFloor)) {
        refb[0] += Wpb[0];
        b0b -= Wpb[0];
        bmb -= Wpb[0];
      }
    }
    if (l0 > T(0)) {
      refb[0] += b0b;
      const T A0b = -b0b;
      const T D4 = ref[4] - A4;
      const T D4b = -b0b * icsq;
      csqb = vfma(-D4b * icsq, D4, csqb);
      refb[4] += D4b;
      const T A4b = -D4b;
      avg_right_bwd(aL[0], aR[0], a6[0], s0, A0b, aLb[0], aRb[0], a6b[0], s0b);
      avg_right_bwd(aL[4], aR[4], a6[4], s0, A4b, aLb[4], aRb[4], a6b[4], s0b);
    }
    if (lm > T(0)) {
      refb[4] += bmb * hic;
      hicb += bmb * (ref[4] - B4);
      refb[1] -= bmb * hrc;
      hrcb -= bmb * (ref[1] - B1);
      avg_right_bwd(aL[4], aR[4], a6[4], sm, -bmb * hic, aLb[4], aRb[4], a6b[4], smb);
      avg_right_bwd(aL[1], aR[1], a6[1], sm, bmb * hrc, aLb[1], aRb[1], a6b[1], smb);
    }
    for (int q = 0; q < 5; ++q) {
      if (lp > T(0)) avg_right_bwd(aL[q], aR[q], a6[q], sp, refb[q], aLb[q], aRb[q], a6b[q], spb);
      else aRb[q] += refb[q];
    }
    lpb += spb * dtdx;
    l0b += s0b * dtdx;
    lmb += smb * dtdx;
  }
  {  // left edge
    const T tm = -lm * dtdx, t0 = -l0 * dtdx, tp = -lp * dtdx;
    T ref[5], refb[5];
    for (int q = 0; q < 5; ++q) {
      ref[q] = (lm < T(0)) ? avg_left(aL[q], aR[q], a6[q], tm) : aL[q];
      refb[q] = T(0);
    }
    T bp = T(0), b0 = T(0), B1 = T(0), B4 = T(0), A0 = T(0), A4 = T(0);
    if (lp < T(0)) {
      B4 = avg_left(aL[4], aR[4], a6[4], tp);
      B1 = avg_left(aL[1], aR[1], a6[1], tp);
      bp = (ref[4] - B4) * hic + (ref[1] - B1) * hrc;
    }
    if (l0 < T(0)) {
      A0 = avg_left(aL[0], aR[0], a6[0], t0);
      A4 = avg_left(aL[4], aR[4], a6[4], t0);
      b0 = (ref[0] - A0) - (ref[4] - A4) * icsq;
    }
    T bpb = 0, b0b = 0, tpb = 0, t0b = 0, tmb = 0;
    for (int q = 2; q < 4; ++q) {
      if (l0 < T(0)) avg_left_bwd(aL[q], aR[q], a6[q], t0, Wmb[q], aLb[q], aRb[q], a6b[q], t0b);
      else refb[q] += Wmb[q];
    }
    {
      const T x4 = ref[4] - csq * bp;
      if (x4 > T(kPFloor)) {
        refb[4] += Wmb[4];
        csqb -= Wmb[4] * bp;
        bpb -= Wmb[4] * csq;
      }
    }
    refb[1] += Wmb[1];  // Wm[1] = ref1 - cr*bp
    crb -= Wmb[1] * bp;
    bpb -= Wmb[1] * cr;
    {
      const T x0 = ref[0] - (b0 + bp);
      if (x0 > T(kRhoFloor)) {
        refb[0] += Wmb[0];
        b0b -= Wmb[0];
        bpb -= Wmb[0];
      }
    }
    if (l0 < T(0)) {
      refb[0] += b0b;
      const T A0b = -b0b;
      const T D4 = ref[4] - A4;
      const T D4b = -b0b * icsq;
      csqb = vfma(-D4b * icsq, D4, csqb);
      refb[4] += D4b;
      const T A4b = -D4b;
      avg_left_bwd(aL[0], aR[0], a6[0], t0, A0b, aLb[0], aRb[0], a6b[0], t0b);
      avg_left_bwd(aL[4], aR[4], a6[4], t0, A4b, aLb[4], aRb[4], a6b[4], t0b);
    }
    if (lp < T(0)) {
      refb[4] += bpb * hic;
      hicb += bpb * (ref[4] - B4);
      refb[1] += bpb * hrc;
      hrcb += bpb * (ref[1] - B1);
      avg_left_bwd(aL[4], aR[4], a6[4], tp, -bpb * hic, aLb[4], aRb[4], a6b[4], tpb);
      avg_left_bwd(aL[1], aR[1], a6[1], tp, -bpb * hrc, aLb[1], aRb[1], a6b[1], tpb);
    }
    for (int q = 0; q < 5; ++q) {
      if (lm < T(0)) avg_left_bwd(aL[q], aR[q], a6[q], tm, refb[q], aLb[q], aRb[q], a6b[q], tmb);
      else aLb[q] += refb[q];
    }
    lmb -= tmb * dtdx;
    l0b -= t0b * dtdx;
    lpb -= tpb * dtdx;
  }
  // shared coefficients
  T unb = lmb + l0b + lpb;
  cb += lpb - lmb;
  rhob = vfma(T(0.5) * hrcb, ic, rhob);
  cb = vfma(-hrcb * hrc, ic, cb);
  csqb = vfma(-hicb * hic, icsq, csqb);
  cb = vfma(crb, ir, cb);
  rhob = vfma(-crb * cr, ir, rhob);
  for (int q = 0; q < 5; ++q) {
    Wb[q] += T(6) * a6b[q];
    aLb[q] -= T(3) * a6b[q];
    aRb[q] -= T(3) * a6b[q];
  }
  csqb = vfma(T(0.5) * cb, ic, csqb);
  const T pb = csqb * gs.gamma * ir;
  rhob = vfma(-csqb * csq, ir, rhob);
  Wb[0] += rhob;
  Wb[1] += unb;
  Wb[4] += pb;
}

// One side of the two-shock solver in reverse: its pressure, wave impedance C,
// their reciprocals, the sign of its velocity jump, and the adjoints of its
// pressure, C and velocity.
template <typename T>
struct ShockSide {
  T p, C, ip, iC, sgn;
  T pb, Cb, ub;
};

// Adjoints of (us, Z, W) of the shock curve at pressure ps -> (ps, p, C, u):
// x = 1 + g1 (ps/p - 1), W = C sqrt(x), us = u -/+ (ps - p)/W,
// Z = 2 W^3/(W^2 + C^2).  Returns the adjoint of ps.  iW = 1/W, iden = 1/(W^2 + C^2).
template <typename T>
CELLO_HD T shock_side_bwd(ShockSide<T>& k, T ps, T W, T iW, T iden, T usb, T Zb, T Wb, const Gas<T>& gs) {
  const T W2 = W * W, C2 = k.C * k.C;
  const T z = T(2) * W2 * (iden * iden) * Zb;
  const T q = (ps - k.p) * iW, qb = k.sgn * usb * iW;
  const T Wbar = vfma(-qb, q, vfma(z, vfma(T(3), C2, W2), Wb));
  const T xb = T(0.5) * Wbar * C2 * iW * gs.g1 * k.ip;   // adjoint of ps/p, over p
  k.ub += usb;
  k.Cb = vfma(Wbar, W * k.iC, vfma(T(-2) * z * W, k.C, k.Cb));
  k.pb -= vfma(xb * ps, k.ip, qb);
  return qb + xb;
}

// Reverse of riemann_flux(): flux adjoints -> adjoints of the two states.
template <typename T>
CELLO_HD void riemann_flux_bwd(const T L[5], const T R[5], const Gas<T>& gs, const T Fb[5], T Lb[5], T Rb[5]) {
  const T rL = L[0], uL = L[1], pL = L[4];
  const T rR = R[0], uR = R[1], pR = R[4];
  // the forward iteration with its exit at a fixed point; pressures and W kept
  T hp[kRiemannIters + 1], hL[kRiemannIters + 1], hR[kRiemannIters + 1];
  unsigned floored = 0;   // bit k: the pressure of evaluation k was floored
  int last = 0, turn = -1;
  T CL, CR, ps_raw0, ps, WLs, WRs, uLs, uRs, ZL, ZR;
  bool solved = false;
  if constexpr (std::is_same<T, double>::value) {
    q64::Side l, r;
    solved = q64::shock_history(L, R, gs, hp, hL, hR, floored, last, turn, ps_raw0, l, r);
    if (solved) {
      ps = hp[last];
      CL = l.C; WLs = l.W; uLs = l.us; ZL = T(2) * l.z;
      CR = r.C; WRs = r.W; uRs = r.us; ZR = T(2) * r.z;
    }
  }
  if (!solved) {
    CL = vsqrt((gs.gamma * pL) * rL);
    CR = vsqrt((gs.gamma * pR) * rR);
    ps_raw0 = ((CR * pL + CL * pR) + (CL * CR) * (uL - uR)) / (CL + CR);
    ps = vmax(ps_raw0, T(kPFloor));
    floored = (ps_raw0 > T(kPFloor)) ? 0u : 1u;
#pragma unroll 1
    for (last = 0;; ++last) {
      WLs = CL * vsqrt(T(1) + gs.g1 * (ps / pL - T(1)));
      WRs = CR * vsqrt(T(1) + gs.g1 * (ps / pR - T(1)));
      uLs = uL - (ps - pL) / WLs;
      uRs = uR + (ps - pR) / WRs;
      ZL = ((T(2) * WLs) * WLs) * WLs / (WLs * WLs + CL * CL);
      ZR = ((T(2) * WRs) * WRs) * WRs / (WRs * WRs + CR * CR);
      hp[last] = ps;
      hL[last] = WLs;
      hR[last] = WRs;
      if (last == kRiemannIters) break;
      const T raw = ps - ((ZL * ZR) * (uRs - uLs)) / (ZL + ZR);
      const T pn = vmax(raw, T(kPFloor));
      if (!(raw > T(kPFloor))) floored |= 2u << last;
      if (pn == ps) break;
      ps = pn;
    }
  }
  const T iD = inverse(ZL + ZR);
  const T us = (ZL * uLs + ZR * uRs) / (ZL + ZR);
  const bool left = us >= T(0);
  const T rs = left ? rL : rR, u_s = left ? uL : uR, p_s = left ? pL : pR, W_s = left ? WLs : WRs;
  const T t1 = left ? L[2] : R[2], t2 = left ? L[3] : R[3];
  const T v_s = left ? -uL : uR, v_star = left ? -us : us;
  const T tau = T(1) / rs - (ps - p_s) / (W_s * W_s);
  const T rstar_raw = (tau > T(0)) ? T(1) / tau : T(kRhoFloor);
  const T rstar = vmax(rstar_raw, T(kRhoFloor));
  const bool shock = ps > p_s;
  T c_s = T(0), c_star = T(0), head, tail;
  if (shock) {
    head = tail = v_s + W_s / rs;
  } else {
    c_s = vsqrt((gs.gamma * p_s) / rs);
    c_star = vsqrt((gs.gamma * ps) / rstar);
    head = v_s + c_s;
    tail = v_star + c_star;
  }
  const bool orig = head <= T(0);
  const bool star = !orig && (tail > T(0));
  const bool fan = !orig && !star;
  T r, u, p, w = T(0), iht = T(0);
  if (orig) {
    r = rs; u = u_s; p = p_s;
  } else if (star) {
    r = rstar; u = us; p = ps;
  } else {
    iht = T(1) / (head - tail);
    w = head * iht;
    r = vfma(w, rstar - rs, rs);
    u = vfma(w, us - u_s, u_s);
    p = vfma(w, ps - p_s, p_s);
  }
  // flux
  const T f0 = r * u;
  const T tt = vfma(t1, t1, t2 * t2);
  const T k2 = vfma(u, u, tt);
  const T E = vfma(p, gs.inv_gm1, (T(0.5) * r) * k2);
  const T Eb = Fb[4] * u;
  const T Er = Eb * r;
  const T f0b = vfma(Fb[1], u, vfma(Fb[2], t1, vfma(Fb[3], t2, Fb[0])));
  const T ub = vfma(Fb[1], f0, vfma(Fb[4], E + p, vfma(f0b, r, Er * u)));
  const T pb = vfma(Fb[4], u, vfma(Eb, gs.inv_gm1, Fb[1]));
  const T rb = vfma(f0b, u, T(0.5) * Eb * k2);
  const T t1b = vfma(Fb[2], f0, Er * t1);
  const T t2b = vfma(Fb[3], f0, Er * t2);
  // sampling
  T rsb = 0, u_sb = 0, p_sb = 0, W_sb = 0, rstarb = 0, usb = 0, psb = 0, v_sb = 0, v_starb = 0;
  if (orig) {
    rsb = rb; u_sb = ub; p_sb = pb;
  } else if (star) {
    rstarb = rb; usb = ub; psb = pb;
  }
  const T irs = inverse(rs);
  if (fan) {   // rarefaction: head = v_s + c_s, tail = v* + c*, c = sqrt(gamma p / rho)
    const T wb = vfma(rb, rstar - rs, vfma(ub, us - u_s, pb * (ps - p_s)));
    rstarb = rb * w; rsb = rb - rstarb;
    usb = ub * w; u_sb = ub - usb;
    psb = pb * w; p_sb = pb - psb;
    v_sb = -wb * tail * (iht * iht);
    v_starb = wb * w * iht;
    const T sb = T(0.5) * v_sb / c_s, xb = T(0.5) * v_starb / c_star, irst = inverse(rstar);
    p_sb = vfma(sb * gs.gamma, irs, p_sb);
    rsb = vfma(-sb * gs.gamma * p_s, irs * irs, rsb);
    psb = vfma(xb * gs.gamma, irst, psb);
    rstarb = vfma(-xb * gs.gamma * ps, irst * irst, rstarb);
  }
  if (rstar_raw > T(kRhoFloor) && tau > T(0)) {  // rstar = 1/tau
    const T taub = -rstarb * rstar * rstar;
    rsb = vfma(-taub, irs * irs, rsb);
    const T iW = inverse(W_s), tw = taub * iW * iW;
    psb -= tw;
    p_sb += tw;
    W_sb = T(2) * tw * (ps - p_s) * iW;
  }
  usb += left ? -v_starb : v_starb;
  ShockSide<T> a, b;
  a.p = pL; a.C = CL; a.ip = inverse(pL); a.iC = inverse(CL); a.sgn = T(-1);
  b.p = pR; b.C = CR; b.ip = inverse(pR); b.iC = inverse(CR); b.sgn = T(1);
  a.pb = a.Cb = a.ub = b.pb = b.Cb = b.ub = T(0);
  // us = (ZL*usL + ZR*usR)/D
  psb += shock_side_bwd(a, ps, WLs, inverse(WLs), inverse(vfma(WLs, WLs, CL * CL)), usb * ZL * iD, usb * (uLs - us) * iD, left ? W_sb : T(0), gs);
  psb += shock_side_bwd(b, ps, WRs, inverse(WRs), inverse(vfma(WRs, WRs, CR * CR)), usb * ZR * iD, usb * (uRs - us) * iD, left ? T(0) : W_sb, gs);
  // Newton iterations in reverse, p_{k+1} = max(p_k - q(p_k), floor): those
  // after a fixed point all have its derivative m = 1 - q', so n of them pass
  // psb m^n on and add (1 + m + ... + m^(n-1)) times one iteration's adjoints;
  // two pressures in turn likewise, with one evaluation of each
  auto iteration = [&](int it, T adj[6]) {   // for psb = 1: (p, C, u) of both sides; returns m
    const T pk = hp[it], WA = hL[it], WB = hR[it];
    const T iA = inverse(WA), dA = inverse(vfma(WA, WA, CL * CL));
    const T iB = inverse(WB), dB = inverse(vfma(WB, WB, CR * CR));
    const T ZA = T(2) * WA * WA * WA * dA, ZB = T(2) * WB * WB * WB * dB;
    const T iZ = inverse(ZA + ZB);
    const T du = vfma(pk - pR, iB, uR) - vfma(pL - pk, iA, uL);
    const T zz = ZA * ZB * iZ, q = zz * du;
    ShockSide<T> x = a, y = b;
    x.pb = x.Cb = x.ub = y.pb = y.Cb = y.ub = T(0);
    T m = T(1);
    m += shock_side_bwd(x, pk, WA, iA, dA, zz, -vfma(ZB, du, -q) * iZ, T(0), gs);
    m += shock_side_bwd(y, pk, WB, iB, dB, -zz, -vfma(ZA, du, -q) * iZ, T(0), gs);
    adj[0] = x.pb; adj[1] = x.Cb; adj[2] = x.ub;
    adj[3] = y.pb; adj[4] = y.Cb; adj[5] = y.ub;
    return m;
  };
  auto add = [&](T sum, const T adj[6]) {
    a.pb = vfma(sum, adj[0], a.pb); a.Cb = vfma(sum, adj[1], a.Cb); a.ub = vfma(sum, adj[2], a.ub);
    b.pb = vfma(sum, adj[3], b.pb); b.Cb = vfma(sum, adj[4], b.Cb); b.ub = vfma(sum, adj[5], b.ub);
  };
  int reps = kRiemannIters - last, it = reps > 0 ? last : last - 1;
  if (turn >= 0 && last - turn > 2 && floored == 0) {
    T adj[2][6], m[2], sum[2] = {T(0), T(0)};
#pragma unroll 1
    for (int k = 0; k < 2; ++k) m[k] = iteration(turn + k, adj[k]);
    for (; it >= turn; --it) {
      sum[(it - turn) & 1] += psb;
      psb *= m[(it - turn) & 1];
    }
#pragma unroll 1
    for (int k = 0; k < 2; ++k) add(sum[k], adj[k]);
  }
#pragma unroll 1
  for (; it >= 0; --it, reps = 1) {
    if (reps == 0) reps = 1;
    if (floored & (2u << it)) {
      psb = T(0);
      continue;
    }
    T adj[6];
    const T m = iteration(it, adj);
    T sum = T(0);
    for (int k = 0; k < reps; ++k) {
      sum += psb;
      psb *= m;
    }
    add(sum, adj);
  }
  if (!(floored & 1u)) {  // p_0 = ((CR pL + CL pR) + (CL CR)(uL - uR)) / (CL + CR)
    const T nb = psb * inverse(CL + CR), du = uL - uR, cc = nb * CL * CR;
    a.pb = vfma(nb, CR, a.pb);
    b.pb = vfma(nb, CL, b.pb);
    a.Cb = vfma(nb, vfma(CR, du, pR) - ps_raw0, a.Cb);
    b.Cb = vfma(nb, vfma(CL, du, pL) - ps_raw0, b.Cb);
    a.ub += cc;
    b.ub -= cc;
  }
  // C = sqrt(gamma p rho)
  const T ga = T(0.5) * gs.gamma * a.Cb * a.iC, gb = T(0.5) * gs.gamma * b.Cb * b.iC;
  Lb[0] += vfma(ga, pL, left ? rsb : T(0));
  Lb[1] += a.ub + (left ? u_sb - v_sb : T(0));
  Lb[2] += left ? t1b : T(0);
  Lb[3] += left ? t2b : T(0);
  Lb[4] += vfma(ga, rL, a.pb + (left ? p_sb : T(0)));
  Rb[0] += vfma(gb, pR, left ? T(0) : rsb);
  Rb[1] += b.ub + (left ? T(0) : u_sb + v_sb);
  Rb[2] += left ? T(0) : t1b;
  Rb[3] += left ? T(0) : t2b;
  Rb[4] += vfma(gb, rR, b.pb + (left ? T(0) : p_sb));
}

}  // namespace cello
