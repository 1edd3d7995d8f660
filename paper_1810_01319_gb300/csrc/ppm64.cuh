// The float64 arithmetic of the PPM sweep with few float64 instructions.
//
// The float64 sweep is bound by the float64 pipe: 1.9 instructions per SM and
// clock measured, against 128 for integers.  These functions return the values of
// their namesakes in ppm.cuh, rounded alike, from less work on that pipe:
//  * Divisions by one divisor share its reciprocal.  With r = 1/b to about an
//    ulp, q = a r and q + r (a - b q), the remainder exact in a fused
//    multiply-add, is the correctly rounded quotient (P. Markstein, IBM J. Res.
//    Dev. 34, 1990, 111-119): 3 instructions per quotient.  Only a quotient (or
//    root) within 2^-50 ulp of the midpoint of two numbers could round differently.
//  * A reciprocal is a float32 seed and one correction of third order, 3
//    instructions; a square root the same on 1/sqrt(x) with a last remainder step,
//    8, which leaves the root's reciprocal as well.
//  * Comparisons, minima, maxima, signs, halving and doubling of numbers known to
//    be finite and away from the ends of the range work on their bits.
//  * A product with an exact factor (a power of two) is fused with the sum it
//    enters: nothing is rounded that was not.
//  * Work whose result is not used (the detector's ratio off shocks, constraints on
//    extrema, waves that do not reach an edge) is behind a branch.
// Each function takes its short way where the arguments allow it (checked on
// their exponents: no float32 seed, product or remainder leaves its range) and is
// the formula of ppm.cuh elsewhere: zeros, NaN and infinities, huge and tiny
// values give what they gave.  A zero result may differ in its sign.
//
// Two steps of 939 16^3 leaves: 55.9 -> 37.8 ms; three steps of a gradient on 64
// leaves, whose adjoint sweep forms the same values, 38.0 -> 29.2 ms.
#pragma once

#include <cstring>

#include "ppm.cuh"

namespace cello {
namespace q64 {

CELLO_HD long long bits(double a) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(a);
#else
  long long v; std::memcpy(&v, &a, 8); return v;
#endif
}
CELLO_HD double from_bits(long long v) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(v);
#else
  double a; std::memcpy(&a, &v, 8); return a;
#endif
}
CELLO_HD unsigned fbits(float a) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(a);
#else
  unsigned v; std::memcpy(&v, &a, 4); return v;
#endif
}
CELLO_HD float from_fbits(unsigned v) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(v);
#else
  float a; std::memcpy(&a, &v, 4); return a;
#endif
}
CELLO_HD unsigned high(double a) { return (unsigned)((unsigned long long)bits(a) >> 32); }
CELLO_HD unsigned mag(double a) { return high(a) & 0x7fffffffu; }   // high word without the sign

CELLO_HD constexpr unsigned exp_word(int e) { return (unsigned)(e + 1023) << 20; }   // high word of 2^e
// The high word lies in that of [2^lo, 2^hi): false for negative numbers, zero, NaN.
template <int LO, int HI>
CELLO_HD bool within(unsigned h) { return h - exp_word(LO) < exp_word(HI) - exp_word(LO); }
CELLO_HD bool is_zero(double a) { return (bits(a) << 1) == 0; }

CELLO_HD double flip(double a) { return from_bits(bits(a) ^ (long long)0x8000000000000000ull); }   // -a
// Comparisons of finite numbers of which the right one is not negative.
CELLO_HD bool gt_pos(double a, double b) { return bits(a) > bits(b); }
CELLO_HD bool positive(double a) { return bits(a) > 0; }
CELLO_HD double max_pos(double a, double floor) { return gt_pos(a, floor) ? a : floor; }
CELLO_HD double absval(double a) { return from_bits(bits(a) & 0x7fffffffffffffffll); }
CELLO_HD double pick(bool c, double a, double b) { return from_bits(c ? bits(a) : bits(b)); }

// A positive number of [2^-126, 2^127) cut to float32, and back.
CELLO_HD float narrow(double a) {
  const unsigned long long v = (unsigned long long)bits(a);
  return from_fbits((unsigned)(v >> 29) - 0xC0000000u);
}
CELLO_HD double widen_pos(float a) {
  return from_bits((long long)(((unsigned long long)fbits(a) << 29) + 0x3800000000000000ull));
}
CELLO_HD float seed_rcp(float a) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.0f, a);
#else
  return 1.0f / a;
#endif
}
CELLO_HD float seed_rsqrt(float a) {
#ifdef __CUDA_ARCH__
  return rsqrtf(a);
#else
  return 1.0f / sqrtf(a);
#endif
}

// 1/b within an ulp, b in [2^-120, 2^120): with e = 1 - b y, 1/b = y / (1 - e) =
// y (1 + e + e^2 + O(e^3)), |e| < 2^-21.
CELLO_HD double rcp(double b) {
  const double y = widen_pos(seed_rcp(narrow(b)));
  const double e = fma(-b, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// a / b with r = 1/b to a few ulp; a zero or in [2^-800, 2^800).
CELLO_HD double quot(double a, double b, double r) {
  const double q = a * r;
  return fma(fma(-b, q, a), r, q);
}
// The same for any a (b and r as above).
CELLO_HD double quot_any(double a, double b, double r) {
  if (within<-800, 800>(mag(a))) return quot(a, b, r);
  return is_zero(a) ? a : a / b;
}
// 1 / b rounded.
CELLO_HD double rcp_rn(double b) {
  const double r = rcp(b);
  return fma(fma(-b, r, 1.0), r, r);
}
// sqrt(x), x in [2^-120, 2^120), and 1/sqrt(x) to about an ulp in inv: with y a
// seed, g = x y, e = (1 - g y) / 2: sqrt(x) = g / sqrt(1 - 2 e) = g (1 + e + 3/2
// e^2 + O(e^3)), the same factor for y; the remainder x - g^2 rounds the root.
CELLO_HD double root(double x, double& inv) {
  const double y = widen_pos(seed_rsqrt(narrow(x)));
  const double h = from_bits(bits(y) - 0x0010000000000000ll);   // y / 2
  const double g0 = x * y;
  const double e = fma(-h, g0, 0.5);
  const double s = fma(e * 1.5, e, e);
  const double g = fma(g0, s, g0), k = fma(h, s, h);            // root, half its reciprocal
  inv = from_bits(bits(k) + 0x0010000000000000ll);
  const double v = fma(fma(-g, g, x), k, g);
  constexpr long long kMant = 0x000fffffffffffffll;
  // the root of the number below a power of 4 is 2^-56 ulp under the midpoint of
  // that power's root and the number below it: the one argument that k cannot
  // round in time (and a common one: 1 - 2^-53)
  const bool under = ((bits(x) + 1) & kMant) == 0 && (bits(v) & kMant) == 0;
  return from_bits(bits(v) - (under ? 1 : 0));
}

// ---- the sweep's functions ----

template <int NQ>
CELLO_HD void primitives(const double U[NQ], const Gas<double>& gs, double W[NQ]) {
  const bool plain = within<-33, 100>(high(U[0]));   // above the floor
  if (!plain) {
    if constexpr (NQ == 6) to_primitive_de(U, gs, W);
    else to_primitive(U, gs, W);
    return;
  }
  const double rho = U[0], r = rcp(rho);
  const double un = quot_any(U[1], rho, r), ut1 = quot_any(U[2], rho, r), ut2 = quot_any(U[3], rho, r);
  const double ke = (0.5 * rho) * (un * un + (ut1 * ut1 + ut2 * ut2));
  const double eint = U[4] - ke;
  W[0] = rho; W[1] = un; W[2] = ut1; W[3] = ut2;
  if constexpr (NQ == 6) {
    W[4] = vmax(gs.gm1 * ((eint > kDualEta1 * U[4]) ? eint : U[5]), kPFloor);
    W[5] = quot_any(U[5], rho, r);
  } else {
    W[4] = vmax(gs.gm1 * eint, kPFloor);
  }
}

// limited_slope: where the differences have one sign, their sum has it too.
CELLO_HD double slope(double am, double a0, double ap) {
  const double dl = a0 - am, dr = ap - a0;
  if (within<-500, 500>(mag(dl)) && within<-500, 500>(mag(dr))) {
    if ((int)(high(dl) ^ high(dr)) < 0) return 0.0;
    constexpr long long kTwo = 0x0010000000000000ll;   // one in the exponent
    const double da2 = ap - am;
    const long long l = bits(absval(dl)), r = bits(absval(dr)), d = bits(absval(da2)) - kTwo;
    long long m = (l < r ? l : r) + kTwo;
    m = d < m ? d : m;
    return from_bits(m | (bits(dl) & (long long)0x8000000000000000ull));
  }
  if (is_zero(dl) || is_zero(dr)) return 0.0;
  return limited_slope(am, a0, ap);
}

CELLO_HD double interface_val(double a0, double a1, double dm0, double dm1) {
  return fma(0.5, a0 + a1, -((dm1 - dm0) * (1.0 / 6.0)));
}

// flatten_tilde: a condition at a time, the ratio where all hold.
CELLO_HD double detector(double pm2, double pm1, double pp1, double pp2, double um1, double up1) {
  if (!(um1 > up1)) return 0.0;   // um1 - up1 > 0
  const double dp1 = pp1 - pm1;
  if (!(vabs(dp1) > kEpsShock * vmin(pp1, pm1))) return 0.0;
  const double dp2 = pp2 - pm2;
  if (dp2 == 0.0) return 0.0;
  return vmax(vmin(kOmega2 * (dp1 / dp2 - kOmega1), 1.0), 0.0);
}

// The flattening coefficient of cell j from the detectors of cells j - 1, j, j + 1
// and the pressures beside it: the upstream one if larger.
CELLO_HD double flattening(double pm1, double pp1, double fj, double fm, double fp) {
  if (is_zero(fj) && is_zero(fm) && is_zero(fp)) return 0.0;
  const double s = pp1 - pm1;
  return (s > 0.0) ? vmax(fj, fm) : ((s < 0.0) ? vmax(fj, fp) : fj);
}

// The edge values of a cell flattened (f), then under the monotonicity
// constraints; da = aR - aL and a6 = 6 (a - (aL + aR) / 2) of the result.
CELLO_HD void edges(double a, double f, double& aL, double& aR, double& da, double& a6) {
  double l = aL, r = aR;
  if (!is_zero(f)) {   // f = 0: 0 a + 1 aL
    const double fa = f * a, g = 1.0 - f;
    l = fa + g * aL;
    r = fa + g * aR;
  }
  const double d1 = r - a, d2 = a - l;
  const bool fast = within<-500, 500>(mag(d1)) && within<-500, 500>(mag(d2));
  const bool ext = fast ? (int)(high(d1) ^ high(d2)) < 0 : (is_zero(d1) || is_zero(d2) || d1 * d2 <= 0.0);
  if (ext) {
    aL = aR = a;
    da = a6 = 0.0;
    return;
  }
  da = r - l;
  double dm = fma(-0.5, l + r, a);
  const double t1 = da * dm, t2 = (da * da) * (1.0 / 6.0);
  const bool cl = gt_pos(t1, t2), cr = gt_pos(flip(t1), t2);
  if (cl || cr) {
    const double a3 = 3.0 * a;
    if (cl) l = fma(-2.0, r, a3);
    else r = fma(-2.0, l, a3);
    da = r - l;
    dm = fma(-0.5, l + r, a);
  }
  aL = l;
  aR = r;
  a6 = 6.0 * dm;
}

// Both edges of a cell, from interface values to traced states (flatten_monotone
// of each field, then trace).
template <int NQ>
CELLO_HD void edge_states(const double W[NQ], double f, double aL[NQ], double aR[NQ], double dtdx,
                          const Gas<double>& gs, double Wm[NQ], double Wp[NQ]) {
  unsigned big = 0;   // every value finite, with room for products
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const unsigned a = mag(W[q]), b = mag(aL[q]), c = mag(aR[q]);
    big = big > a ? big : a;
    big = big > b ? big : b;
    big = big > c ? big : c;
  }
  if (!(big < exp_word(50) && within<-34, 50>(high(W[0])) && within<-68, 50>(high(W[4])) && gs.gamma < 16.0 &&
        mag(dtdx) < exp_word(100))) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) flatten_monotone(W[q], f, aL[q], aR[q]);
    trace<double, NQ>(W, aL, aR, dtdx, gs, Wm, Wp);
    return;
  }
  double da[NQ], a6[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) edges(W[q], f, aL[q], aR[q], da[q], a6[q]);
  const double rho = W[0], un = W[1];
  const double ir = rcp(rho);
  const double csq = quot(gs.gamma * W[4], rho, ir);
  double ic;
  const double c = root(csq, ic);
  const double lm = un - c, lp = un + c;
  const bool movr = positive(un), movl = positive(flip(un));
  const double icsq = ic * ic;
  // averages over the domain of dependence of a wave: s = its speed dtdx
  auto right = [&](int q, double hs, double k) { return aR[q] - hs * (da[q] - k * a6[q]); };
  auto left = [&](int q, double hs, double k) { return aL[q] + hs * (da[q] + k * a6[q]); };
  auto weights = [&](double s, double& hs, double& k) {
    hs = 0.5 * s;
    k = 1.0 - (2.0 / 3.0) * s;
  };
  {  // right edge
    double hs = 0.0, k = 0.0, h0 = 0.0, k0 = 0.0;   // hs = 0: the edge value
    if (positive(lp)) weights(lp * dtdx, hs, k);
    double b0 = 0.0;
    const double r0 = right(0, hs, k), r1 = right(1, hs, k), r4 = right(4, hs, k);
    if (movr) {
      weights(un * dtdx, h0, k0);
      b0 = (r0 - right(0, h0, k0)) - quot_any(r4 - right(4, h0, k0), csq, icsq);
    }
    Wp[1] = r1;
    Wp[4] = r4;
    if (positive(lm)) {
      double hm, km;
      weights(lm * dtdx, hm, km);
      const double bm = (r4 - right(4, hm, km)) * quot(0.5, csq, icsq) -
                        (r1 - right(1, hm, km)) * quot(0.5 * rho, c, ic);
      b0 = b0 + bm;
      Wp[1] = r1 + quot(c, rho, ir) * bm;
      Wp[4] = r4 - csq * bm;
    }
    Wp[0] = max_pos(r0 - b0, kRhoFloor);
    Wp[4] = max_pos(Wp[4], kPFloor);
    hs = pick(movr, h0, hs);
    k = pick(movr, k0, k);
    Wp[2] = right(2, hs, k);
    Wp[3] = right(3, hs, k);
#pragma unroll
    for (int q = 5; q < NQ; ++q) Wp[q] = right(q, hs, k);
  }
  {  // left edge
    double hs = 0.0, k = 0.0, h0 = 0.0, k0 = 0.0;
    if (positive(flip(lm))) weights(-lm * dtdx, hs, k);
    double b0 = 0.0;
    const double r0 = left(0, hs, k), r1 = left(1, hs, k), r4 = left(4, hs, k);
    if (movl) {
      weights(-un * dtdx, h0, k0);
      b0 = (r0 - left(0, h0, k0)) - quot_any(r4 - left(4, h0, k0), csq, icsq);
    }
    Wm[1] = r1;
    Wm[4] = r4;
    if (positive(flip(lp))) {
      double hp, kp;
      weights(-lp * dtdx, hp, kp);
      const double bp = (r4 - left(4, hp, kp)) * quot(0.5, csq, icsq) +
                        (r1 - left(1, hp, kp)) * quot(0.5 * rho, c, ic);
      b0 = b0 + bp;
      Wm[1] = r1 - quot(c, rho, ir) * bp;
      Wm[4] = r4 - csq * bp;
    }
    Wm[0] = max_pos(r0 - b0, kRhoFloor);
    Wm[4] = max_pos(Wm[4], kPFloor);
    hs = pick(movl, h0, hs);
    k = pick(movl, k0, k);
    Wm[2] = left(2, hs, k);
    Wm[3] = left(3, hs, k);
#pragma unroll
    for (int q = 5; q < NQ; ++q) Wm[q] = left(q, hs, k);
  }
}

// 1/a within an ulp.
CELLO_HD double inverse(double a) { return within<-120, 120>(high(a)) ? rcp(a) : 1.0 / a; }

// The two states of an interface are ordinary: see two_shock.
template <int NQ>
CELLO_HD bool ordinary(const double L[NQ], const double R[NQ], const Gas<double>& gs) {
  unsigned big = 0;
#pragma unroll
  for (int q = 1; q < NQ; ++q) {
    if (q == 4) continue;
    big = big > mag(L[q]) ? big : mag(L[q]);
    big = big > mag(R[q]) ? big : mag(R[q]);
  }
  return big < exp_word(48) && within<-34, 48>(high(L[0])) && within<-34, 48>(high(R[0])) &&
         within<-68, 48>(high(L[4])) && within<-68, 48>(high(R[4])) && gs.gamma < 16.0 && gs.gamma > 1.001;
}

// One side of the two-shock solver at the pressure ps: W, u*, and z = Z / 2 (a
// power of two less throughout).
struct Side {
  double C, C2, iC, p, ip, u;
  double W, iW, t, us, z;
  CELLO_HD void set(const double* S, const Gas<double>& gs) {
    p = S[4];
    u = S[1];
    C = root((gs.gamma * p) * S[0], iC);
    C2 = C * C;
    ip = rcp(p);
  }
  CELLO_HD bool at(double ps, const Gas<double>& gs, bool right) {
    const double x = 1.0 + gs.g1 * (quot(ps, p, ip) - 1.0);
    if (!within<-60, 120>(high(x))) return false;
    double ix;
    W = C * root(x, ix);
    iW = iC * ix;
    const double d = quot(ps - p, W, iW);
    us = right ? u + d : u - d;
    t = W * W;
    const double den = t + C2;
    z = quot(t * W, den, rcp(den));
    return true;
  }
};

// riemann_flux.  A pressure that returns after two steps alternates for the rest
// of the iteration: the last one follows from the number of steps left.
template <int NQ>
CELLO_HD bool two_shock(const double L[NQ], const double R[NQ], const Gas<double>& gs, double F[NQ], double* uf) {
  const double rL = L[0], uL = L[1], pL = L[4];
  const double rR = R[0], uR = R[1], pR = R[4];
  if (!ordinary<NQ>(L, R, gs)) return false;
  Side l, r;
  l.set(L, gs);
  r.set(R, gs);
  const double Cs = l.C + r.C;
  double ps = quot_any((r.C * pL + l.C * pR) + (l.C * r.C) * (uL - uR), Cs, rcp(Cs));
  ps = max_pos(ps, kPFloor);
  double before = ps, zs, izs;
#pragma unroll 1
  for (int it = 0;; ++it) {
    if (!within<-68, 50>(high(ps)) || !l.at(ps, gs, false) || !r.at(ps, gs, true)) return false;
    zs = l.z + r.z;
    izs = rcp(zs);
    if (it >= kRiemannIters) break;
    const double pn = max_pos(fma(-2.0, quot_any((l.z * r.z) * (r.us - l.us), zs, izs), ps), kPFloor);
    if (bits(pn) == bits(ps)) break;   // fixed point
    if (it > 0 && bits(pn) == bits(before)) {
      if (((kRiemannIters - it) & 1) == 0) break;   // the last pressure is this one
      it = kRiemannIters - 1;                       // it is the other one
    }
    before = ps;
    ps = pn;
  }
  const double us = quot_any(l.z * l.us + r.z * r.us, zs, izs);

  const bool left = !positive(flip(us));
  const double rs = pick(left, rL, rR), u_s = pick(left, uL, uR), p_s = pick(left, pL, pR);
  const double W_s = pick(left, l.W, r.W), iW = pick(left, l.iW, r.iW), W2 = pick(left, l.t, r.t);
  const double t1 = pick(left, L[2], R[2]), t2 = pick(left, L[3], R[3]);
  const double v_s = pick(left, flip(uL), uR), v_star = pick(left, flip(us), us);
  const double ir = rcp(rs);
  const double tau = quot(1.0, rs, ir) - quot(ps - p_s, W2, iW * iW);
  double rstar = kRhoFloor, irstar = 1.0 / kRhoFloor;
  if (within<-45, 100>(high(tau))) {
    rstar = rcp_rn(tau);
    irstar = tau;
    if (!gt_pos(rstar, kRhoFloor)) {
      rstar = kRhoFloor;
      irstar = 1.0 / kRhoFloor;
    }
  } else if (tau > 0.0) {
    return false;
  }
  double r_, u_, p_;
  double head, tail;
  if (gt_pos(ps, p_s)) {   // shock
    head = tail = v_s + quot(W_s, rs, ir);
  } else {
    double unused;
    head = v_s + root(quot(gs.gamma * p_s, rs, ir), unused);
    tail = head;
    if (positive(head)) tail = v_star + root(quot(gs.gamma * ps, rstar, irstar), unused);
  }
  if (!positive(head)) {
    r_ = rs; u_ = u_s; p_ = p_s;
  } else if (positive(tail)) {
    r_ = rstar; u_ = us; p_ = ps;
  } else {
    const double w = head / (head - tail);
    r_ = rs + w * (rstar - rs);
    u_ = u_s + w * (us - u_s);
    p_ = p_s + w * (ps - p_s);
  }
  const double f0 = r_ * u_;
  F[0] = f0;
  F[1] = f0 * u_ + p_;
  F[2] = f0 * t1;
  F[3] = f0 * t2;
  const double E = p_ * gs.inv_gm1 + (0.5 * r_) * (u_ * u_ + (t1 * t1 + t2 * t2));
  F[4] = u_ * (E + p_);
  if constexpr (NQ > 5) {
    F[5] = f0 * pick(left, L[5], R[5]);
    *uf = u_;
  }
  return true;
}

template <int NQ>
CELLO_HD void two_shock_flux(const double L[NQ], const double R[NQ], const Gas<double>& gs, double F[NQ],
                             double* uf = nullptr) {
  if (!two_shock<NQ>(L, R, gs, F, uf)) riemann_flux<double, NQ>(L, R, gs, F, uf);
}

// The iteration of two_shock with every pressure and both W of it kept (hp, hL,
// hR; entry `last` is the final one) and bit k of floored set where pressure k
// came from the floor; raw0 is pressure 0 before its floor.  A pressure that
// returns after two steps fills the rest from the two before, the first of which
// is entry `turn` (-1: none does).
CELLO_HD bool shock_history(const double L[5], const double R[5], const Gas<double>& gs, double hp[], double hL[],
                            double hR[], unsigned& floored, int& last, int& turn, double& raw0, Side& l, Side& r) {
  turn = -1;
  if (!ordinary<5>(L, R, gs)) return false;
  l.set(L, gs);
  r.set(R, gs);
  const double Cs = l.C + r.C;
  raw0 = quot_any((r.C * l.p + l.C * r.p) + (l.C * r.C) * (l.u - r.u), Cs, rcp(Cs));
  floored = gt_pos(raw0, kPFloor) ? 0u : 1u;
  double ps = max_pos(raw0, kPFloor);
  last = 0;
#pragma unroll 1
  for (;; ++last) {
    if (!within<-68, 50>(high(ps)) || !l.at(ps, gs, false) || !r.at(ps, gs, true)) return false;
    hp[last] = ps;
    hL[last] = l.W;
    hR[last] = r.W;
    if (last == kRiemannIters) return true;
    const double zs = l.z + r.z;
    const double raw = fma(-2.0, quot_any((l.z * r.z) * (r.us - l.us), zs, rcp(zs)), ps);
    const double pn = max_pos(raw, kPFloor);
    if (!gt_pos(raw, kPFloor)) floored |= 2u << last;
    if (bits(pn) == bits(ps)) return true;
    ps = pn;
    if (last == 0 || bits(pn) != bits(hp[last - 1])) continue;
    const bool here = ((kRiemannIters - last) & 1) == 0;   // the last pressure is this one
    turn = last - 1;
    while (last < kRiemannIters) {
      ++last;
      hp[last] = hp[last - 2];
      hL[last] = hL[last - 2];
      hR[last] = hR[last - 2];
      floored |= (floored >> (last - 2) & 1u) << last;
    }
    return here || (l.at(ps, gs, false) && r.at(ps, gs, true));
  }
}

}  // namespace q64
}  // namespace cello
