// md_fx_coef.h -- the fixed-point pair kernel's coefficients (md_fx.cuh) of one
// type pair, computed on the host (plain C++).
#pragma once

#include <math.h>
#include <string.h>

#include "md_fx.cuh"

// A number as the unevaluated sum of two doubles (106 bits), for coefficients
// of more than 53 bits.  The product's error term is exact (one FMA).
struct MdDd {
  double h, l;
};
inline MdDd md_dd_mul(MdDd a, MdDd b) {
  const double p = a.h * b.h;
  const double e = fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
  const double h = p + e;
  return {h, e - (h - p)};
}
inline MdDd md_dd_div(MdDd a, MdDd b) {
  const double q = a.h / b.h;
  const double r = fma(-q, b.h, a.h) + (a.l - q * b.l);
  const double e = r / b.h;
  const double h = q + e;
  return {h, e - (h - q)};
}
// a 2^s rounded to an integer
inline long long md_dd_fixed(MdDd a, int s) {
  const double h = ldexp(a.h, s), f = floor(h);
  return (long long)f + llrint((h - f) + ldexp(a.l, s));
}

// An atom that may receive kmax contributions: its sums hold 2^11 of the largest,
// 2^(MD_FIX_EMAX + 1) each, without overflow.  The power of two by which the
// contributions have to be smaller where there may be more.
inline int md_fx_dense(unsigned int kmax) {
  int kb = 0;
  while (kb < 31 && (kmax >> kb)) kb++;
  const int d = kb - (63 - MD_FIX_BITS - (MD_FIX_EMAX + 1));
  return d > 0 ? d : 0;
}

// Eq. 1's fixed-point coefficients of one type pair (md_fx.cuh).
// qq, rc_coul: the Coulomb term (rc_coul <= 0: none).  only: the context's only
// pair type, without a Coulomb term (the one-type form where B allows it).
// dense: see md_fx_dense.
inline void md_set_fx(PairFx& p, bool only, int dense, double eps, double sigma, double rc, int R,
                      double lmax, double qq, double rc_coul) {
  memset(&p, 0, sizeof(p));
  // exact sigma^2 as m 2^e, m < 2^106
  int es = 0;
  const unsigned __int128 ms = (unsigned long long)ldexp(frexp(sigma, &es), 53);
  const unsigned __int128 m = ms * ms;
  const int e = 2 * (es - 53);
  // m 2^(e + s), rounded, for results below 2^63
  auto scaled = [&](int s) {
    const int sh = -(e + s);
    if (sh <= 0) return (unsigned long long)(m << -sh);
    if (sh > 110) return 0ULL;
    return (unsigned long long)((m + ((unsigned __int128)1 << (sh - 1))) >> sh);
  };
  const double ratio = ldexp(1.0, 2 * R) / (sigma * sigma);  // 4^R / sigma^2
  p.e2 = 2.0 * eps;
  p.smin = ~0u;  // nothing in fixed point
  // cutoff band: r^2 here (3 units, positions within 2^-53), fma(dz,dz,
  // fma(dy,dy, dx*dx)) on FP64 separations of coordinates up to 1.25 lmax
  const double su = ldexp(1.0, 62 - 2 * R);
  bool narrow = true;
  auto bounds = [&](double r, unsigned int& lo, unsigned int& hi) {
    const double sc = r * r * su, band = ldexp(sc, -44) + r * lmax * ldexp(su, -47) + 64.0;
    lo = sc - band > 0.0 ? (unsigned int)floor(ldexp(sc - band, -32)) : 0u;
    hi = sc + band < ldexp(1.0, 63) ? (unsigned int)ceil(ldexp(sc + band, -32)) : ~0u;
    narrow = narrow && band < 0.25 * sc;
  };
  bounds(rc, p.cut_lo, p.cut_hi);
  if (rc_coul > 0.0) bounds(rc_coul, p.cc_lo, p.cc_hi);
  if (!(ratio < ldexp(1.0, 40)) || !(ratio > ldexp(1.0, -2)) || !narrow) return;
  // largest tau with |F| below the accumulators' range for every smaller one
  // (|F| = 24 eps / sigma tau^3.5 |2 tau^3 - 1|, largest of the attractive
  // branch 2.397 eps / sigma at tau^3 = 7 / 26)
  const double fs = 24.0 * eps / sigma, flim0 = ldexp(1.0 - ldexp(1.0, -10), MD_FIX_EMAX + 1 - dense);
  const bool coul = rc_coul > 0.0 && qq != 0.0;  // each term then gets half the range
  const double flim = coul ? 0.5 * flim0 : flim0;
  auto force = [&](double t) { return fs * pow(t, 3.5) * fabs(2.0 * t * t * t - 1.0); };
  const double ta = pow(7.0 / 26.0, 1.0 / 3.0);
  double lo = 0.0, hi = MD_FX_TAU_MAX;
  if (force(ta) > flim) {
    hi = ta;
  } else if (force(hi) <= flim) {
    lo = hi;
  } else {
    lo = ta;
  }
  for (int k = 0; k < 60 && lo < hi; k++) {
    const double mid = 0.5 * (lo + hi);
    (force(mid) <= flim ? lo : hi) = mid;
  }
  double tl = lo * (1.0 - 1e-9);
  if (coul && fabs(qq) * tl > flim * sigma * sigma) tl = flim * sigma * sigma / fabs(qq);
  if (!(tl > 1e-3)) return;
  // general form: largest |w| over tau < tl, w = tau^3 (2 tau^3 - 1), at tl or, on
  // the attractive branch, at tau^3 = 1/4 (-1/8); |w| < 2^we
  const double tw = cbrt(0.25);
  auto wabs = [](double t) { return t * t * t * fabs(2.0 * t * t * t - 1.0); };
  int we = 0;
  frexp(1.001 * (tl > tw && wabs(tw) > wabs(tl) ? wabs(tw) : wabs(tl)), &we);
  p.zsh = 6 - we;
  const MdDd s2 = md_dd_mul({sigma, 0.0}, {sigma, 0.0}), s6 = md_dd_mul(s2, md_dd_mul(s2, s2));
  const MdDd c6 = md_dd_mul(md_dd_mul({24.0, 0.0}, {eps, 0.0}), s6);
  const MdDd cc = md_dd_div(md_dd_mul({24.0, 0.0}, {eps, 0.0}), s2);  // C
  int ce = 0;
  frexp(cc.h, &ce);
  const int cx = 63 - ce;
  p.cm = md_dd_fixed(cc, cx);
  p.sh = cx - 9 + p.zsh - 45 - R;
  if (p.sh > 12) {  // small forces: more bits than the counts can use
    const int d = p.sh - 12;
    p.cm = d < 62 ? p.cm >> d : 0;
    p.sh = 12;
  }
  if (coul) {
    // |fpair| <= |F| / r: keep both terms below 2^61 in units of 2^-p
    const int pm = (int)floor(61.0 - log2(flim * sqrt(tl) / sigma)), pp = p.sh + 45 + R;
    if (pp > pm) {
      p.cm >>= pp - pm < 62 ? pp - pm : 62;
      p.sh -= pp - pm;
    }
    int qe = 0;
    frexp(qq, &qe);
    p.cq = md_dd_fixed({qq, 0.0}, 62 - qe);
    p.csh = 62 - qe - 9 + 3 * R - (p.sh + 45 + R);
    if (p.csh < -24) return;
    if (p.csh > 62) {  // the term is far below P's unit
      p.cq = 0;
      p.csh = 62;
    }
  }
  if (p.sh < 1) return;
  p.B = 0;
  while (ldexp(1.0, p.B) < 1.001 * tl * ratio) p.B++;  // tau's scale: tl, small for stiff pairs
  if (p.B <= MD_FX_BMAX) {
    const double q = ldexp(1.0, p.B) / ratio;  // between tl and 2.1 tl where B > 0
    // C q^4 = 24 eps sigma^6 2^(4B - 8R) = kf 2^ke; k2 in [2^55, 2^56], k1 = 4 k2 q^3
    int ke = 0;
    frexp(ldexp(c6.h, 4 * p.B - 8 * R), &ke);
    p.k2 = md_dd_fixed(c6, 4 * p.B - 8 * R + 56 - ke);
    p.k1 = md_dd_fixed(md_dd_mul(c6, s6), 4 * p.B - 8 * R + 56 - ke + 2 + 3 * p.B - 6 * R);
    // |w| = 4 k2 (tau / q)^3 |2 tau^3 - 1| < 2^58 wmax
    double wmax = 0.0;
    for (int k = 1; k <= 256; k++) {
      const double t = tl * k / 256.0, x = t / q;
      wmax = fmax(wmax, x * x * x * fabs(2.0 * t * t * t - 1.0));
    }
    frexp(wmax * 1.02, &we);
    p.zsh1 = 5 - we < 0 ? 0 : 5 - we;  // |w 2^zsh1| < 2^63
    p.sh1 = 57 + p.zsh1 - ke - 45 - R;  // P = fpair 2^(57 + zsh1 - ke)
    if (p.sh1 > 12) {
      const int d = p.sh1 - 12;
      p.k1 = d < 62 ? p.k1 >> d : 0;
      p.k2 = d < 62 ? p.k2 >> d : 0;
      p.sh1 = 12;
    }
    if (p.sh1 < 1) p.B = MD_FX_BMAX + 1;  // the general form
  }
  // The general form is exact to some units of 2^-57 on the scale of tau = 1,
  // 24 eps / sigma of them in a contribution near sigma; beyond 2^9 eps / sigma
  // that would pass a count (the one-type form's scale follows tl)
  if (!(only && p.B <= MD_FX_BMAX) && eps > 512.0 * sigma) return;
  int c = 0;
  while (scaled(c + 1 - 2 * R) < (1ULL << 63)) c++;  // sigma^2 / 4^R 2^c in [2^62, 2^63)
  p.csign = scaled(c - 2 * R);
  p.tsh = c - 62;
  // (a stiff pair whose force leaves the range beyond 2^R: nothing in fixed point)
  const double smin = ceil(ldexp(1.0, 30) / (ratio * tl)) + 1.0;
  if (smin < 4294967295.0) p.smin = (unsigned int)smin;
}
