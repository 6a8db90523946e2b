// Evaluates the fixed-point pair force on the host as the kernel does (the
// decision between fixed point and FP64, then the counts), over coefficients and
// separations read from stdin, and reports every contribution that is out of
// the accumulators' range or off the exact force (128-bit floats).
//
// One line per pair type: eps sigma rc rcmax lmax qq rc_coul samples dense
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "md_fx_coef.h"

#ifdef __SIZEOF_FLOAT128__
typedef __float128 Q;
#else
typedef long double Q;  // 128 bits on Arm
#endif
static_assert(sizeof(Q) == 16, "");

static Q q_scale(Q x, int e) {
  for (; e > 0; e--) x *= 2;
  for (; e < 0; e++) x /= 2;
  return x;
}
static Q q_sqrt(Q x) {
  Q y = (Q)std::sqrt((double)x);
  for (int k = 0; k < 3; k++) y = (y + x / y) / 2;
  return y;
}
static double next_uniform(unsigned long long& s) {
  unsigned long long z = (s += 0x9e3779b97f4a7c15ULL);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return (double)((z ^ (z >> 31)) >> 11) * 0x1p-53;
}

int main() {
  double eps, sigma, rc, rcmax, lmax, qq, rcc;
  int samples, dense;
  unsigned long long seed = 1;
  while (scanf("%lf %lf %lf %lf %lf %lf %lf %d %d", &eps, &sigma, &rc, &rcmax, &lmax, &qq, &rcc,
               &samples, &dense) == 9) {
    int R;
    if (std::frexp(rcmax, &R) == 0.5) R--;
    const bool coul = rcc > 0.0;
    PairFx forms[2];  // the only type, and one of several
    for (int form = 0; form < 2; form++)
      md_set_fx(forms[form], form == 0 && !coul, dense, eps, sigma, rc, R, lmax, qq, rcc);
    int fixed = 0, bad = 0, in_range = 0;
    double worst = 0.0, rlow = 1e300;
    const double rmax = coul && rcc > rc ? rcc : rc;
    for (int it = 0; it < samples; it++) {
      const double r = rmax * (0.2 + 0.8 * next_uniform(seed));
      const double ct = 2.0 * next_uniform(seed) - 1.0, ph = 6.283185307 * next_uniform(seed);
      const double st = std::sqrt(1.0 - ct * ct);
      const double d[3] = {r * st * std::cos(ph), r * st * std::sin(ph), r * ct};
      for (int form = 0; form < 2; form++) {
        const PairFx& c = forms[form];
        const bool single = form == 0;  // the one-type form, or the general one
        if (single && (coul || c.B > MD_FX_BMAX)) continue;
        long long A[3];
        for (int k = 0; k < 3; k++) A[k] = (long long)std::ldexp(d[k], 63 - R - 8) * 256;
        int k = 0;
        if (!single) {
          unsigned int any = 0;
          for (int q = 0; q < 3; q++) {
            const int h = (int)(A[q] >> 32);
            any |= (unsigned int)(h ^ (h >> 31));
          }
          k = (any ? __builtin_clz(any) : 32) - 2;
          if (k < 0) k = 0;
          for (int q = 0; q < 3; q++) A[q] = (long long)((unsigned long long)A[q] << k);
        }
        const unsigned long long Sn = md_fx_r2(A[0], A[1], A[2]);
        const unsigned long long S = single ? Sn : (2 * k < 64 ? Sn >> (2 * k) : 0);
        const unsigned int S1 = (unsigned int)(S >> 32);
        const bool in_lj = S1 < c.cut_lo, in_co = coul && S1 < c.cc_lo;
        if (in_lj || in_co) in_range++;
        // the FP64 path, or no force
        if (S1 <= c.smin || (!in_lj && S1 <= c.cut_hi) ||
            (coul && !in_co && S1 <= c.cc_hi) || !(in_lj || in_co))
          continue;
        fixed++;
        if (r < rlow) rlow = r;
        const float sf = (float)(unsigned int)Sn * 0x1p-32f + (float)(unsigned int)(Sn >> 32);
        const int B = single ? c.B : 5;
        unsigned long long T, rho = 0, x3;
        if (coul) {
          rho = md_fx_rsqrt(Sn, (unsigned int)std::nearbyint((1.0f / std::sqrt(sf)) * 0x1p43f));
          T = md_mulhi_u(rho, rho) << 2;
        } else {
          T = md_fx_rcp(Sn, (unsigned int)std::nearbyint(std::ldexp(1.0f / sf, 61 - B)), B);
        }
        long long P = single ? md_fx_force1(T, c, x3)
                             : md_fx_force(((md_mulhi_u(T, c.csign) >> (c.tsh - 2 * k)) << 6) + 32,
                                           c.cm, c.zsh).P;
        if (coul) P = (in_lj ? P : 0) + (in_co ? md_fx_coul(rho, T, c, k) : 0);
        Q e[3], r2 = 0;
        for (int q = 0; q < 3; q++) {
          e[q] = q_scale((Q)A[q], R - 63 - k);
          r2 += e[q] * e[q];
        }
        const Q x2 = (Q)sigma * (Q)sigma / r2, x6 = x2 * x2 * x2;
        Q f = in_lj ? (Q)24 * (Q)eps * x6 * (2 * x6 - 1) / r2 : (Q)0;
        Q mag = in_lj ? (Q)24 * (Q)eps * x6 * (2 * x6 + 1) / r2 : (Q)0;
        if (in_co) {
          const Q g = (Q)qq / (r2 * q_sqrt(r2));
          f += g;
          mag += g < 0 ? -g : g;
        }
        for (int q = 0; q < 3; q++) {
          const long long n = md_fx_count(P, A[q], single ? c.sh1 : c.sh + k);
          const double off = std::fabs((double)((Q)n - q_scale(f * e[q], MD_FIX_BITS)));
          // one count for the rounding, 2^-46 of the magnitude for the arithmetic
          const double tol = 1.0 + (double)q_scale(mag * (e[q] < 0 ? -e[q] : e[q]),
                                                   MD_FIX_BITS - 46);
          if (off / tol > worst) worst = off / tol;
          if (!(off <= tol) || std::llabs(n) >= 1LL << (MD_FIX_BITS + MD_FIX_EMAX + 1 - dense)) bad++;
        }
      }
    }
    printf("%d %d %d %.6g %.17g %u\n", bad, fixed, in_range, worst, rlow, forms[0].smin);
  }
  return 0;
}
