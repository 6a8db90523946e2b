// md_fx.cuh -- Eq. 1's pair force in 64-bit fixed point (integer
// instructions only), for the FP64 contexts' fixed-point pair kernel
// (md_pair_fx.cuh).
//
// GB300 issues one FP64 instruction per 64 cycles and scheduler (2 lanes per
// clock and SM), but a 32 x 32 + 64 -> 64-bit multiply-add every two cycles.
// A truncated 64-bit high product is three of those, so a force evaluated in
// 60-odd-bit fixed point costs fewer cycles than its eight FP64 operations,
// and it is more exact: the errors below are absolute ones of 2^-50 and less
// against the 2^-44 unit in which the force contributions are summed.
//
// Number formats (R: the largest cutoff is at most 2^R):
//   A   = d 2^(63 - R) per axis          separation, |A| < 2^63
//   S   = r^2 2^(62 - 2R)                squared distance, < 2^62 inside rc
//   T   = t 2^(63 - B), t = 4^R / r^2    t < 2^B
//   P   = fpair 2^p                      F_i = -fpair d
// and a contribution's count is P A 2^(44 - p - 63 + R), rounded.  Over
// liquid separations the force is 1.4 times closer to the exact one than the
// same formula in FP64 (rms over r uniform in 0.82 .. 2.5, random directions:
// 0.58 against 0.82 units of 2^-44).
// Pairs outside these ranges (closer than 0.816 sigma, forces beyond the
// accumulators' range, md_fx_dense, within a band around a cutoff, positions without a
// fixed-point form) are evaluated in FP64 by the caller.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MD_HD __host__ __device__ __forceinline__
#else
#define MD_HD inline
#endif

// The force accumulators' unit is 2^-MD_FIX_BITS.
#define MD_FIX_BITS 44
// Largest binary exponent e of a contribution 2^e <= |g| that may go to a
// fixed-point accumulator: |g| < 2^(MD_FIX_EMAX + 1) keeps the conversion a
// right shift.
#define MD_FIX_EMAX 7

// Per type pair; built on the host (md_set_fx).
struct PairFx {
  // high words of S: at or below smin FP64 path (r or the force out of range),
  // below cut_lo inside the cutoff, above cut_hi outside; between the last two
  // the FP64 path decides
  unsigned int smin, cut_lo, cut_hi;
  // one-type form, with q = 2^B sigma^2 / 4^R and C = 24 eps / sigma^2:
  long long k2;               // C q^4 2^(p - 1 - zsh1), p = sh1 + 45 + R; below 2^56
  long long k1;               // 4 k2 q^3, below 2^63
  int B, zsh1, sh1;           // 4^R / r^2 < 2^B for S > smin, B <= MD_FX_BMAX
  // general form (S normalized per pair):
  int zsh, sh;                // |w 2^(57 + zsh)| < 2^63; as sh1
  int tsh;                    // c - 62
  unsigned long long csign;   // sigma^2 / 4^R 2^c, in [2^62, 2^63)
  long long cm;               // C = cm 2^-(p + 9 - zsh), in [2^62, 2^63)
  double e2;                  // 2 eps
  // lj/cut/coul/cut (general form): rc_coul's bounds as cut_lo, cut_hi, and
  // qq = cq 2^-x in 62 bits with csh = x - 9 + 3R - p
  unsigned int cc_lo, cc_hi;
  long long cq;
  int csh;
};

#define MD_FX_BMAX 7

// Largest tau = sigma^2 / r^2 of the fixed-point path: tau^3 (2 tau^3 - 1) and
// tau^4 (2 tau^3 - 1) then stay below 2^4.3 and 2^4.9.
#define MD_FX_TAU_MAX 1.5

// Dropped terms would bias every product the same way, and a bias survives the
// sums over pairs: each function below adds their mean.

// (a b) >> 64 for a, b < 2^63, within 1.25 units (the low halves' product and
// the cross terms' fraction are dropped, their mean is 0.75).
MD_HD unsigned long long md_mulhi_u(unsigned long long a, unsigned long long b) {
  const unsigned int a1 = (unsigned int)(a >> 32), a0 = (unsigned int)a;
  const unsigned int b1 = (unsigned int)(b >> 32), b0 = (unsigned int)b;
  unsigned long long t = (unsigned long long)a1 * b0 + 0xc0000000ULL;
  t = (unsigned long long)a0 * b1 + t;  // < 2^64: a1, b1 < 2^31
#ifdef __CUDA_ARCH__  // an add with carry (the C form moves t >> 32 into a register pair)
  unsigned long long r = (unsigned long long)a1 * b1;
  asm("{.reg .u32 l, h, tl, th; mov.b64 {l, h}, %0; mov.b64 {tl, th}, %1;"
      " add.cc.u32 l, l, th; addc.u32 h, h, 0; mov.b64 %0, {l, h};}"
      : "+l"(r)
      : "l"(t));
  return r;
#else
  return (unsigned long long)a1 * b1 + (t >> 32);
#endif
}

// The same for signed a, b (|a|, |b| < 2^63): the low halves enter with 31
// bits so that every product is a signed 32 x 32 one.  Within 2.25 units.
MD_HD long long md_mulhi_s(long long a, long long b) {
  const int a1 = (int)(a >> 32), a0 = (int)((unsigned int)a >> 1);
  const int b1 = (int)(b >> 32), b0 = (int)((unsigned int)b >> 1);
  long long t = (long long)a1 * b0 + 0x60000000LL;
  t = (long long)a0 * b1 + t;
  return (long long)a1 * b1 + (t >> 31);
}

// S = (Ax^2 + Ay^2 + Az^2) / 2^64, within 2.5 units (even A).
// (The cross sum overflows only for |dx| + |dy| + |dz| >= 2^(R + 1), where S
// is above 2^62 whatever its low bits.)
MD_HD unsigned long long md_fx_r2(long long Ax, long long Ay, long long Az) {
  const int x1 = (int)(Ax >> 32), y1 = (int)(Ay >> 32), z1 = (int)(Az >> 32);
  const int x0 = (int)((unsigned int)Ax >> 1), y0 = (int)((unsigned int)Ay >> 1),
            z0 = (int)((unsigned int)Az >> 1);
  unsigned long long t = (unsigned long long)((long long)x1 * x0) + (3ULL << 29);
  t += (unsigned long long)((long long)y1 * y0);
  t += (unsigned long long)((long long)z1 * z0);
  unsigned long long s = (unsigned long long)((long long)t >> 30);
  s += (unsigned long long)((long long)x1 * x1);
  s += (unsigned long long)((long long)y1 * y1);
  s += (unsigned long long)((long long)z1 * z1);
  return s;
}

// T = (2^62 / S) 2^(63 - B) for 2^(62 - B) < S, B <= 7.  y: an approximation
// of 2^32 / S within 2^-22.6 relative (the FP32 reciprocal of S rounded to
// FP32).  Y0 = y scaled to 31 bits; e = 1 - S Y0 / 2^(93 - B), |e| < 2^-22,
// is formed exactly to 2^-53 (E32), and 1 / (1 - e) ~ 1 + e + e^2 (Markstein,
// IBM J. Res. Dev. 34 (1990) 111): the result is within 2^-53 relative.
MD_HD unsigned long long md_fx_rcp(unsigned long long S, unsigned int Y0, int B) {
  const unsigned int s1 = (unsigned int)(S >> 32), s0 = (unsigned int)S;
  const unsigned long long lo = (unsigned long long)s0 * Y0;
  const unsigned long long ph = (unsigned long long)s1 * Y0 + (lo >> 32);
  const long long e = (long long)((1ULL << (61 - B)) + (1ULL << (7 - B)) - ph);
  int c = (int)(e >> (8 - B));  // e 2^53, rounded
  const int h = c >> 16;
  c += (h * h + (1 << 20)) >> 21;
  return ((unsigned long long)Y0 << 32) +
         (unsigned long long)(((long long)(int)Y0 * c) >> 21);
}

// rho 2^60 with rho = (2^62 / S)^(1/2) for 2^58 <= S < 2^62 (rho <= 4), from
// Y0 = rho 2^28 within 2^-22 relative: e = 1 - S Y0^2 / 2^118 and the series
// (1 - e)^(-1/2) ~ 1 + e / 2 + 3 e^2 / 8; within 2^-53 relative.
MD_HD unsigned long long md_fx_rsqrt(unsigned long long S, unsigned int Y0) {
  const unsigned long long Q = (unsigned long long)Y0 * Y0;  // <= 2^60
  const long long e = (long long)((1ULL << 56) - md_mulhi_u(S, Q << 2));
  int c = (int)((e + 8) >> 4);  // e 2^52
  const int h = c >> 16;
  c += (3 * h * h + (1 << 21)) >> 22;
  return ((unsigned long long)Y0 << 32) +
         (unsigned long long)(((long long)(int)Y0 * c) >> 21);
}

// P of the Coulomb term: qq rho t 8^(k - R) 2^p with rho t 2^55 in v.
MD_HD long long md_fx_coul(unsigned long long rho, unsigned long long T, const PairFx& c, int k) {
  const unsigned long long v = md_mulhi_u(rho, T << 1);
  const long long f = md_mulhi_s(c.cq, (long long)v);
  const int s = c.csh - 3 * k;
  return s > 0 ? (f + (1LL << (s - 1))) >> s : f << -s;
}

// P of the one-type form, five products.  With x = T 2^-63 (tau = q x):
// T2 = x^2 2^62, x3 = x^3 2^62, u = k2 (2 tau^3 - 1) (below 2^59), w = 4 x^3 u.
MD_HD long long md_fx_force1(unsigned long long T, const PairFx& c, unsigned long long& x3) {
  const unsigned long long T2 = md_mulhi_u(T, T);
  x3 = md_mulhi_u(T2 << 1, T);
  const long long u =
      (long long)md_mulhi_u((unsigned long long)c.k1, x3 << 1) - c.k2;
  const long long w = md_mulhi_s((long long)(x3 << 1), u << 3);
  return md_mulhi_s((long long)T, w << c.zsh1);
}

// The general form, from tau 2^62: tau^3 2^59, w = tau^3 (2 tau^3 - 1) 2^57 and
// P = cm tau w.  (w is shifted before the product with tau, not after it: its
// error then counts for far pairs with their small tau.)
struct FxForce {
  unsigned long long tau3;
  long long w;
  long long P;
};
MD_HD FxForce md_fx_force(unsigned long long tau, long long cm, int zsh) {
  FxForce r;
  const unsigned long long tau2 = md_mulhi_u(tau, tau);  // 2^60
  r.tau3 = md_mulhi_u(tau2 << 1, tau);                   // 2^59
  const long long u = (long long)(r.tau3 << 2) - (1LL << 60);  // (2 tau^3 - 1) 2^60
  r.w = md_mulhi_s((long long)(r.tau3 << 2), u);               // 2^61 2^60 / 2^64
  r.P = md_mulhi_s(cm, md_mulhi_s((long long)tau, r.w << zsh));  // z 2^(55 + zsh)
  return r;
}

// The count of one component: P A / 2^64 rounded to a multiple of 2^sh and
// shifted (the constant also makes up for the dropped product of the low halves).
MD_HD long long md_fx_count(long long P, long long A, int sh) {
  const int p1 = (int)(P >> 32), p0 = (int)((unsigned int)P >> 1);
  const int a1 = (int)(A >> 32), a0 = (int)((unsigned int)A >> 1);
  long long t = (long long)p1 * a0 + ((1LL << (30 + sh)) + 0x20000000LL);
  t = (long long)p0 * a1 + t;
  return ((long long)p1 * a1 + (t >> 31)) >> sh;
}
