// md_pair_fx.cuh -- the FP64 contexts' fixed-point pair kernel (arXiv
// 2508.13523, Eq. 1 and Sec. 4; Sec. 4.1: half list with reductions, full
// list, T threads per atom).
//
// Positions are 64-bit fixed-point numbers (XFix), separations their
// differences, Eq. 1's force is evaluated in 64-bit fixed point (md_fx.cuh)
// and every contribution is a 2^-44 count summed exactly in 64-bit integers:
// the owner's share in registers, f_j's (half list) by global integer
// reductions.  No FP64 instruction per pair, so the FP64 pipe (64 cycles per
// instruction and scheduler) no longer decides, and a pair costs little
// enough that lanes need not be repacked: each lane walks its own row.
//
// The row's skin part (pairs outside rc at the build) goes first, through an
// FP32 test against a certified upper bound of rc^2 that needs 16 bytes per
// entry; the few survivors wait in the lane's shared-memory slots and are
// then taken after the inner entries, so that the force code runs for lanes
// that almost all have a pair inside rc.
//
// What bounds it (864,000 atoms, half list, ncu): the multiply-add pipe 68 %,
// issue 64 %, L1 62 % and L2 54 % busy, no one of them alone; 240 warp
// instructions per 32 pairs against 560 in the kernel it replaced (8 FP64
// operations per pair, in-range pairs repacked through per-warp queues, owner
// sums in shared memory).  Per launch inside a step, before and after: half
// list 4,000,000 atoms 2.34 -> 1.46 ms, 32,000 atoms 63 -> 23 us; full list
// 256,000 atoms 355 -> 180 us; with energy and virial, half list, 4,000,000
// atoms 2.95 -> 1.76 ms.  Tried and left
// out: the next record's gather one pair ahead (8 more registers, 4 % slower),
// and dealing the entries above the warp's mean row length to its idle lanes
// (22 % fewer rounds, but the owner's position and box become variables: no
// gain at 4,000,000 atoms, 8 % slower at 256,000).  Slower than what it replaced
// where most forces leave the sums' range, eps / sigma of 100 and more: 32,000
// atoms, eps 100 half 78.5 -> 79.5, full 127.7 -> 135 us a step.
//
// Cutoff decisions are the oracle's: the fixed-point r^2 decides outside a
// band around rc^2 that covers both its own error and that of
// fma(dz,dz, fma(dy,dy, dx*dx)) on FP64 separations; inside it, and for pairs
// that the fixed-point force does not cover (r < 0.816 sigma; forces beyond
// the accumulators' range, which with eps = sigma = 1 begins at r = 0.865 and on
// lists of more than 2^11, 2^12 and 2^13 stencil candidates at 0.905, 0.945 and
// 0.985; an atom without a fixed-point position),
// md_pair_fx_slow evaluates the pair in FP64.
#pragma once

#include "md_device.cuh"
#include "md_fx.cuh"
#include "md_internal.cuh"
#include "md_pair.cuh"

#define MD_FX_SLOTS 8  // skin survivors that wait per lane

// Sums of one pair taken in FP64.
struct FxSlow {
  long long q[3];  // counts for atom j (owner: minus these)
  double e;        // energy, or r^-6 with one type (Eq. 1 alone)
  double s[3];     // image shift taken off d
  double g[3];     // fpair d
  int in;
};

// The pair (i, j) in FP64, as the oracle evaluates it.  Contributions beyond
// the accumulators' range are added to f here; the others are returned.
template <bool HALF, bool EV, bool SINGLE, bool COUL>
__device__ __noinline__ void md_pair_fx_slow(const PairArgs& a, const PairCoef* coef, int64_t i,
                                             int j, FxSlow& o) {
  const int64_t n = a.n;
  // range of the accumulators (MD_FIX_BITS)
  const int kb = 32 - __clz((int)min(*a.kmax, 0x7fffffffu));
  const int ex_lim = min(1023 + MD_FIX_EMAX + 1, 1023 + 63 - MD_FIX_BITS - kb);
  const double4_32a xi = md_ld4(a.x4 + i), xj = md_ld4(a.x4 + j);
  const int tag = md_tag_of(xi);
  const RepGeo* g = a.rep + MD_TAG_REP(tag);
  const PairCoef& c = coef[SINGLE ? 0 : MD_TAG_TYPE(tag) * a.nt + md_type_of(xj)];
  const double ex = __dsub_rn(xj.x, xi.x), ey = __dsub_rn(xj.y, xi.y), ez = __dsub_rn(xj.z, xi.z);
  const double dx = md_min_image(ex, g->L[0], g->halfL_bits[0]);
  const double dy = md_min_image(ey, g->L[1], g->halfL_bits[1]);
  const double dz = md_min_image(ez, g->L[2], g->halfL_bits[2]);
  const double r2 = md_r2(dx, dy, dz);
  o.q[0] = o.q[1] = o.q[2] = 0;
  o.in = md_lt_pos(r2, COUL ? c.cutmax_bits : c.cutsq_bits);
  if (!o.in) return;
  double r2inv, r6inv, fpair, qr = 0.0;
  if (COUL) {  // Eq. 1 below rc, plus qq / r below rc_coul
    const double rinv = md_rsqrt(r2);
    r2inv = rinv * rinv;
    r6inv = r2inv * r2inv * r2inv;
    const double flj = r6inv * (c.lj1 * r6inv - c.lj2) * r2inv;
    qr = md_lt_pos(r2, c.cutsq_coul_bits) ? c.qq * rinv : 0.0;
    fpair = __fma_rn(qr, r2inv, md_lt_pos(r2, c.cutsq_bits) ? flj : 0.0);
  } else {
    r2inv = md_rcp(r2);
    r6inv = r2inv * r2inv * r2inv;
    fpair = r6inv * (c.lj1 * r6inv - c.lj2) * r2inv;
  }
  const double gx = fpair * dx, gy = fpair * dy, gz = fpair * dz;
  if (!(md_fix(gx, ex_lim, o.q[0]) & md_fix(gy, ex_lim, o.q[1]) & md_fix(gz, ex_lim, o.q[2]))) {
    o.q[0] = o.q[1] = o.q[2] = 0;
    if (a.fmark) *(volatile int*)a.fmark = 1;
    atomicAdd(a.f + i, md_neg(gx));
    atomicAdd(a.f + n + i, md_neg(gy));
    atomicAdd(a.f + 2 * n + i, md_neg(gz));
    if (HALF) {
      atomicAdd(a.f + j, gx);
      atomicAdd(a.f + n + j, gy);
      atomicAdd(a.f + 2 * n + j, gz);
    }
  }
  if (EV) {
    o.e = SINGLE ? r6inv : r6inv * (c.lj3 * r6inv - c.lj4);
    if (COUL) o.e = (md_lt_pos(r2, c.cutsq_bits) ? o.e : 0.0) + qr;
    o.s[0] = md_abs_gt(ex, g->halfL_bits[0]) ? copysign(g->L[0], ex) : 0.0;
    o.s[1] = md_abs_gt(ey, g->halfL_bits[1]) ? copysign(g->L[1], ey) : 0.0;
    o.s[2] = md_abs_gt(ez, g->halfL_bits[2]) ? copysign(g->L[2], ez) : 0.0;
    o.g[0] = gx;
    o.g[1] = gy;
    o.g[2] = gz;
  }
}

// Dynamic shared memory of the kernel: the tables of the types that there are
// (what FP64 pairs and energies need of PairCoef is read from global memory).
// What a block does not take stays L1, which the gathers live on.
inline size_t md_pair_fx_smem(bool single, int nt) {
  return single ? 0 : (sizeof(PairFx) + sizeof(float)) * (size_t)md_tab_entries(nt);
}

// The tile loop of the kernel: every block of the launch runs it (k_pair_fx,
// and the pair phase of k_step_fused).  All threads of the block must call
// it.  T lanes per atom; U: skin entries per round of the FP32 test, their
// gathers in flight together.
// COUL: lj/cut/coul/cut, in the general form.
template <bool HALF, bool EV, bool SINGLE, bool COUL, int T, int U>
__device__ __forceinline__ void md_pair_fx_tiles(const PairArgs& a, const float cut_hi1,
                                                 const float* __restrict__ cut_hi_tab) {
  static_assert(!(SINGLE && COUL), "the Coulomb style takes the general form");
  extern __shared__ double s_tab[];  // md_pair_fx_smem
  PairFx* sf = reinterpret_cast<PairFx*>(s_tab);
  float* scut = reinterpret_cast<float*>(sf + md_tab_entries(a.nt));
  __shared__ int sslot[MD_FX_SLOTS][MD_BLOCK];
  __shared__ double simg[EV ? 6 : 1][MD_BLOCK];  // the virial's image terms, own column
  __shared__ int s_tile;
  if (!SINGLE) {
    for (int k = threadIdx.x; k < a.nt * a.nt; k += blockDim.x) {
      sf[k] = a.fxt[k];
      scut[k] = cut_hi_tab[k];
    }
  }
  if (EV) {
#pragma unroll
    for (int k = 0; k < 6; k++) simg[k][threadIdx.x] = 0.0;
  }
  __syncthreads();
  const int64_t n = a.n;
  const int ntiles = (int)((n * T + MD_BLOCK - 1) / MD_BLOCK);
  for (int it = 0;; it++) {
    int64_t tile;
    if (a.tile_ctr) {
      if (threadIdx.x == 0) s_tile = md_next_tile(a.tile_ctr, a.nslots, ntiles);
      __syncthreads();
      tile = s_tile;
      __syncthreads();
    } else {
      tile = it == 0 ? (int64_t)blockIdx.x : -1;
    }
    if (tile < 0) break;
    const int64_t gid = tile * MD_BLOCK + threadIdx.x;
    const int64_t i = gid / T;
    const int t = (int)(gid % T);
    const bool active = i < n;
    const int64_t ia = active ? i : 0;
    const int nin = active ? __ldg(a.numneigh + ia) : 0;
    const int nsk = active ? __ldg(a.numneigh + n + ia) : 0;
    const int32_t* row = a.nbr + (ia >> 5) * (int64_t)a.maxneigh * 32 + (ia & 31) + t * 32;
    const XFix own = md_ld_xfix(a.xq + ia);
    const int tag = (int)own.w;
    const RepGeo* g = a.rep + MD_TAG_REP(tag);
    const int sh0 = 63 - a.fxR - (int)(own.w >> 32);  // D to A
    const unsigned gh = (unsigned)g->gh;
    long long ax = 0, ay = 0, az = 0;  // counts for the partners (owner: minus)
    unsigned long long s6 = 0;         // one type: sum x^3 2^(62 - ev_shift)
    double e0 = 0.0;                   // several types: energy; one type: r^-6 of FP64 pairs
    int npair = 0;
    bool img = false;  // this thread has image terms
    auto slow = [&](int j) {
      FxSlow o;
      md_pair_fx_slow<HALF, EV, SINGLE, COUL>(a, SINGLE ? &a.c1 : a.coef, ia, j, o);
      if (o.in) {
        ax += o.q[0];
        ay += o.q[1];
        az += o.q[2];
        if (HALF) {
          if (o.q[0]) atomicAdd(a.fix + j, (unsigned long long)o.q[0]);
          if (o.q[1]) atomicAdd(a.fix + n + j, (unsigned long long)o.q[1]);
          if (o.q[2]) atomicAdd(a.fix + 2 * n + j, (unsigned long long)o.q[2]);
        }
        if (EV) {
          e0 += o.e;
          npair++;
          img = true;
          double* m = &simg[0][threadIdx.x];
          m[0 * MD_BLOCK] = __fma_rn(-o.s[0], o.g[0], m[0 * MD_BLOCK]);
          m[1 * MD_BLOCK] = __fma_rn(-o.s[1], o.g[1], m[1 * MD_BLOCK]);
          m[2 * MD_BLOCK] = __fma_rn(-o.s[2], o.g[2], m[2 * MD_BLOCK]);
          m[3 * MD_BLOCK] = __fma_rn(-o.s[0], o.g[1], m[3 * MD_BLOCK]);
          m[4 * MD_BLOCK] = __fma_rn(-o.s[0], o.g[2], m[4 * MD_BLOCK]);
          m[5 * MD_BLOCK] = __fma_rn(-o.s[1], o.g[2], m[5 * MD_BLOCK]);
        }
      }
    };
    // inner entries, then the survivors
    auto pair = [&](int j, const XFix& o) {
      long long Dx = o.x - own.x, Dy = o.y - own.y, Dz = o.z - own.z;
      int shf = 0;  // EV: image shifts taken off d, 2 bits per axis (+L: 1, -L: 2)
      // |D| beyond 2^(R + F) or half the box on some axis: a periodic image
      // may be nearer (rare: only pairs across the boundary)
      auto far = [&](long long D) { return (unsigned)(int)(D >> 32) + gh >= 2u * gh; };
      if (far(Dx) | far(Dy) | far(Dz)) {
        // (x_j - x_i is rounded to FP64's 53 bits before the edge is taken
        // off, as the FP64 separation is)
        auto image = [&](long long& D, int k) {
          const long long L = g->Lx[k], h = g->hx[k];
          if (D > h || D < -h) {
            if (EV) shf |= (D < 0 ? 2 : 1) << (2 * k);
            const long long r = __double2ll_rn(__ll2double_rn(D));
            D = D < 0 ? r + L : r - L;
          }
          return (D >> (63 - sh0)) == (D >> 63);
        };
        if ((tag | (int)o.w) & MD_TAG_OFFGRID) {  // no fixed-point position
          slow(j);
          return;
        }
        if (!(image(Dx, 0) & image(Dy, 1) & image(Dz, 2))) return;  // beyond 2^R on some axis
      }
      long long Ax = Dx << sh0, Ay = Dy << sh0, Az = Dz << sh0;
      const PairFx& c = SINGLE ? a.fx1 : sf[MD_TAG_TYPE(tag) * a.nt + MD_TAG_TYPE((int)o.w)];
      int k = 0;
      if (!SINGLE) {  // normalize: the largest |A| to bit 61 (S's cross sum stays in range)
        const int x1 = (int)(Ax >> 32), y1 = (int)(Ay >> 32), z1 = (int)(Az >> 32);
        k = max(__clz((x1 ^ (x1 >> 31)) | (y1 ^ (y1 >> 31)) | (z1 ^ (z1 >> 31))) - 2, 0);
        Ax <<= k;
        Ay <<= k;
        Az <<= k;
      }
      const unsigned long long Sn = md_fx_r2(Ax, Ay, Az);
      const unsigned long long S = SINGLE ? Sn : (2 * k < 64 ? Sn >> (2 * k) : 0);
      const unsigned int S1 = (unsigned int)(S >> 32);
      const bool in_lj = S1 < c.cut_lo, in_co = COUL && S1 < c.cc_lo;
      if (COUL) {
        if ((S1 <= c.smin) | (!in_lj & (S1 <= c.cut_hi)) | (!in_co & (S1 <= c.cc_hi))) {
          slow(j);
          return;
        }
        if (!(in_lj | in_co)) return;
      } else if (!(S1 > c.smin & in_lj)) {
        if (S1 <= c.cut_hi) slow(j);
        return;
      }
      const float sfl = __fmaf_rn((float)(unsigned int)Sn, 0x1p-32f,
                                  (float)(unsigned int)(Sn >> 32));
      const int B = SINGLE ? c.B : 5;  // general: Sn >= 2^58
      float y;
      unsigned long long Tr, rho = 0;
      if (COUL) {
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(sfl));
        rho = md_fx_rsqrt(Sn, __float2uint_rn(y * 0x1p43f));
        Tr = md_mulhi_u(rho, rho) << 2;
      } else {
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(sfl));
        Tr = md_fx_rcp(Sn, __float2uint_rn(y * __int_as_float((127 + 61 - B) << 23)), B);
      }
      FxForce fo;  // tau3: one type: x^3 2^62 (md_fx_force1)
      if (SINGLE)
        fo.P = md_fx_force1(Tr, c, fo.tau3);
      else
        fo = md_fx_force(((md_mulhi_u(Tr, c.csign) >> (c.tsh - 2 * k)) << 6) + 32, c.cm, c.zsh);
      if (COUL) {
        fo.P = in_lj ? fo.P : 0;
        fo.P += in_co ? md_fx_coul(rho, Tr, c, k) : 0;
      }
      const int sh = SINGLE ? c.sh1 : c.sh + k;
      const long long qx = md_fx_count(fo.P, Ax, sh);
      ax += qx;
      if (HALF) atomicAdd(a.fix + j, (unsigned long long)qx);
      const long long qy = md_fx_count(fo.P, Ay, sh);
      ay += qy;
      if (HALF) atomicAdd(a.fix + n + j, (unsigned long long)qy);
      const long long qz = md_fx_count(fo.P, Az, sh);
      az += qz;
      if (HALF) atomicAdd(a.fix + 2 * n + j, (unsigned long long)qz);
      if (EV) {
        npair++;
        if (SINGLE)
          s6 += fo.tau3 >> a.ev_shift;
        else if (!COUL || in_lj)  // 4 eps (tau^6 - tau^3) = 2 eps (w - tau^3)
          e0 += c.e2 * 0x1p-57 * __ll2double_rn(fo.w - (long long)(fo.tau3 >> 2));
        if (COUL && in_co)  // qq / r = qq rho 2^(k - R)
          e0 += a.coef[MD_TAG_TYPE(tag) * a.nt + MD_TAG_TYPE((int)o.w)].qq *
                __ull2double_rn(rho) *
                __longlong_as_double((long long)(1023 - 60 + k - a.fxR) << 52);
        if (shf) {  // rare
          img = true;
          auto shift = [&](int k3) {
            const int b = (shf >> (2 * k3)) & 3;
            return b == 1 ? g->L[k3] : (b == 2 ? -g->L[k3] : 0.0);
          };
          const double sx = shift(0), sy = shift(1), sz = shift(2);
          const double gx = md_fold(qx), gy = md_fold(qy), gz = md_fold(qz);
          double* m = &simg[0][threadIdx.x];
          m[0 * MD_BLOCK] = __fma_rn(-sx, gx, m[0 * MD_BLOCK]);
          m[1 * MD_BLOCK] = __fma_rn(-sy, gy, m[1 * MD_BLOCK]);
          m[2 * MD_BLOCK] = __fma_rn(-sz, gz, m[2 * MD_BLOCK]);
          m[3 * MD_BLOCK] = __fma_rn(-sx, gy, m[3 * MD_BLOCK]);
          m[4 * MD_BLOCK] = __fma_rn(-sx, gz, m[4 * MD_BLOCK]);
          m[5 * MD_BLOCK] = __fma_rn(-sy, gz, m[5 * MD_BLOCK]);
        }
      }
    };
    // Rounds (almost always one): fill the lane's slots from the skin part,
    // take the inner entries (first round) and the slots.
    int left = nin > t ? (nin - t + T - 1) / T : 0;  // inner entries not yet taken
    int q = t;                                       // next skin entry
    do {
      int nsv = 0;
      {
        const float4 hi = md_ld_hi<0>(a.xs, ia);
        const float Lf0 = g->Lf[0], Lf1 = g->Lf[1], Lf2 = g->Lf[2];
        const float hf0 = g->halfLf[0], hf1 = g->halfLf[1], hf2 = g->halfLf[2];
        auto test = [&](int j, const float4& hj) {
          float dx = hj.x - hi.x, dy = hj.y - hi.y, dz = hj.z - hi.z;
          dx = fabsf(dx) > hf0 ? dx - copysignf(Lf0, dx) : dx;
          dy = fabsf(dy) > hf1 ? dy - copysignf(Lf1, dy) : dy;
          dz = fabsf(dz) > hf2 ? dz - copysignf(Lf2, dz) : dz;
          const float r2f = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, dx * dx));
          const float cut =
              SINGLE ? cut_hi1
                     : scut[MD_TAG_TYPE(tag) * a.nt + MD_TAG_TYPE(__float_as_int(hj.w))];
          if (r2f <= cut) sslot[nsv++][threadIdx.x] = j;
        };
        // entry s of the skin part is at k = maxneigh - 1 - s
        const int32_t* ps = row + (int64_t)(a.maxneigh - 1 - t - q) * 32;
        if (U == 2) {
          for (; q + T < nsk && nsv <= MD_FX_SLOTS - 2; q += 2 * T, ps -= 2 * T * 32) {
            const int j0 = __ldcs(ps), j1 = __ldcs(ps - T * 32);
            const float4 h0 = md_ld_hi<0>(a.xs, j0), h1 = md_ld_hi<0>(a.xs, j1);
            test(j0, h0);
            test(j1, h1);
          }
        }
        for (; q < nsk && (U == 1 || q + T >= nsk) && nsv < MD_FX_SLOTS; q += T, ps -= T * 32) {
          const int j = __ldcs(ps);
          test(j, md_ld_hi<0>(a.xs, j));
        }
      }
      const int own_in = left, tot = left + nsv;
      left = 0;
      auto entry = [&](int k) {
        return k < own_in ? __ldcs(row + (int64_t)k * (T * 32)) : sslot[k - own_in][threadIdx.x];
      };
      int jn = tot > 0 ? entry(0) : 0;
      for (int k = 0; k < tot; k++) {
        const int j = jn;
        const XFix o = md_ld_xfix(a.xq + j);
        if (k + 1 < tot) jn = entry(k + 1);
        pair(j, o);
      }
    } while (q < nsk);

    if (T > 1) {
#pragma unroll
      for (int off = T / 2; off > 0; off >>= 1) {
        ax += __shfl_xor_sync(0xffffffffu, ax, off);
        ay += __shfl_xor_sync(0xffffffffu, ay, off);
        az += __shfl_xor_sync(0xffffffffu, az, off);
      }
    }
    if (active && t == 0) {
      if (HALF) {
        atomicAdd(a.fix + i, (unsigned long long)(-ax));
        atomicAdd(a.fix + n + i, (unsigned long long)(-ay));
        atomicAdd(a.fix + 2 * n + i, (unsigned long long)(-az));
      } else {  // full list: the owner's sum is the whole count
        a.fix[i] = (unsigned long long)(-ax);
        a.fix[n + i] = (unsigned long long)(-ay);
        a.fix[2 * n + i] = (unsigned long long)(-az);
      }
    }
    if (EV) {
      const double evw = HALF ? 1.0 : 0.5;  // a full list visits each pair twice
      // one type: -(lj4 / 2) sum r^-6, the rest of the energy is trace(W) / 12
      // (r^-6 = x^3 2^(3 B - 6 R))
      const double e = SINGLE ? -0.5 * a.c1.lj4 *
                                    __fma_rn(__ull2double_rn(s6),
                                             __longlong_as_double(
                                                 (long long)(1023 - 62 + a.ev_shift +
                                                             3 * a.fx1.B - 6 * a.fxR)
                                                 << 52),
                                             e0)
                              : e0;
      md_warp_add_ev(e, npair, img, &simg[0][threadIdx.x], evw,
                     active ? MD_TAG_REP(tag) : -1, a.ev, a.ev_spread,
                     (int)(gid >> 5) % a.ev_spread);
    }
  }
}

// Resident blocks per SM the register allocation must allow (9: 56 registers).
// 4,000,000 atoms, force-only half list: 8, 9 and 10 blocks measured 1.60,
// 1.53 and 1.57 ms; energy/virial half list with 6, 7, 8, 9 and 10 blocks 2.49,
// 2.35, 2.27, 2.42 and 2.76 ms, full list 8, 9 and 10 blocks 3.21, 3.14 and 3.53
// (whole energy passes, with the passes over atoms of that time).
#define MD_FX_MINB 9
constexpr int md_pair_fx_minb(bool half, bool ev) { return ev && half ? 8 : MD_FX_MINB; }

template <bool HALF, bool EV, bool SINGLE, bool COUL, int T, int U>
__global__ void __launch_bounds__(MD_BLOCK, md_pair_fx_minb(HALF, EV))
    k_pair_fx(const __grid_constant__ PairArgs a, const float cut_hi1,
              const float* __restrict__ cut_hi_tab) {
  if (md_stopped(a.stop)) return;
  md_pair_fx_tiles<HALF, EV, SINGLE, COUL, T, U>(a, cut_hi1, cut_hi_tab);
}

template <bool HALF, bool EV, bool SINGLE, bool COUL, int T, int U>
cudaError_t md_pair_fx_launch1(const PairArgs& a, float cut1, const float* cut_tab,
                               cudaStream_t s, int carve) {
  int occ = 1;
  const size_t smem = md_pair_fx_smem(SINGLE, a.nt);
  cudaError_t e =
      md_prepare_kernel((const void*)k_pair_fx<HALF, EV, SINGLE, COUL, T, U>, carve, smem, &occ);
  if (e != cudaSuccess) return e;
  unsigned blocks = (unsigned)md_blocks(a.n * T);
  if (a.tile_ctr) {
    const unsigned cap = (unsigned)(a.nslots * occ);
    if (blocks > cap) blocks = cap;
  }
  k_pair_fx<HALF, EV, SINGLE, COUL, T, U><<<blocks, MD_BLOCK, smem, s>>>(a, cut1, cut_tab);
  return cudaGetLastError();
}

template <bool HALF, bool EV, bool SINGLE, bool COUL, int U>
cudaError_t md_pair_fx_launch_u(const PairArgs& a, int t, float cut1, const float* cut_tab,
                                cudaStream_t s, int carve) {
  switch (t) {
    case 2: return md_pair_fx_launch1<HALF, EV, SINGLE, COUL, 2, U>(a, cut1, cut_tab, s, carve);
    case 4: return md_pair_fx_launch1<HALF, EV, SINGLE, COUL, 4, U>(a, cut1, cut_tab, s, carve);
    case 8: return md_pair_fx_launch1<HALF, EV, SINGLE, COUL, 8, U>(a, cut1, cut_tab, s, carve);
    default: return cudaErrorInvalidValue;
  }
}

template <bool HALF, bool SINGLE>
cudaError_t md_pair_fx_launch_t(const PairArgs& a, bool ev, int t, int u, float cut1,
                                const float* cut_tab, cudaStream_t s, int carve) {
  if (ev) return md_pair_fx_launch_u<HALF, true, SINGLE, false, 2>(a, t, cut1, cut_tab, s, carve);
  return u == 1 ? md_pair_fx_launch_u<HALF, false, SINGLE, false, 1>(a, t, cut1, cut_tab, s, carve)
                : md_pair_fx_launch_u<HALF, false, SINGLE, false, 2>(a, t, cut1, cut_tab, s, carve);
}

// t: lanes per atom (2, 4 or 8); u: skin entries per round of a force-only
// launch (1 or 2; 2 with energy and virial)
cudaError_t md_pair_fx_launch(const PairArgs& a, bool half, bool ev, bool single, int t, int u,
                              float cut1, const float* cut_tab, cudaStream_t s, int carve);
// lj/cut/coul/cut (md_pair_coul.cu): two skin entries per round
cudaError_t md_pair_fx_coul_launch(const PairArgs& a, bool half, bool ev, int t, float cut1,
                                   const float* cut_tab, cudaStream_t s, int carve);
