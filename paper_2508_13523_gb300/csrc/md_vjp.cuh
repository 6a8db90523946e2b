// md_vjp.cuh -- the adjoint of the pair force kernel: vector-Jacobian
// products of the forces with respect to positions and to the per-type-pair
// (eps, sigma), over the same tiled neighbor list (arXiv 2508.13523, Eq. 1
// and its pairwise derivative, Sec. 4).
//
// For a pair (i, j) inside rc with d = x_j - x_i, q = |d|^2, the force on i
// is -g(q) d and on j +g(q) d, with
//   g(q)  = 24 eps (2 sigma^12 q^-7 - sigma^6 q^-4) = r^-2 r^-6 (lj1 r^-6 - lj2),
//   g'(q) = 24 eps (-14 sigma^12 q^-8 + 4 sigma^6 q^-5)
//         = r^-4 r^-6 (-7 lj1 r^-6 + 4 lj2).
// Given the cotangent c = dL/dF and w = c_i - c_j, e = -d:
//   xbar_i += J w, xbar_j -= J w,   J w = g w + 2 g' e (e . w),
//   dL/deps   += (e . w) g / eps,
//   dL/dsigma += (e . w) r^-2 r^-6 (12 lj1 r^-6 - 6 lj2) / sigma.
// Cutoffs are held fixed.  A full list visits each pair from both ends: each
// visit adds J w to its own atom only and half of the parameter terms.
//
// FP64: bound by the FP64 pipe (about 44 operations a pair at 64 cycles each:
// 150 us of the 272 us at 62,500 mixture atoms).  Mixed: no FP64 operation per
// pair; the cotangent is read as FP32 (16 bytes), the parameter terms are FP32
// values with their rounding errors in the thread's own shared-memory column
// (one row per thread put all lanes on the same banks), and the sums' atomics
// are spread over rows.  62,500 atoms, half list, before and after: mixed 140 ->
// 59 us, FP64 350 -> 272 us.
#pragma once

#include <type_traits>

#include "md_device.cuh"
#include "md_internal.cuh"

struct VjpCoef {
  double inv_eps, inv_sigma;
  float inv_epsf, inv_sigmaf;
};

#define MD_GBAR_ROWS 128

struct VjpArgs {
  const double4_32a* x4;
  const XSplit* xs;
  const XSplit* xb;      // positions at the last build (split)
  float rin;             // rlist rounded up: atoms this far inside every face need no image
  const double4_32a* c;  // cotangent per sorted atom (x, y, z, unused)
  const float4* cf;      // the same rounded to FP32 (mixed precision)
  const int32_t* numneigh;
  const int32_t* nbr;
  double* xbar;          // SoA per sorted atom, accumulated (+=)
  double* gbar;          // rows of 2 nt^2: dL/deps then dL/dsigma, entry [min][max]; the
                         // blocks' sums are spread over the rows so that their atomics
                         // do not queue on the same addresses
  int rows;              // 1 or MD_GBAR_ROWS
  const PairCoef* coef;
  const VjpCoef* vcoef;
  PairCoef c1;
  VjpCoef v1;
  const RepGeo* rep;
  float cut1;            // certified FP32 bounds of rc^2 (Geo::cut_hi): the only one,
  const float* cut_tab;  // the nt*nt table
  int64_t n;
  int nt;
  int maxneigh;
};

#define MD_VJP_SLOTS 8  // skin entries that wait per lane

template <int PREC, bool HALF, int TPA, bool SINGLE>
__global__ void __launch_bounds__(MD_BLOCK) k_vjp(const VjpArgs a) {
  constexpr bool MIX = PREC == MD_PREC_MIXED;
  // md_vjp_smem.  sg: parameter terms of each thread by partner type: [tj]
  // eps, [nt + tj] sigma; thread-private columns (no bank conflicts), reduced
  // at the end (mixed: FP32 values with their rounding errors, md_acc2).
  // Types are clamped to those there are, as the columns end with them.
  extern __shared__ double s_tab[];
  double* sg = s_tab;
  PairCoef* sc = reinterpret_cast<PairCoef*>(sg + 2 * a.nt * MD_BLOCK);
  VjpCoef* sv = reinterpret_cast<VjpCoef*>(sc + a.nt * a.nt);
  float* scut = reinterpret_cast<float*>(sv + a.nt * a.nt);
  if (!SINGLE) {
    for (int k = threadIdx.x; k < a.nt * a.nt; k += blockDim.x) {
      sc[k] = a.coef[k];
      sv[k] = a.vcoef[k];
      scut[k] = a.cut_tab[k];
    }
    for (int k = 0; k < 2 * a.nt; k++) sg[k * MD_BLOCK + threadIdx.x] = 0.0;
    __syncthreads();
  }
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t i = gid / TPA;
  const int t = (int)(gid % TPA);
  const bool active = i < a.n;
  const int64_t ia = active ? i : 0;
  const int64_t n = a.n;
  const int nin = active ? __ldg(a.numneigh + ia) : 0;
  const int nsk = active ? __ldg(a.numneigh + n + ia) : 0;
  const int32_t* row = a.nbr + (ia >> 5) * (int64_t)a.maxneigh * 32 + (ia & 31);
  const int32_t* skin = row + (int64_t)(a.maxneigh - 1) * 32;
  const double4_32a ci = MIX ? double4_32a{} : a.c[ia];
  const double half = HALF ? 1.0 : 0.5;

  // The lane's entries in rounds (almost always one): an FP32 test of the hi
  // parts picks the skin entries that may be inside rc (few), then the inner
  // entries and the picked ones go through `take`, so that the derivative's
  // code runs for lanes that almost all have a pair in range.  A lane waits for
  // its gathers most of the time: two skin entries a round, the cotangent
  // loaded with the position and the next entry's index before the pair
  // (64,000 atoms of two types, mixed half list: 64 -> 59 us).
  __shared__ int sslot[MD_VJP_SLOTS][MD_BLOCK];
  auto walk = [&](const RepGeo* g, int type, auto take) {
    const float4 hi = md_ld_hi<MIX ? 1 : 0>(a.xs, ia);
    const float hf0 = g->halfLf[0], hf1 = g->halfLf[1], hf2 = g->halfLf[2];
    int left = nin, q = t;
    do {
      int nsv = 0;
      auto test = [&](const float4& hj, int j) {
        float dx = hj.x - hi.x, dy = hj.y - hi.y, dz = hj.z - hi.z;
        dx = fabsf(dx) > hf0 ? dx - copysignf(g->Lf[0], dx) : dx;
        dy = fabsf(dy) > hf1 ? dy - copysignf(g->Lf[1], dy) : dy;
        dz = fabsf(dz) > hf2 ? dz - copysignf(g->Lf[2], dz) : dz;
        const float r2f = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, dx * dx));
        const float cut = SINGLE ? a.cut1
                                 : scut[type * a.nt + MD_TAG_TYPE(__float_as_int(hj.w))];
        if (r2f <= cut) sslot[nsv++][threadIdx.x] = j;
      };
      // two entries a round, their gathers in flight together
      for (; q + TPA < nsk && nsv < MD_VJP_SLOTS - 1; q += 2 * TPA) {
        const int j0 = __ldcs(skin - (int64_t)q * 32);
        const int j1 = __ldcs(skin - (int64_t)(q + TPA) * 32);
        const float4 h0 = md_ld_hi<MIX ? 1 : 0>(a.xs, j0), h1 = md_ld_hi<MIX ? 1 : 0>(a.xs, j1);
        test(h0, j0);
        test(h1, j1);
      }
      if (q + TPA >= nsk && q < nsk && nsv < MD_VJP_SLOTS) {
        const int j = __ldcs(skin - (int64_t)q * 32);
        test(md_ld_hi<MIX ? 1 : 0>(a.xs, j), j);
        q += TPA;
      }
      const int own = left > t ? (left - t + TPA - 1) / TPA : 0;
      left = 0;
      auto entry = [&](int k) {
        return k < own ? __ldcs(row + (int64_t)(t + k * TPA) * 32) : sslot[k - own][threadIdx.x];
      };
      int j = own + nsv > 0 ? entry(0) : 0;
      for (int k = 0; k < own + nsv; k++) {
        const int jn = k + 1 < own + nsv ? entry(k + 1) : 0;
        take(j);
        j = jn;
      }
    } while (q < nsk);
  };

  double bx = 0.0, by = 0.0, bz = 0.0;  // xbar_i
  double ge0 = 0.0, gs0 = 0.0;          // parameter terms when SINGLE
  double* slot = SINGLE ? nullptr : sg + threadIdx.x;
  float2* slot2 = reinterpret_cast<float2*>(slot);
  float geh = 0.f, gel = 0.f, gsh = 0.f, gsl = 0.f;  // mixed: parameter terms when SINGLE
  int ti;

  if (PREC == MD_PREC_FP64) {
    const double4_32a xi = md_ld4(a.x4 + ia);
    const int tag_i = md_tag_of(xi);
    ti = min((int)MD_TAG_TYPE(tag_i), a.nt - 1);
    const RepGeo* g = a.rep + MD_TAG_REP(tag_i);
    // An atom that was at least rlist from every face at the last build has
    // no pair across the boundary until the next build (both ends of a
    // listed pair move continuously, unwrapped): its rows need no minimum
    // image.  The test is warp-uniform so that the other warps keep the
    // image code (which the compiler makes unconditional) off their pairs.
    const float4 bh = md_ld_hi<0>(a.xb, ia);
    const float r0 = a.rin + g->Lf[0] * 0x1p-20f, r1 = a.rin + g->Lf[1] * 0x1p-20f,
                r2b = a.rin + g->Lf[2] * 0x1p-20f;
    const bool inner_atom = bh.x >= r0 && bh.x <= g->Lf[0] - r0 && bh.y >= r1 &&
                            bh.y <= g->Lf[1] - r1 && bh.z >= r2b && bh.z <= g->Lf[2] - r2b;
    const bool no_image = __all_sync(0xffffffffu, inner_atom || !active);
    auto pairs = [&](auto wrap) {
      constexpr bool WRAP = decltype(wrap)::value;
      const double L0 = g->L[0], L1 = g->L[1], L2 = g->L[2];
      const long long h0 = g->halfL_bits[0], h1 = g->halfL_bits[1], h2 = g->halfL_bits[2];
      walk(g, ti, [&](int j) {
        const double4_32a xj = md_ld4(a.x4 + j);
        const double4_32a cj = md_ld4(a.c + j);  // with the position: nearly every pair needs it
        double dx = __dsub_rn(xj.x, xi.x);
        double dy = __dsub_rn(xj.y, xi.y);
        double dz = __dsub_rn(xj.z, xi.z);
        if (WRAP) {
          dx = md_min_image(dx, L0, h0);
          dy = md_min_image(dy, L1, h1);
          dz = md_min_image(dz, L2, h2);
        }
        const double r2 = md_r2(dx, dy, dz);
        const int tj = SINGLE ? 0 : min(md_type_of(xj), a.nt - 1);
        const PairCoef& cf = SINGLE ? a.c1 : sc[ti * a.nt + tj];
        if (md_lt_pos(r2, cf.cutsq_bits)) {
          // with t = r^-2 r^-6, A = lj1 r^-6 t, B = lj2 t:
          //   g = A - B,  g' = r^-2 (-7 A + 4 B),  r^-2 r^-6 (12 lj1 r^-6 - 6 lj2) = 12 A - 6 B
          const double r2inv = md_rcp(r2);
          const double r6inv = r2inv * r2inv * r2inv;
          const double tt = r2inv * r6inv;
          const double A = (cf.lj1 * r6inv) * tt;
          const double B = cf.lj2 * tt;
          const double gq = A - B;
          const double wx = ci.x - cj.x, wy = ci.y - cj.y, wz = ci.z - cj.z;
          const double dw = __fma_rn(dz, wz, __fma_rn(dy, wy, dx * wx));  // d . w = -(e . w)
          // J w = g w + 2 g' e (e . w) = g w + 2 g' (d . w) d
          const double sc2 = (2.0 * r2inv) * (dw * __fma_rn(-7.0, A, 4.0 * B));
          const double jx = __fma_rn(sc2, dx, gq * wx);
          const double jy = __fma_rn(sc2, dy, gq * wy);
          const double jz = __fma_rn(sc2, dz, gq * wz);
          bx += jx;
          by += jy;
          bz += jz;
          if (HALF) {
            atomicAdd(a.xbar + j, -jx);
            atomicAdd(a.xbar + n + j, -jy);
            atomicAdd(a.xbar + 2 * n + j, -jz);
          }
          // parameter terms without their 1/eps, 1/sigma factors (applied
          // once per table entry at the end); e . w = -(d . w)
          const double hw = HALF ? -dw : -0.5 * dw;
          const double de = hw * gq;
          const double ds = hw * __fma_rn(12.0, A, -6.0 * B);
          if (SINGLE) {
            ge0 += de;
            gs0 += ds;
          } else {
            slot[tj * MD_BLOCK] += de;
            slot[(a.nt + tj) * MD_BLOCK] += ds;
          }
        }
      });
    };
    if (no_image)
      pairs(std::integral_constant<bool, false>{});
    else
      pairs(std::integral_constant<bool, true>{});
  } else {
    const XSplit si = md_ld_split(a.xs + ia);
    const int tag_i = __float_as_int(si.hi.w);
    ti = min((int)MD_TAG_TYPE(tag_i), a.nt - 1);
    const RepGeo* g = a.rep + MD_TAG_REP(tag_i);
    const float Lf0 = g->Lf[0], Lf1 = g->Lf[1], Lf2 = g->Lf[2];
    const float Ll0 = g->Llo[0], Ll1 = g->Llo[1], Ll2 = g->Llo[2];
    const float hf0 = g->halfLf[0], hf1 = g->halfLf[1], hf2 = g->halfLf[2];
    const float4 cif = a.cf[ia];
    const float cix = cif.x, ciy = cif.y, ciz = cif.z;
    float axh = 0.f, axl = 0.f, ayh = 0.f, ayl = 0.f, azh = 0.f, azl = 0.f;
    walk(g, ti, [&](int j) {
      const XSplit sj = md_ld_split(a.xs + j);
      const float4 cj = __ldg(a.cf + j);  // with the position: nearly every pair needs it
      float hx = sj.hi.x - si.hi.x, lx = sj.lo.x - si.lo.x;
      float hy = sj.hi.y - si.hi.y, ly = sj.lo.y - si.lo.y;
      float hz = sj.hi.z - si.hi.z, lz = sj.lo.z - si.lo.z;
      if (fabsf(hx) > hf0) {
        const float sg = copysignf(1.f, hx);
        hx -= sg * Lf0;
        lx -= sg * Ll0;
      }
      if (fabsf(hy) > hf1) {
        const float sg = copysignf(1.f, hy);
        hy -= sg * Lf1;
        ly -= sg * Ll1;
      }
      if (fabsf(hz) > hf2) {
        const float sg = copysignf(1.f, hz);
        hz -= sg * Lf2;
        lz -= sg * Ll2;
      }
      const float dx = hx + lx, dy = hy + ly, dz = hz + lz;
      const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, dx * dx));
      const int tj = SINGLE ? 0 : min((int)MD_TAG_TYPE(__float_as_int(sj.hi.w)), a.nt - 1);
      const PairCoef& cf = SINGLE ? a.c1 : sc[ti * a.nt + tj];
      // the forward kernel's cutoff decision: FP64 r^2 inside the band
      bool in = r2 < cf.cutsqf;
      if ((r2 > cf.cut_lof) & (r2 < cf.cut_hif))
        in = md_lt_pos(md_r2_split(a.xs + j, si, hf0, hf1, hf2, Lf0, Lf1, Lf2, Ll0, Ll1, Ll2),
                       cf.cutsq_bits);
      if (in) {
        const float r2inv = __frcp_rn(r2);
        const float r6inv = r2inv * r2inv * r2inv;
        const float gq = r6inv * (cf.lj1f * r6inv - cf.lj2f) * r2inv;
        const float gp = r2inv * r2inv * r6inv * (-7.0f * cf.lj1f * r6inv + 4.0f * cf.lj2f);
        const float wx = cix - cj.x, wy = ciy - cj.y, wz = ciz - cj.z;
        const float ew = -(dx * wx + dy * wy + dz * wz);
        const float s = -2.0f * gp * ew;
        const float jx = __fmaf_rn(s, dx, gq * wx);
        const float jy = __fmaf_rn(s, dy, gq * wy);
        const float jz = __fmaf_rn(s, dz, gq * wz);
        md_acc2(axh, axl, jx);
        md_acc2(ayh, ayl, jy);
        md_acc2(azh, azl, jz);
        if (HALF) {
          atomicAdd(a.xbar + j, -md_widen(jx));
          atomicAdd(a.xbar + n + j, -md_widen(jy));
          atomicAdd(a.xbar + 2 * n + j, -md_widen(jz));
        }
        const float hw = (float)half * ew;
        // parameter terms: no FP64 operation per pair (an FP64 add costs 64
        // cycles of its pipe); value and rounding error in FP32
        const float de = hw * gq;
        const float ds = hw * r2inv * r6inv * (12.0f * cf.lj1f * r6inv - 6.0f * cf.lj2f);
        if (SINGLE) {
          md_acc2(geh, gel, de);
          md_acc2(gsh, gsl, ds);
        } else {
          float2 e2 = slot2[tj * MD_BLOCK], s2 = slot2[(a.nt + tj) * MD_BLOCK];
          md_acc2(e2.x, e2.y, de);
          md_acc2(s2.x, s2.y, ds);
          slot2[tj * MD_BLOCK] = e2;
          slot2[(a.nt + tj) * MD_BLOCK] = s2;
        }
      }
    });
    if (SINGLE) {
      ge0 = md_widen(geh) + md_widen(gel);
      gs0 = md_widen(gsh) + md_widen(gsl);
    }
    bx = md_widen(axh) + md_widen(axl);
    by = md_widen(ayh) + md_widen(ayl);
    bz = md_widen(azh) + md_widen(azl);
  }

  if (TPA > 1) {
#pragma unroll
    for (int off = TPA / 2; off > 0; off >>= 1) {
      bx += __shfl_xor_sync(0xffffffffu, bx, off);
      by += __shfl_xor_sync(0xffffffffu, by, off);
      bz += __shfl_xor_sync(0xffffffffu, bz, off);
    }
  }
  if (active && t == 0) {
    if (HALF) {
      atomicAdd(a.xbar + i, bx);
      atomicAdd(a.xbar + n + i, by);
      atomicAdd(a.xbar + 2 * n + i, bz);
    } else {  // only this thread touches atom i's entries
      a.xbar[i] += bx;
      a.xbar[n + i] += by;
      a.xbar[2 * n + i] += bz;
    }
  }
  // parameter terms: entry [min(ti,tj)][max(ti,tj)] of each table
  const int nt2 = a.nt * a.nt;
  double* grow = a.gbar + (int64_t)(blockIdx.x % (unsigned)a.rows) * 2 * nt2;
  if (SINGLE) {
    double v[2] = {ge0, gs0};
#pragma unroll
    for (int k = 0; k < 2; k++) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(grow, v[0] * a.v1.inv_eps);
      atomicAdd(grow + nt2, v[1] * a.v1.inv_sigma);
    }
  } else {
    // each warp sums each table entry over its lanes (a lane has terms of
    // entry (ea, eb) if its atom's type is one of the two): one atomic per
    // entry and warp
    const int tt = active ? ti : -1;
    for (int w = 0; w < 2; w++)
      for (int ea = 0; ea < a.nt; ea++)
        for (int eb = ea; eb < a.nt; eb++) {
          const int o = tt == ea ? eb : (tt == eb ? ea : -1);
          double v = 0.0;
          if (MIX) {  // FP32 pairs
            float2 p = o >= 0 ? slot2[(w * a.nt + o) * MD_BLOCK] : make_float2(0.f, 0.f);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
              const float h = __shfl_xor_sync(0xffffffffu, p.x, off);
              p.y = __fadd_rn(p.y, __shfl_xor_sync(0xffffffffu, p.y, off));
              md_acc2(p.x, p.y, h);
            }
            v = md_widen(p.x) + md_widen(p.y);
          } else {
            if (o >= 0) v = slot[(w * a.nt + o) * MD_BLOCK];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
          }
          if ((threadIdx.x & 31) == 0 && v != 0.0) {
            const VjpCoef& vc = sv[ea * a.nt + eb];
            atomicAdd(grow + w * nt2 + ea * a.nt + eb, v * (w ? vc.inv_sigma : vc.inv_eps));
          }
        }
  }
}

// Dynamic shared memory: parameter terms and tables of the types that there are
// (with room for MD_MAX_TYPES in every block, L1 was down to 28 KB: 64,000
// atoms of two types, mixed half list 70 -> 64 us).
inline size_t md_vjp_smem(bool single, int nt) {
  return single ? 0
                : sizeof(double) * 2 * nt * MD_BLOCK +
                      (sizeof(PairCoef) + sizeof(VjpCoef)) * (size_t)(nt * nt) +
                      sizeof(float) * (size_t)(nt * nt + MD_MAX_TYPES);
}

template <int PREC, bool HALF, bool SINGLE>
cudaError_t md_vjp_launch_tpa(const VjpArgs& a, int tpa, unsigned blocks, cudaStream_t s) {
  const size_t smem = md_vjp_smem(SINGLE, a.nt);
  switch (tpa) {
    case 2: k_vjp<PREC, HALF, 2, SINGLE><<<blocks, MD_BLOCK, smem, s>>>(a); break;
    case 4:  // FP64 alone (vjp_lanes)
      if constexpr (PREC == MD_PREC_FP64)
        k_vjp<PREC, HALF, 4, SINGLE><<<blocks, MD_BLOCK, smem, s>>>(a);
      else
        return cudaErrorInvalidValue;
      break;
    case 8: k_vjp<PREC, HALF, 8, SINGLE><<<blocks, MD_BLOCK, smem, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int PREC>
cudaError_t md_vjp_launch_prec(const VjpArgs& a, bool half, bool single, int tpa,
                               unsigned blocks, cudaStream_t s) {
  if (half)
    return single ? md_vjp_launch_tpa<PREC, true, true>(a, tpa, blocks, s)
                  : md_vjp_launch_tpa<PREC, true, false>(a, tpa, blocks, s);
  return single ? md_vjp_launch_tpa<PREC, false, true>(a, tpa, blocks, s)
                : md_vjp_launch_tpa<PREC, false, false>(a, tpa, blocks, s);
}

cudaError_t md_vjp_launch_fp64(const VjpArgs& a, bool half, bool single, int tpa,
                               unsigned blocks, cudaStream_t s);
cudaError_t md_vjp_launch_mixed(const VjpArgs& a, bool half, bool single, int tpa,
                                unsigned blocks, cudaStream_t s);
