// md_pair_q.cuh -- FP64 pair kernel with warp-level compaction of in-range
// pairs (arXiv 2508.13523, Eq. 1 and Sec. 4; Sec. 4.1 names the two sources
// of GPU divergence this removes: rows of different length and the cutoff
// branch).
//
// On GB300 the FP64 pipe is the bottleneck of the FP64 form, and in a
// one-thread-per-atom loop a warp issues every FP64 instruction for all 32
// lanes even when only some lanes have a pair inside rc (rows end at
// different lengths; skin pairs are mostly outside rc).  Here each warp
//   phase 1: takes one list entry per lane and tests it in FP32 against a
//            certified upper bound of rc^2 (positions' FP32 split and the FP32
//            arithmetic bounded as in the list build); entries that are
//            certainly outside rc are dropped, the rest are appended to one
//            of two per-warp queues in shared memory (ballot + popc): queue
//            1 if the FP32 separation along some axis is close to or above
//            half the box (a periodic image may be nearer), queue 0 if
//            certainly not;
//   phase 2: whenever 32 entries are queued, all 32 lanes take one each and
//            do the exact FP64 work: separation, minimum image (queue 1
//            only), r^2, the exact cutoff test, the force, and global
//            reductions into the owner's force and (half list) f_j, which
//            start from zero.
// The two queues keep the minimum image, which the compiler turns into
// three unconditional FP64 subtractions, off the ~98 % of pairs (in a large
// box) that never cross the boundary.
// The FP64 decisions and arithmetic per pair are those of k_pair; only the
// summation of the contributions into f_i differs: FP64 reductions into f
// (order-dependent rounding).  The fixed-point sums are md_pair_fx.cuh's.
// COUL adds the second pair style's cut Coulomb term qq / r (1/r from the
// rsqrt seed and one series round; r^-2 = (1/r)^2 instead of md_rcp).
#pragma once

#include <type_traits>

#include "md_device.cuh"
#include "md_internal.cuh"
#include "md_pair.cuh"

#define MD_Q_CAP 64  // queue entries per warp (a ring; at most 63 in use)
// Resident blocks per SM the register allocation must allow (force-only
// launches): 10 x 128 threads caps the kernel at 48 registers, which it
// fits without spills.
#define MD_Q_MINB 10

// The tile loop of the compacted kernel; all threads of the block must call it.
template <bool HALF, bool EV, bool SINGLE, bool COUL>
__device__ __forceinline__ void md_pair_q_tiles(const PairArgs& a, const float cut_hi1,
                                                const float* __restrict__ cut_hi_tab) {
  constexpr int W = MD_BLOCK / 32;
  __shared__ PairCoef sc[SINGLE ? 1 : MD_MAX_TYPES * MD_MAX_TYPES];
  __shared__ float scut[SINGLE ? 1 : MD_MAX_TYPES * MD_MAX_TYPES];
  __shared__ int qj[2][W][MD_Q_CAP];            // queue 0: no image, 1: may wrap
  __shared__ unsigned char qo[2][W][MD_Q_CAP];
  __shared__ double4_32a xown[W][32];      // owner positions (x, y, z, tag)
  __shared__ double sev[EV ? W : 1][8][32];  // owner energy/virial accumulators
  if (!SINGLE) {
    for (int k = threadIdx.x; k < a.nt * a.nt; k += blockDim.x) {
      sc[k] = a.coef[k];
      scut[k] = cut_hi_tab[k];
    }
  }
  if (!SINGLE) __syncthreads();
  __shared__ int s_tile;
  const int ntiles = (int)((a.n + MD_BLOCK - 1) / MD_BLOCK);
  for (int it = 0;; it++) {
    if (threadIdx.x == 0)
      s_tile = a.tile_ctr ? md_next_tile(a.tile_ctr, a.nslots, ntiles)
                          : (it == 0 ? (int)blockIdx.x : -1);
    __syncthreads();
    const int64_t tile = s_tile;
    __syncthreads();
    if (tile < 0) break;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = tile * MD_BLOCK + threadIdx.x;
    const bool active = i < a.n;
    const int64_t ia = active ? i : 0;
    const int64_t n = a.n;
    const int nin = active ? __ldg(a.numneigh + ia) : 0;
    const int nsk = active ? __ldg(a.numneigh + n + ia) : 0;
    const int cnt = nin + nsk;
    const int32_t* row = a.nbr + (ia >> 5) * (int64_t)a.maxneigh * 32 + (ia & 31);
    const int32_t* skin = row + (int64_t)(a.maxneigh - 1) * 32;
    const double4_32a xi = md_ld4(a.x4 + ia);
    const int tag_i = md_tag_of(xi);
    const int ti = MD_TAG_TYPE(tag_i);
    const RepGeo* g = a.rep + MD_TAG_REP(tag_i);
    // FP32 view of the own position (phase 1)
    const float4 hi = md_ld_hi<0>(a.xs, ia);
    const float Lf0 = g->Lf[0], Lf1 = g->Lf[1], Lf2 = g->Lf[2];
    const float hf0 = g->halfLf[0], hf1 = g->halfLf[1], hf2 = g->halfLf[2];
    // routing bound (1 - 2^-12) L/2: the FP32 separation of the hi parts is
    // within 3 * 2^-24 L of the FP64 one, so |d32| <= this bound on every
    // axis means |d| < L/2 in FP64 (no periodic image is nearer)
    const float hm0 = hf0 * (1.f - 0x1p-12f), hm1 = hf1 * (1.f - 0x1p-12f),
                hm2 = hf2 * (1.f - 0x1p-12f);
    xown[w][lane] = xi;
    if (EV) {
  #pragma unroll
      for (int k = 0; k < 8; k++) sev[w][k][lane] = 0.0;
    }
    __syncthreads();

    // Energy and virial: when every active atom of the warp lies in one box
    // (always for a single box), each lane sums the pairs it drains in
    // registers -- E, a pair count, and for the rare pairs taken through a
    // periodic image (queue 1 only) the virial's image terms -s_a g_b (s the
    // shift taken off d, g = fpair d) -- and the warp reduces them once;
    // otherwise they go to per-owner shared accumulators and then to the
    // owners' boxes.  The rest of the virial, sum_a x_a (x) F_a, is summed
    // per atom after the forces are complete.  The shuffle and vote run on
    // every lane.
    const int rep_i = MD_TAG_REP(tag_i);
    bool uni = false;
    int rep0 = -1;
    if (EV) {
      const int r0 = __shfl_sync(0xffffffffu, rep_i, 0);
      uni = __all_sync(0xffffffffu, !active || rep_i == r0);
      rep0 = __any_sync(0xffffffffu, active) ? r0 : -1;
    }
    double e0 = 0.0;  // this lane's energy sum (uniform warps; the virial's image
                      // terms, rare, go to the lane's own column of sev)
    int npair = 0;
    // one type, Eq. 1 alone: with lj1 = 12 lj3 and lj2 = 6 lj4 a pair's
    // energy is fpair r^2 / 12 - (lj4 / 2) r^-6, and the sum of fpair r^2 is
    // the trace of the virial, which the sum over atoms gives; so the loop
    // sums r^-6 alone (one FP64 add a pair) and the trace's share is added
    // where the energy is read (md_capi.cu, fill_thermo).  All pairs of the
    // box take this form, the shared-accumulator path too.
    constexpr bool S2 = SINGLE && !COUL;
    double s6 = 0.0;
    const double evw = HALF ? 1.0 : 0.5;
    int q = 0;            // this lane's next list entry
    unsigned head[2] = {0, 0}, tail[2] = {0, 0};  // warp-uniform ring counters

    // phase 2: one queued pair per lane, exact FP64
    auto drain = [&](auto queue, unsigned take) {
      constexpr int Q = decltype(queue)::value;
      const unsigned e = head[Q] + lane;
      if (lane < take) {
        const int j = qj[Q][w][e % MD_Q_CAP];
        const int o = qo[Q][w][e % MD_Q_CAP];
        const double4_32a xo = xown[w][o];
        const double4_32a xj = md_ld4(a.x4 + j);
        double dx = __dsub_rn(xj.x, xo.x);
        double dy = __dsub_rn(xj.y, xo.y);
        double dz = __dsub_rn(xj.z, xo.z);
        double shx = 0.0, shy = 0.0, shz = 0.0;  // EV: the image shift s L taken off d
        if (Q == 1) {
          const RepGeo* go = a.rep + MD_TAG_REP(md_tag_of(xo));
          const long long h0 = go->halfL_bits[0], h1 = go->halfL_bits[1],
                          h2 = go->halfL_bits[2];
          if (EV) {
            shx = md_abs_gt(dx, h0) ? copysign(go->L[0], dx) : 0.0;
            shy = md_abs_gt(dy, h1) ? copysign(go->L[1], dy) : 0.0;
            shz = md_abs_gt(dz, h2) ? copysign(go->L[2], dz) : 0.0;
          }
          dx = md_min_image(dx, go->L[0], h0);
          dy = md_min_image(dy, go->L[1], h1);
          dz = md_min_image(dz, go->L[2], h2);
        }
        const double r2 = md_r2(dx, dy, dz);
        const int to = MD_TAG_TYPE(md_tag_of(xo));
        const PairCoef& c = SINGLE ? a.c1 : sc[to * a.nt + md_type_of(xj)];
        if (md_lt_pos(r2, COUL ? c.cutmax_bits : c.cutsq_bits)) {
          double r2inv, r6inv, fpair, qr = 0.0;
          if (COUL) {  // Eq. 1 below rc, plus qq / r below rc_coul (selects, no branch)
            const double rinv = md_rsqrt(r2);
            r2inv = rinv * rinv;
            r6inv = r2inv * r2inv * r2inv;
            const double flj = r6inv * (c.lj1 * r6inv - c.lj2) * r2inv;
            qr = c.qq * rinv;
            qr = md_lt_pos(r2, c.cutsq_coul_bits) ? qr : 0.0;
            fpair = __fma_rn(qr, r2inv, md_lt_pos(r2, c.cutsq_bits) ? flj : 0.0);
          } else {
            r2inv = md_rcp(r2);
            r6inv = r2inv * r2inv * r2inv;
            fpair = r6inv * (c.lj1 * r6inv - c.lj2) * r2inv;
          }
          const double gx = fpair * dx, gy = fpair * dy, gz = fpair * dz;
          const int64_t io = tile * MD_BLOCK + w * 32 + o;
          atomicAdd(a.f + io, md_neg(gx));
          atomicAdd(a.f + n + io, md_neg(gy));
          atomicAdd(a.f + 2 * n + io, md_neg(gz));
          if (HALF) {
            atomicAdd(a.f + j, gx);
            atomicAdd(a.f + n + j, gy);
            atomicAdd(a.f + 2 * n + j, gz);
          }
          if (EV) {  // the virial is x (x) F per atom afterwards, less the image terms
            const bool img = (shx != 0.0) | (shy != 0.0) | (shz != 0.0);
            auto energy = [&]() {
              if (S2) return -0.5 * c.lj4 * r6inv;
              double en = r6inv * (c.lj3 * r6inv - c.lj4);
              if (COUL) en = (md_lt_pos(r2, c.cutsq_bits) ? en : 0.0) + qr;
              return en;
            };
            if (uni) {
              if (S2)
                s6 += r6inv;
              else
                e0 += energy();
              npair++;
              if (img) {  // this lane's column: no other lane writes it
                double* m = &sev[w][0][lane];
                m[1 * 32] = __fma_rn(-shx, gx, m[1 * 32]);
                m[2 * 32] = __fma_rn(-shy, gy, m[2 * 32]);
                m[3 * 32] = __fma_rn(-shz, gz, m[3 * 32]);
                m[4 * 32] = __fma_rn(-shx, gy, m[4 * 32]);
                m[5 * 32] = __fma_rn(-shx, gz, m[5 * 32]);
                m[6 * 32] = __fma_rn(-shy, gz, m[6 * 32]);
              }
            } else {
              atomicAdd(&sev[w][0][o], evw * energy());
              atomicAdd(&sev[w][7][o], evw);
              if (img) {
                atomicAdd(&sev[w][1][o], -evw * shx * gx);
                atomicAdd(&sev[w][2][o], -evw * shy * gy);
                atomicAdd(&sev[w][3][o], -evw * shz * gz);
                atomicAdd(&sev[w][4][o], -evw * shx * gy);
                atomicAdd(&sev[w][5][o], -evw * shx * gz);
                atomicAdd(&sev[w][6][o], -evw * shy * gz);
              }
            }
          }
        }
      }
      head[Q] += take;
      __syncwarp();
    };
    const std::integral_constant<int, 0> q0{};
    const std::integral_constant<int, 1> q1{};

    // phase 1: one list entry per lane per round; the survivors are pushed
    // (and full queues drained), so fewer than 32 entries wait before a push
    for (;; q++) {
      if (!__any_sync(0xffffffffu, q < cnt)) break;
      bool cand = false, wrap = false;
      int j = 0;
      if (q < cnt) {
        j = __ldcs(q < nin ? row + (int64_t)q * 32 : skin - (int64_t)(q - nin) * 32);
        const float4 hj = md_ld_hi<0>(a.xs, j);
        float dx = hj.x - hi.x, dy = hj.y - hi.y, dz = hj.z - hi.z;
        wrap = (fabsf(dx) > hm0) | (fabsf(dy) > hm1) | (fabsf(dz) > hm2);
        dx = fabsf(dx) > hf0 ? dx - copysignf(Lf0, dx) : dx;
        dy = fabsf(dy) > hf1 ? dy - copysignf(Lf1, dy) : dy;
        dz = fabsf(dz) > hf2 ? dz - copysignf(Lf2, dz) : dz;
        const float r2f = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, dx * dx));
        const float cut =
            SINGLE ? cut_hi1 : scut[ti * a.nt + MD_TAG_TYPE(__float_as_int(hj.w))];
        cand = r2f <= cut;
      }
      const unsigned lt = (1u << lane) - 1u;
      const unsigned b0 = __ballot_sync(0xffffffffu, cand && !wrap);
      const unsigned b1 = __ballot_sync(0xffffffffu, cand && wrap);
      if (cand) {
        const int Q = wrap ? 1 : 0;
        const unsigned slot = tail[Q] + __popc((wrap ? b1 : b0) & lt);
        qj[Q][w][slot % MD_Q_CAP] = j;
        qo[Q][w][slot % MD_Q_CAP] = (unsigned char)lane;
      }
      tail[0] += __popc(b0);
      tail[1] += __popc(b1);
      __syncwarp();
      if (tail[0] - head[0] >= 32) drain(q0, 32);
      if (tail[1] - head[1] >= 32) drain(q1, 32);
    }
    while (tail[0] != head[0]) drain(q0, tail[0] - head[0] < 32 ? tail[0] - head[0] : 32);
    while (tail[1] != head[1]) drain(q1, tail[1] - head[1] < 32 ? tail[1] - head[1] : 32);
    __syncwarp();
    if (EV) {
      const int slot = (int)(((int64_t)tile * (MD_BLOCK / 32) + w) % a.ev_spread);
      double ev[8];
      if (uni) {  // every lane's sums belong to box rep0
        ev[0] = S2 ? -0.5 * a.c1.lj4 * s6 : e0;
  #pragma unroll
        for (int k = 1; k < 7; k++) ev[k] = sev[w][k][lane];
  #pragma unroll
        for (int k = 0; k < 7; k++) ev[k] *= evw;
        ev[7] = evw * (double)npair;
        md_warp_add_rep<8>(ev, rep0, a.ev, a.ev_spread, slot);
      } else {
  #pragma unroll
        for (int k = 0; k < 8; k++) ev[k] = sev[w][k][lane];
        md_warp_add_rep<8>(ev, active ? rep_i : -1, a.ev, a.ev_spread, slot);
      }
    }
  }
}

// Resident blocks per SM the register allocation must allow.
// The energy/virial launches: at 4M atoms (fcc liquid) 7, 8 and 10 blocks
// (72, 64 and 48 registers; 48 spills a few words) measured 3.49, 3.37 and
// 3.60 ms per half-list launch and 5.80, 5.60 and 5.38 ms per full-list one.
constexpr int md_pair_q_minb(bool half, bool ev) { return ev ? (half ? 8 : 10) : MD_Q_MINB; }

template <bool HALF, bool EV, bool SINGLE, bool COUL>
__global__ void __launch_bounds__(MD_BLOCK, md_pair_q_minb(HALF, EV))
    k_pair_q(const PairArgs a, const float cut_hi1, const float* __restrict__ cut_hi_tab) {
  if (md_stopped(a.stop)) return;
  md_pair_q_tiles<HALF, EV, SINGLE, COUL>(a, cut_hi1, cut_hi_tab);
}

template <bool HALF, bool EV, bool SINGLE, bool COUL>
cudaError_t md_pair_q_launch5(const PairArgs& a, float cut1, const float* cut_tab,
                              unsigned blocks, cudaStream_t s, int carve) {
  int occ = 1;
  cudaError_t e =
      md_prepare_kernel((const void*)k_pair_q<HALF, EV, SINGLE, COUL>, carve, 0, &occ);
  if (e != cudaSuccess) return e;
  if (a.tile_ctr) {
    const unsigned cap = (unsigned)(a.nslots * occ);
    if (blocks > cap) blocks = cap;
  }
  k_pair_q<HALF, EV, SINGLE, COUL><<<blocks, MD_BLOCK, 0, s>>>(a, cut1, cut_tab);
  return cudaGetLastError();
}

template <bool COUL>
cudaError_t md_pair_q_launch_t(const PairArgs& a, bool half, bool ev, bool single, float cut1,
                               const float* cut_tab, unsigned blocks, cudaStream_t s,
                               int carve) {
  if (half) {
    if (ev)
      return single ? md_pair_q_launch5<true, true, true, COUL>(a, cut1, cut_tab, blocks, s, carve)
                    : md_pair_q_launch5<true, true, false, COUL>(a, cut1, cut_tab, blocks, s, carve);
    return single ? md_pair_q_launch5<true, false, true, COUL>(a, cut1, cut_tab, blocks, s, carve)
                  : md_pair_q_launch5<true, false, false, COUL>(a, cut1, cut_tab, blocks, s, carve);
  }
  if (ev)
    return single ? md_pair_q_launch5<false, true, true, COUL>(a, cut1, cut_tab, blocks, s, carve)
                  : md_pair_q_launch5<false, true, false, COUL>(a, cut1, cut_tab, blocks, s, carve);
  return single ? md_pair_q_launch5<false, false, true, COUL>(a, cut1, cut_tab, blocks, s, carve)
                : md_pair_q_launch5<false, false, false, COUL>(a, cut1, cut_tab, blocks, s, carve);
}

// md_pair_fp64.cu, and the lj/cut/coul/cut style (md_pair_coul.cu)
cudaError_t md_pair_q_launch(const PairArgs& a, bool half, bool ev, bool single, float cut1,
                             const float* cut_tab, unsigned blocks, cudaStream_t s, int carve);
cudaError_t md_pair_q_coul_launch(const PairArgs& a, bool half, bool ev, bool single,
                                  float cut1, const float* cut_tab, unsigned blocks,
                                  cudaStream_t s, int carve);
