// md_neigh.cu -- cell binning by counting sort and prefix scan, and the
// neighbor-list build with skin (arXiv 2508.13523, Sec. 4: a list built and
// periodically updated; Sec. 4.1: half lists with each pair once, full lists
// with each pair in both atoms' lists; App. B: 64-bit row offsets with
// 32-bit column indices).
//
// Rebuild pipeline, all on the context's stream:
//   k_wrap_bin    wrap x into [0,L) (x - L*floor(x/L), L -> 0), cell index,
//                 histogram with atomics (rank of each atom in its cell)
//   scan          exclusive prefix sum of the histogram -> cell starts
//   k_scatter     perm[start[c] + rank] = atom
//   k_sort_gather permuted copies of x, v, f, id, cell; an atom's place in its
//                 cell is the number of the cell's atoms with a smaller
//                 index: a stable, deterministic counting sort
//   k_restore     the copies back, so that every pointer stays fixed (CUDA
//                 graphs capture them), with the position records (xs,
//                 md_split; xq) and the build snapshot (xb)
//   k_build_cell  27-cell stencil (one cell along an axis with < 3 cells), one
//                 block per cell; sparse boxes: k_build, one thread per atom.
//                 FP32 test with certified bounds, FP64 only inside the band
//                 where FP32 cannot decide; writes tiled lists
// The host then reads the largest count; if it exceeds the capacity the
// list storage grows and k_build runs again.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "md_device.cuh"
#include "md_fx_coef.h"
#include "md_internal.cuh"

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// x - L*floor(x/L) with correctly rounded division and product (no
// contraction); a result equal to L becomes 0.  For 0 <= x < L the rounded
// quotient is below 1 (x <= L - ulp(L) / 2, and 1 - 2^-53 is a double) and x
// stays: an integer test instead of the division.
__device__ __forceinline__ double wrap1(double x, double L) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  if (b < (unsigned long long)__double_as_longlong(L)) return x;
  double q = floor(__ddiv_rn(x, L));
  double w = __dsub_rn(x, __dmul_rn(L, q));
  return (w == L) ? 0.0 : w;
}

__device__ __forceinline__ int cell_coord(double x, double cinv, int nc) {
  int c = (int)(x * cinv);  // x >= 0 after the wrap: truncation is floor
  return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

__global__ void k_wrap_bin(double4_32a* __restrict__ x4, int64_t n,
                           const RepGeo* __restrict__ rep, int32_t* __restrict__ cell,
                           int32_t* __restrict__ cnt, int32_t* __restrict__ rank) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double4_32a p = x4[i];
  const RepGeo& g = rep[MD_TAG_REP(md_tag_of(p))];
  p.x = wrap1(p.x, g.L[0]);
  p.y = wrap1(p.y, g.L[1]);
  p.z = wrap1(p.z, g.L[2]);
  x4[i] = p;
  int cx = cell_coord(p.x, g.cinv[0], g.nc[0]);
  int cy = cell_coord(p.y, g.cinv[1], g.nc[1]);
  int cz = cell_coord(p.z, g.cinv[2], g.nc[2]);
  int c = md_cell_index(g, cx, cy, cz);
  cell[i] = c;
  rank[i] = atomicAdd(&cnt[c], 1);
}

// ---- exclusive scan (three passes, block sums kept in int64) ---------------
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    T u = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += u;
  }
  return v;
}

// Exclusive scan of the SCAN_TILE items owned by this block; returns the
// block total to thread 0 via *total.
template <typename TIN, typename TOUT>
__device__ void block_scan_tile(const TIN* in, TOUT* out, int64_t n, int64_t base,
                                TOUT carry, int64_t* total) {
  __shared__ int64_t wsum[SCAN_THREADS / 32];
  TOUT v[SCAN_ITEMS];
  TOUT s = 0;
  int64_t first = base + (int64_t)threadIdx.x * SCAN_ITEMS;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; k++) {
    int64_t idx = first + k;
    v[k] = idx < n ? (TOUT)in[idx] : (TOUT)0;
    s += v[k];
  }
  int64_t incl = warp_incl_scan<int64_t>((int64_t)s);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  int64_t woff = 0, btot = 0;
#pragma unroll
  for (int w = 0; w < SCAN_THREADS / 32; w++) {
    if (w < warp) woff += wsum[w];
    btot += wsum[w];
  }
  TOUT run = carry + (TOUT)(woff + incl - (int64_t)s);
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; k++) {
    int64_t idx = first + k;
    if (idx < n) out[idx] = run;
    run += v[k];
  }
  if (threadIdx.x == 0) *total = btot;
  __syncthreads();
}

template <typename TOUT>
__global__ void k_scan_tiles(const int32_t* __restrict__ in, TOUT* __restrict__ out,
                             int64_t n, int64_t* __restrict__ tile_sums) {
  int64_t t;
  block_scan_tile<int32_t, TOUT>(in, out, n, (int64_t)blockIdx.x * SCAN_TILE, (TOUT)0, &t);
  if (threadIdx.x == 0) {
    tile_sums[blockIdx.x] = t;
    if (gridDim.x == 1) out[n] = (TOUT)t;  // one tile: the scan is complete
  }
}

// One block: exclusive scan of the tile sums in place, any count.
__global__ void k_scan_top(int64_t* __restrict__ sums, int64_t m) {
  __shared__ int64_t carry_s;
  if (threadIdx.x == 0) carry_s = 0;
  __syncthreads();
  for (int64_t base = 0; base < m; base += SCAN_TILE) {
    int64_t t;
    int64_t carry = carry_s;
    block_scan_tile<int64_t, int64_t>(sums, sums, m, base, carry, &t);
    if (threadIdx.x == 0) carry_s = carry + t;
    __syncthreads();
  }
  if (threadIdx.x == 0) sums[m] = carry_s;
}

template <typename TOUT>
__global__ void k_scan_add(TOUT* __restrict__ out, int64_t n,
                           const int64_t* __restrict__ tile_off) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] += (TOUT)tile_off[i / SCAN_TILE];
  if (i == 0) {
    int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    out[n] = (TOUT)tile_off[tiles];
  }
}

__global__ void k_scatter(const int32_t* __restrict__ cell, const int32_t* __restrict__ rank,
                          const int32_t* __restrict__ start, int32_t* __restrict__ perm,
                          int64_t n) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  perm[start[cell[i]] + rank[i]] = (int32_t)i;
}

__global__ void k_sort_gather(const int32_t* __restrict__ perm,
                              const int32_t* __restrict__ start, int64_t n,
                              const double4_32a* __restrict__ x4, const double* __restrict__ v,
                              const double* __restrict__ f, const int32_t* __restrict__ id,
                              const int32_t* __restrict__ cell, double4_32a* __restrict__ x4n,
                              double* __restrict__ vn, double* __restrict__ fn,
                              int32_t* __restrict__ idn, int32_t* __restrict__ celln) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int o = perm[s];
  const double4_32a x = x4[o];
  const double vx = v[o], vy = v[n + o], vz = v[2 * n + o];
  const double fx = f[o], fy = f[n + o], fz = f[2 * n + o];
  const int ido = id[o], c = cell[o];
  const int b = start[c], e = start[c + 1];
  int64_t p = b;
  for (int q = b; q < e; q++) p += perm[q] < o;
  x4n[p] = x;
  vn[p] = vx;
  vn[n + p] = vy;
  vn[2 * n + p] = vz;
  fn[p] = fx;
  fn[n + p] = fy;
  fn[2 * n + p] = fz;
  idn[p] = ido;
  celln[p] = c;
}

__global__ void k_restore(const double4_32a* __restrict__ x4n, const double* __restrict__ vn,
                          const double* __restrict__ fn, const int32_t* __restrict__ idn,
                          const int32_t* __restrict__ celln, int64_t n,
                          double4_32a* __restrict__ x4, double* __restrict__ v,
                          double* __restrict__ f, int32_t* __restrict__ id,
                          int32_t* __restrict__ cell, XSplit* __restrict__ xs,
                          XSplit* __restrict__ xb, XFix* __restrict__ xq, const XGrid gr) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double4_32a p = x4n[i];
  const double vx = vn[i], vy = vn[n + i], vz = vn[2 * n + i];
  const double fx = fn[i], fy = fn[n + i], fz = fn[2 * n + i];
  const int32_t k = idn[i], c = celln[i];
  x4[i] = p;
  v[i] = vx;
  v[n + i] = vy;
  v[2 * n + i] = vz;
  f[i] = fx;
  f[n + i] = fy;
  f[2 * n + i] = fz;
  id[i] = k;
  cell[i] = c;
  md_store_pos(p, gr, xs, xq, i, xb);
}

// md_ld_hi with the records' kind (hs) at run time
__device__ __forceinline__ float4 ld_hi(const XSplit* xs, int64_t i, int hs) {
  return __ldg(reinterpret_cast<const float4*>(xs) + (i << hs));
}

// FP32 minimum image of one component (float positions in [0, L]).
__device__ __forceinline__ float min_image_f(float d, float L, float halfL) {
  return fabsf(d) > halfL ? d - copysignf(L, d) : d;
}

// Neighbor build, one thread per atom (cell-sorted order).  Candidate j is
// kept iff its FP64 minimum-image r2 < rlist2, where
//   r2 = fma(dz,dz, fma(dy,dy, dx*dx)),  d = x_j - x_i - L*rint((x_j-x_i)/L).
// The FP32 distance of the hi parts decides whenever it is outside
// [lo2f, hi2f]; those bounds are certified on the host from the FP32
// rounding of positions and arithmetic, so the kept set is exactly the FP64
// one.  Half list: only the pairs i owns (md_owns), each pair once.
// Row order: pairs with r2f < rc^2 of their type pair ("inner") from the
// front, the rest ("skin") from the back, so that in the force kernel the
// inner loop is almost branch-free and the skin loop mostly skips the force.
template <bool HALF>
__global__ void __launch_bounds__(MD_BLOCK)
    k_build(const double4_32a* __restrict__ x4, const XSplit* __restrict__ xs, int hs,
            const int32_t* __restrict__ cell, const int32_t* __restrict__ start, int64_t n,
            Geo gg, const RepGeo* __restrict__ rep, int32_t* __restrict__ numneigh,
            int32_t* __restrict__ nbr, int maxneigh, unsigned int* __restrict__ maxcount) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 hi = ld_hi(xs, i, hs);
  const int tag = __float_as_int(hi.w);
  const int ti = MD_TAG_TYPE(tag);
  const RepGeo& g = rep[MD_TAG_REP(tag)];  // fields read on use (fewer registers)
  int cx, cy, cz;
  md_cell_coords(g, cell[i], cx, cy, cz);
  int32_t* out = nbr + (i >> 5) * (int64_t)maxneigh * 32 + (i & 31);
  int nin = 0, nsk = 0;  // entries written (nin + nsk <= maxneigh)
  int total = 0;         // entries found
  int cand = -1;         // atoms in the stencil's cells other than i
  double4_32a xi;
  bool have_xi = false;
  const int ii = (int)i;

  // candidate j at FP32 separation (dx, dy, dz) of the hi parts, nearest image
  auto consider = [&](int j, float dx, float dy, float dz, float wj) {
    const float r2f = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, dx * dx));
    if (r2f > gg.hi2f) return;
    bool keep = true;
    if (r2f >= gg.lo2f) {  // undecided in FP32: the exact FP64 test
      if (!have_xi) {
        xi = x4[i];
        have_xi = true;
      }
      const double4_32a xj = x4[j];
      const double ex = md_min_image(__dsub_rn(xj.x, xi.x), g.L[0], g.halfL_bits[0]);
      const double ey = md_min_image(__dsub_rn(xj.y, xi.y), g.L[1], g.halfL_bits[1]);
      const double ez = md_min_image(__dsub_rn(xj.z, xi.z), g.L[2], g.halfL_bits[2]);
      keep = md_lt_pos(md_r2(ex, ey, ez), gg.rlist2_bits);
    }
    if (keep) {
      const bool inner = r2f < gg.cutsqf[ti * gg.nt + MD_TAG_TYPE(__float_as_int(wj))];
      if (nin + nsk < maxneigh) {
        if (inner)
          out[(int64_t)(nin++) * 32] = j;
        else
          out[(int64_t)(maxneigh - 1 - nsk++) * 32] = j;
      }
      total++;
    }
  };

  if (g.nc[0] >= 3 && g.nc[1] >= 3 && g.nc[2] >= 3) {
    // Every axis has >= 3 cells of side >= rlist: each stencil cell is one
    // periodic image, so the image shift (0 or -+L) is fixed per cell and
    // added to the separation exactly as the per-candidate minimum image
    // would (the same two FP32 roundings).  Cells along z that are adjacent
    // in the sorted order and share the shift are scanned as one run.
    // Half list: i owns j < i iff i + j is odd and j > i iff i + j is even
    // (md_owns), so each run is walked with stride 2 on the owned parity.
    auto run = [&](int b, int e, float sx, float sy, float sz) {
      auto visit = [&](int j) {
        const float4 hj = ld_hi(xs, j, hs);
        consider(j, __fadd_rn(__fsub_rn(hj.x, hi.x), sx), __fadd_rn(__fsub_rn(hj.y, hi.y), sy),
                 __fadd_rn(__fsub_rn(hj.z, hi.z), sz), hj.w);
      };
      // one loop per run, so that lanes of the same cell (same run, different
      // i) run the same number of iterations
      if (HALF) {
        const int le = min(e, ii);                   // owned j < i: parity of i + 1
        const int j0 = b + ((b ^ (ii + 1)) & 1);
        const int nlo = le > j0 ? (le - j0 + 1) >> 1 : 0;
        const int hb = max(b, ii + 1);               // owned j > i: parity of i
        const int j1 = hb + ((hb ^ ii) & 1);
        const int nhi = e > j1 ? (e - j1 + 1) >> 1 : 0;
        for (int t = 0; t < nlo + nhi; t++) visit(t < nlo ? j0 + 2 * t : j1 + 2 * (t - nlo));
      } else {
        const bool self = ii >= b && ii < e;
        const int cnt = e - b - (self ? 1 : 0);
        for (int t = 0; t < cnt; t++) visit(b + t + ((self && b + t >= ii) ? 1 : 0));
      }
    };
    for (int ox = -1; ox <= 1; ox++) {
      int qx = cx + ox;
      float sx = 0.f;
      if (qx < 0) { qx += g.nc[0]; sx = -g.Lf[0]; }
      else if (qx >= g.nc[0]) { qx -= g.nc[0]; sx = g.Lf[0]; }
      for (int oy = -1; oy <= 1; oy++) {
        int qy = cy + oy;
        float sy = 0.f;
        if (qy < 0) { qy += g.nc[1]; sy = -g.Lf[1]; }
        else if (qy >= g.nc[1]) { qy -= g.nc[1]; sy = g.Lf[1]; }
        int rb = 0, re = 0;
        float rs = 0.f;
        bool open = false;
        for (int oz = -1; oz <= 1; oz++) {
          int qz = cz + oz;
          float sz = 0.f;
          if (qz < 0) { qz += g.nc[2]; sz = -g.Lf[2]; }
          else if (qz >= g.nc[2]) { qz -= g.nc[2]; sz = g.Lf[2]; }
          const int q = md_cell_index(g, qx, qy, qz);
          const int b = start[q], e = start[q + 1];
          cand += e - b;
          if (open && b == re && sz == rs) {
            re = e;
          } else {
            if (open) run(rb, re, sx, sy, rs);
            rb = b;
            re = e;
            rs = sz;
            open = true;
          }
        }
        run(rb, re, sx, sy, rs);
      }
    }
  } else {
    // some axis has a single cell: per-candidate minimum image
    for (int ox = g.lo[0]; ox <= g.hi[0]; ox++) {
      int qx = cx + ox;
      qx = qx < 0 ? qx + g.nc[0] : (qx >= g.nc[0] ? qx - g.nc[0] : qx);
      for (int oy = g.lo[1]; oy <= g.hi[1]; oy++) {
        int qy = cy + oy;
        qy = qy < 0 ? qy + g.nc[1] : (qy >= g.nc[1] ? qy - g.nc[1] : qy);
        for (int oz = g.lo[2]; oz <= g.hi[2]; oz++) {
          int qz = cz + oz;
          qz = qz < 0 ? qz + g.nc[2] : (qz >= g.nc[2] ? qz - g.nc[2] : qz);
          const int q = md_cell_index(g, qx, qy, qz);
          const int b = start[q], e = start[q + 1];
          cand += e - b;
          for (int j = b; j < e; j++) {
            if (j == ii) continue;
            if (HALF && !md_owns(ii, j)) continue;
            const float4 hj = ld_hi(xs, j, hs);
            consider(j, min_image_f(hj.x - hi.x, g.Lf[0], g.halfLf[0]),
                     min_image_f(hj.y - hi.y, g.Lf[1], g.halfLf[1]),
                     min_image_f(hj.z - hi.z, g.Lf[2], g.halfLf[2]), hj.w);
          }
        }
      }
    }
  }
  // on overflow the rows are incomplete (but in bounds); the host sees
  // total > maxneigh, grows the list and rebuilds
  numneigh[i] = nin;
  numneigh[n + i] = nsk;
  atomicMax(maxcount, (unsigned int)total);
  // every pair of atom i in any list built now joins i to a stencil
  // candidate, so cand bounds the force contributions atom i receives in
  // one pair launch (the range of the fixed-point accumulators)
  atomicMax(maxcount + 1, (unsigned int)cand);
}

// Neighbor build, one block per cell: the cell's stencil atoms (FP32 hi
// parts, image shift added) are staged in shared memory, a warp tests 32 of
// them (one per lane) against each atom of the cell in turn and keeps the
// ballots, and then lane a writes atom a's row from its ballots, so that the
// rows of consecutive atoms are written together.  Membership and row parts
// are those of k_build: FP32 decides outside [lo2f, hi2f], the exact FP64 test
// inside.  Row order: stencil cells in order, ascending index in a cell.
// Half list: the atoms that an even i owns (md_owns) are the even j of later
// cells and the odd j of earlier ones, and the reverse for an odd i; so the
// candidates are staged as two lists, each tested against the cell's atoms of
// one parity only (the own cell's atoms are in both and tested one by one).
constexpr int BC_WARPS = MD_BLOCK / 32;
constexpr int BC_CAP = 768;           // staged candidates (half list: two lists of half as many)
constexpr int BC_CHUNKS = BC_CAP / 32;
constexpr int BC_OWN = 0;             // the own cell comes first among the 27

template <bool HALF, bool SINGLE>
__global__ void __launch_bounds__(MD_BLOCK)
    k_build_cell(const double4_32a* __restrict__ x4, const XSplit* __restrict__ xs, int hs,
                 const int32_t* __restrict__ start, int64_t n, const Geo gg,
                 const RepGeo* __restrict__ rep, int32_t* __restrict__ numneigh,
                 int32_t* __restrict__ nbr, int maxneigh, unsigned int* __restrict__ maxcount) {
  constexpr int NL = HALF ? 2 : 1;                // candidate lists
  constexpr int LCAP = BC_CAP / NL;               // slots of a list
  constexpr int LCH = BC_CHUNKS / NL;             // its chunks of 32
  __shared__ float4 cx[BC_CAP];                   // x, y, z, tag
  __shared__ int cj[BC_CAP];
  __shared__ float4 own[32];
  __shared__ uint2 mask[LCH][32];  // ballots: kept, kept and inside rc
  __shared__ int s_b[27], s_e[27], s_off[NL][28];
  __shared__ float s_sh[27][3];
  __shared__ float scut[MD_MAX_TYPES * MD_MAX_TYPES];
  __shared__ int part_in[BC_WARPS][32], part_sk[BC_WARPS][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ob = start[blockIdx.x], oe = start[blockIdx.x + 1];
  if (ob + (int)blockIdx.y * 32 >= oe) return;
  const RepGeo& g = rep[MD_TAG_REP(__float_as_int(ld_hi(xs, ob, hs).w))];
  const bool img = g.nc[0] < 3 || g.nc[1] < 3 || g.nc[2] < 3;  // minimum image per pair
  const bool one = g.nc[0] * g.nc[1] * g.nc[2] == 1;  // the box is one cell, its own stencil
  if (threadIdx.x < gg.nt * gg.nt) scut[threadIdx.x] = gg.cutsqf[threadIdx.x];
  const float cut1 = gg.cutsqf[0];
  // the stencil's cells: their atoms, image shifts and places in the lists
  int cand = 0;
  if (w == 0) {
    int b = 0, e = 0;
    if (lane < 27) {
      int c0[3];
      md_cell_coords(g, (int)blockIdx.x, c0[0], c0[1], c0[2]);
      const int q27 = lane == BC_OWN ? 13 : (lane <= 13 ? lane - 1 : lane);
      const int o[3] = {q27 / 9 - 1, q27 / 3 % 3 - 1, q27 % 3 - 1};
      bool in = true;
      for (int a = 0; a < 3; a++) {
        in = in && o[a] >= g.lo[a] && o[a] <= g.hi[a];
        int q = c0[a] + o[a];
        float s = 0.f;
        if (q < 0) {
          q += g.nc[a];
          s = -g.Lf[a];
        } else if (q >= g.nc[a]) {
          q -= g.nc[a];
          s = g.Lf[a];
        }
        c0[a] = q;
        s_sh[lane][a] = img ? 0.f : s;
      }
      if (in) {
        const int q = md_cell_index(g, c0[0], c0[1], c0[2]);
        b = start[q];
        e = start[q + 1];
      }
      s_b[lane] = b;
      s_e[lane] = e;
    }
    cand = e - b;
#pragma unroll
    for (int l = 0; l < NL; l++) {
      // list l holds what atoms of parity l need
      int k = e - b;
      if (HALF && lane != BC_OWN) {
        const int par = b >= oe ? l : 1 - l;  // later cell: own parity
        k = ((e + 1 - par) >> 1) - ((b + 1 - par) >> 1);
      }
      int s = k;
      for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, s, d);
        if (lane >= d) s += up;
      }
      if (lane < 27) s_off[l][lane] = s - k;
      if (lane == 26) s_off[l][27] = s;
    }
    cand = __reduce_add_sync(0xffffffffu, cand);
  }
  __syncthreads();
  int most = 0;
  int len = s_off[0][27];
  if (HALF) len = max(len, s_off[NL - 1][27]);
  for (int i0 = ob + (int)blockIdx.y * 32; i0 < oe; i0 += 32 * (int)gridDim.y) {
    const int na = min(32, oe - i0);
    int nin = 0, nsk = 0;  // lane a: entries of atom i0 + a found so far (all warps alike)
    const int i = i0 + lane;
    int32_t* out = nbr + (int64_t)(i >> 5) * maxneigh * 32 + (i & 31);
    __syncthreads();
    if (threadIdx.x < na) own[threadIdx.x] = ld_hi(xs, i0 + (int)threadIdx.x, hs);
    for (int p0 = 0; p0 < len; p0 += LCAP) {
      // stage the candidates of slots p0 .. p0 + LCAP - 1 of each list
      if (one) {  // (a warp per cell would leave one warp to stage the whole box)
        for (int k = p0 + (int)threadIdx.x; k < min(oe - ob, p0 + LCAP); k += MD_BLOCK) {
          const float4 h = ld_hi(xs, ob + k, hs);
#pragma unroll
          for (int l = 0; l < NL; l++) {
            cx[l * LCAP + k - p0] = h;
            cj[l * LCAP + k - p0] = ob + k;
          }
        }
      }
      for (int c = one ? 27 : w; c < 27; c += BC_WARPS) {
        const int b = s_b[c], e = s_e[c];
        const float s0 = s_sh[c][0], s1 = s_sh[c][1], s2 = s_sh[c][2];
        for (int j = b + lane; j < e; j += 32) {
          float4 h = ld_hi(xs, j, hs);
          h.x += s0;
          h.y += s1;
          h.z += s2;
          auto put = [&](int l, int slot) {
            slot -= p0;
            if (slot >= 0 && slot < LCAP) {
              cx[l * LCAP + slot] = h;
              cj[l * LCAP + slot] = j;
            }
          };
          if (!HALF) {
            put(0, s_off[0][c] + (j - b));
          } else if (c == BC_OWN) {
            put(0, s_off[0][c] + (j - b));
            put(NL - 1, s_off[NL - 1][c] + (j - b));
          } else {
            const int l = b >= oe ? (j & 1) : 1 - (j & 1);
            put(l, s_off[l][c] + ((j - b) >> 1));
          }
        }
      }
      __syncthreads();
      // chunks of 32 candidates, one per lane, against the atoms
      for (int ch = w; ch < BC_CHUNKS; ch += BC_WARPS) {
        const int l = HALF ? ch / LCH : 0, c = ch - l * LCH;
        const int left = s_off[l][27] - p0 - 32 * c;  // candidates from this chunk on
        if (left <= 0) continue;
        float4 h = make_float4(3.0e38f, 0.f, 0.f, 0.f);  // no candidate: beyond every cutoff, type 0
        int j = -1;
        if (lane < left) {  // (the slots from there on were never written)
          h = cx[l * LCAP + 32 * c + lane];
          j = cj[l * LCAP + 32 * c + lane];
        }
        const int tj = MD_TAG_TYPE(__float_as_int(h.w));
        const int a0 = HALF ? ((i0 ^ l) & 1) : 0, da = HALF ? 2 : 1;
        // IMG: minimum image per pair; OWN: the chunk holds own-cell atoms (each
        // pair's ownership is tested); EXACT: FP64 where FP32 cannot decide.
        // Returns whether some lane met such a pair.
        auto chunk = [&](auto img_, auto own_, auto exact_) {
          constexpr bool IMG = decltype(img_)::value, OWN = decltype(own_)::value,
                         EXACT = decltype(exact_)::value;
          bool und = false;
#pragma unroll 2
          for (int a = a0; a < na; a += da) {
            const float4 o = own[a];
            float dx = h.x - o.x, dy = h.y - o.y, dz = h.z - o.z;
            if (IMG) {
              dx = min_image_f(dx, g.Lf[0], g.halfLf[0]);
              dy = min_image_f(dy, g.Lf[1], g.halfLf[1]);
              dz = min_image_f(dz, g.Lf[2], g.halfLf[2]);
            }
            const float r2f = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, dx * dx));
            bool keep = r2f < gg.lo2f;
            if (EXACT) {
              if (!keep && r2f <= gg.hi2f) {
                const double4_32a xi = x4[i0 + a], xj = x4[j];
                const double ex = md_min_image(__dsub_rn(xj.x, xi.x), g.L[0], g.halfL_bits[0]);
                const double ey = md_min_image(__dsub_rn(xj.y, xi.y), g.L[1], g.halfL_bits[1]);
                const double ez = md_min_image(__dsub_rn(xj.z, xi.z), g.L[2], g.halfL_bits[2]);
                keep = md_lt_pos(md_r2(ex, ey, ez), gg.rlist2_bits);
              }
            } else {
              und |= !keep & (r2f <= gg.hi2f);
            }
            if (OWN) {
              const int ii = i0 + a;
              keep = keep && j != ii;
              if (HALF && j >= ob && j < oe) keep = keep && md_owns(ii, j);
            }
            const float cut =
                SINGLE ? cut1 : scut[MD_TAG_TYPE(__float_as_int(o.w)) * gg.nt + tj];
            const unsigned int bk = __ballot_sync(0xffffffffu, keep);
            const unsigned int bi = __ballot_sync(0xffffffffu, keep & (r2f < cut));
            if (lane == 0) mask[c][a] = make_uint2(bk, bi);
          }
          return und;
        };
        const std::true_type yes{};
        const std::false_type no{};
        if (img) {
          chunk(yes, yes, yes);
        } else {
          const bool mixed = 32 * c + p0 < s_off[l][BC_OWN + 1];  // own-cell slots come first
          const bool und = mixed ? chunk(no, yes, no) : chunk(no, no, no);
          if (__any_sync(0xffffffffu, und)) chunk(no, yes, yes);
        }
      }
      __syncthreads();
      // each warp writes the entries of a quarter of the chunks
      const int l = HALF ? (i & 1) : 0;
      const int nch = min(LCH, (s_off[l][27] - p0 + 31) >> 5);
      const int c0 = w * nch / BC_WARPS, c1 = (w + 1) * nch / BC_WARPS;
      int pi = 0, ps = 0;
      if (lane < na) {
        for (int c = c0; c < c1; c++) {
          const uint2 m = mask[c][lane];
          pi += __popc(m.y);
          ps += __popc(m.x & ~m.y);
        }
      }
      part_in[w][lane] = pi;
      part_sk[w][lane] = ps;
      __syncthreads();
      int ki = nin, ks = nsk;
#pragma unroll
      for (int q = 0; q < BC_WARPS; q++) {
        const int qi = part_in[q][lane], qs = part_sk[q][lane];
        if (q < w) {
          ki += qi;
          ks += qs;
        }
        nin += qi;
        nsk += qs;
      }
      if (lane < na && nin + nsk <= maxneigh) {
        int32_t* fi = out + (int64_t)ki * 32;
        int32_t* fs = out + (int64_t)(maxneigh - 1 - ks) * 32;
        for (int c = c0; c < c1; c++) {
          const uint2 m = mask[c][lane];
          const int* jt = cj + l * LCAP + 32 * c;
          for (unsigned int k = m.y; k; k &= k - 1, fi += 32) *fi = jt[__ffs(k) - 1];
          for (unsigned int k = m.x & ~m.y; k; k &= k - 1, fs -= 32) *fs = jt[__ffs(k) - 1];
        }
      }
      __syncthreads();
    }
    // on overflow rows are left as they were; the host sees a count above
    // maxneigh, grows the list and rebuilds, or lets nothing read them (list_rc)
    if (w == 0 && lane < na) {
      const int a = min(nin, maxneigh);
      numneigh[i] = a;
      numneigh[n + i] = min(nsk, maxneigh - a);
      most = max(most, nin + nsk);
    }
  }
  if (w == 0) {
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) {
      atomicMax(maxcount, (unsigned int)most);
      // every pair of an atom in any list built now joins it to a stencil
      // candidate, so their number bounds the force contributions an atom
      // receives in one pair launch (the range of the fixed-point accumulators)
      atomicMax(maxcount + 1, (unsigned int)cand);
    }
  }
}

__global__ void k_sum_counts(const int32_t* __restrict__ numneigh, int64_t n,
                             unsigned long long* __restrict__ total) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long v = i < n ? (unsigned long long)numneigh[i] : 0ull;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(total, v);
}

// Row length of each caller-order atom.
__global__ void k_csr_counts(const int32_t* __restrict__ numneigh, const int32_t* __restrict__ id,
                             int64_t n, int32_t* __restrict__ cnt_orig) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  cnt_orig[id[p]] = numneigh[p] + numneigh[n + p];
}

__global__ void k_csr_fill(const int32_t* __restrict__ numneigh, const int32_t* __restrict__ nbr,
                           const int32_t* __restrict__ id, int64_t n, int maxneigh,
                           const int64_t* __restrict__ offsets, int32_t* __restrict__ idx) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int32_t* row = nbr + (p >> 5) * (int64_t)maxneigh * 32 + (p & 31);
  int64_t o = offsets[id[p]];
  const int nin = numneigh[p], nsk = numneigh[n + p];
  for (int k = 0; k < nin; k++) idx[o + k] = id[row[(int64_t)k * 32]];
  for (int k = 0; k < nsk; k++) idx[o + nin + k] = id[row[(int64_t)(maxneigh - 1 - k) * 32]];
}

}  // namespace

// ---- host side -----------------------------------------------------------------

// Tile sums for every scan of the context: over its cells (the rebuild) and
// over its atoms (the list export).  One buffer that stays where it is, because
// the rebuild graph holds its address.
int md_scan_alloc(md_ctx* c) {
  const int64_t most = c->ncell > c->n ? c->ncell : c->n;
  const int64_t tiles = (most + SCAN_TILE - 1) / SCAN_TILE + 1;
  if (cudaMalloc(&c->scan_tmp, sizeof(int64_t) * tiles) == cudaSuccess) return MD_OK;
  c->scan_tmp = nullptr;
  cudaGetLastError();
  return MD_ENOMEM;
}

template <typename TOUT>
static int scan_impl(md_ctx* c, const int32_t* in, TOUT* out, int64_t n) {
  int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
  if (tiles > 0) {
    k_scan_tiles<TOUT><<<(unsigned)tiles, SCAN_THREADS, 0, c->stream>>>(in, out, n, c->scan_tmp);
    c->launches++;
  }
  if (tiles == 1) {
    MD_CUDA(cudaGetLastError());
    return MD_OK;
  }
  k_scan_top<<<1, SCAN_THREADS, 0, c->stream>>>(c->scan_tmp, tiles);
  k_scan_add<TOUT><<<(unsigned)md_blocks(n > 0 ? n : 1), MD_BLOCK, 0, c->stream>>>(out, n,
                                                                                   c->scan_tmp);
  c->launches += 2;
  MD_CUDA(cudaGetLastError());
  return MD_OK;
}

int md_scan_i32(md_ctx* c, const int32_t* in, int32_t* out, int64_t n) {
  return scan_impl<int32_t>(c, in, out, n);
}
int md_scan_i64(md_ctx* c, const int32_t* in, int64_t* out, int64_t n) {
  return scan_impl<int64_t>(c, in, out, n);
}

static int grow_list(md_ctx* c, int new_max) {
  int64_t tiles = (c->n + 31) / 32;
  int64_t need = tiles * 32 * (int64_t)new_max;
  md_drop_graphs(c);  // captured graphs hold the old pointer and capacity
  if (need > c->nbr_alloc) {
    if (c->nbr) cudaFree(c->nbr);
    c->nbr = nullptr;
    c->nbr_alloc = 0;
    if (cudaMalloc(&c->nbr, sizeof(int32_t) * need) != cudaSuccess) {
      c->nbr = nullptr;
      cudaGetLastError();
      return MD_ENOMEM;
    }
    c->nbr_alloc = need;
  }
  c->maxneigh = new_max;
  return MD_OK;
}

void md_drop_segments(md_ctx* c) {
  if (!c->graphs) return;
  for (auto& kv : *c->graphs) cudaGraphExecDestroy(kv.second.first);
  c->graphs->clear();
}

void md_drop_graphs(md_ctx* c) {
  if (c->rebuild_graph) cudaGraphExecDestroy(c->rebuild_graph);
  c->rebuild_graph = nullptr;
  md_drop_segments(c);
}

static int launch_build(md_ctx* c) {
  unsigned nb = (unsigned)md_blocks(c->n);
  const bool half = c->list_kind == MD_LIST_HALF;
  const int hs = c->xq ? 0 : 1;
  // A block per cell costs 4 to 5 ns a cell whatever the cell holds (its set-up
  // is a chain of latencies), a thread per atom 0.3 to 0.6 ns an atom, but at
  // least 50 us.  So few atoms per cell keep one thread per atom, unless the
  // cells are too few to fill the chip.  2,048,000 atoms with rlist 2.8, half
  // list, per atom against per cell: 2.3 atoms a cell 656 against 4,263 us, 9.0
  // 1,232 against 1,577 us, full list there 1,873 against 1,674 us; 256,000
  // atoms, 14.6 a cell 261 against 199 us; 55,296 atoms, half list: 8,000 cells
  // of 6.9 atoms 100 against 88 us, 12,167 cells of 4.5 81 against 103 us.
  if (c->cells_used <= 8192 || c->n >= (half ? 12 : 8) * c->cells_used) {
    // one block per cell and 32 of its atoms; where the fullest box's cells hold
    // more than others' the blocks loop over the rest
    int64_t gy = (c->occ_max + 31) / 32;
    const int64_t most = (8192 + c->n / 8) / c->ncell;
    gy = gy < most ? gy : most;
    gy = gy < 1 ? 1 : gy > 65535 ? 65535 : gy;
    const dim3 grid((unsigned)c->ncell, (unsigned)gy);
    auto kern = half ? (c->nt == 1 ? k_build_cell<true, true> : k_build_cell<true, false>)
                     : (c->nt == 1 ? k_build_cell<false, true> : k_build_cell<false, false>);
    kern<<<grid, MD_BLOCK, 0, c->stream>>>(c->x4, c->xs, hs, c->start, c->n, c->geo, c->rep,
                                           c->numneigh, c->nbr, c->maxneigh, c->dmax + 1);
  } else if (half) {
    k_build<true><<<nb, MD_BLOCK, 0, c->stream>>>(c->x4, c->xs, hs, c->cell, c->start, c->n,
                                                  c->geo, c->rep, c->numneigh, c->nbr,
                                                  c->maxneigh, c->dmax + 1);
  } else {
    k_build<false><<<nb, MD_BLOCK, 0, c->stream>>>(c->x4, c->xs, hs, c->cell, c->start, c->n,
                                                   c->geo, c->rep, c->numneigh, c->nbr,
                                                   c->maxneigh, c->dmax + 1);
  }
  c->launches++;
  MD_CUDA(cudaGetLastError());
  return MD_OK;
}

// The list from the sorted positions; its largest count and number of stencil
// candidates go to the host.
static int enqueue_build(md_ctx* c) {
  MD_CUDA(cudaMemsetAsync(c->dmax, 0, 3 * sizeof(unsigned int), c->stream));
  MD_TRY(launch_build(c));
  MD_CUDA(cudaMemcpyAsync(c->h_pinned + 9, c->dmax + 1, 2 * sizeof(unsigned int),
                          cudaMemcpyDeviceToHost, c->stream));
  return MD_OK;
}

// Wrap, sort and build, all on the stream.
static int enqueue_rebuild(md_ctx* c) {
  const int64_t n = c->n;
  const unsigned nb = (unsigned)md_blocks(n);
  cudaStream_t s = c->stream;
  // dmax[0]: displacement since the previous build, dangerous if > skin/2;
  // dmax[5]: a fused step's barrier gave up
  MD_CUDA(cudaMemcpyAsync(c->h_pinned + 12, c->dmax, 6 * sizeof(unsigned int),
                          cudaMemcpyDeviceToHost, s));
  MD_CUDA(cudaMemsetAsync(c->cnt, 0, sizeof(int32_t) * c->ncell, s));
  k_wrap_bin<<<nb, MD_BLOCK, 0, s>>>(c->x4, n, c->rep, c->cell, c->cnt, c->rank);
  c->launches++;
  MD_TRY(md_scan_i32(c, c->cnt, c->start, c->ncell));
  k_scatter<<<nb, MD_BLOCK, 0, s>>>(c->cell, c->rank, c->start, c->perm, n);
  k_sort_gather<<<nb, MD_BLOCK, 0, s>>>(c->perm, c->start, n, c->x4, c->v, c->f, c->id, c->cell,
                                        c->x4_alt, c->v_alt, c->f_alt, c->id_alt, c->cell_alt);
  k_restore<<<nb, MD_BLOCK, 0, s>>>(c->x4_alt, c->v_alt, c->f_alt, c->id_alt, c->cell_alt, n,
                                    c->x4, c->v, c->f, c->id, c->cell, c->xs, c->xb, c->xq,
                                    c->xgrid);
  c->launches += 3;
  MD_CUDA(cudaGetLastError());
  return enqueue_build(c);
}

// From a context's third rebuild on the sequence is one graph launch (12 small
// operations otherwise, whose launches take longer than their work in small
// boxes: 32,000 atoms 70 -> 62 us a rebuild); the first two run directly, since
// most contexts that only load states never need a third.
static int run_rebuild(md_ctx* c) {
  if (!c->rebuild_graph && c->rebuilds++ >= 2) {
    if (cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();  // a stream that cannot be captured
      return enqueue_rebuild(c);
    }
    const int64_t saved = c->launches;
    const int rc = enqueue_rebuild(c);
    c->rebuild_kernels = (int)(c->launches - saved);
    c->launches = saved;
    cudaGraph_t g = nullptr;
    const cudaError_t e = cudaStreamEndCapture(c->stream, &g);
    if (rc != MD_OK || e != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return rc != MD_OK ? rc : md_cuda_fail(e);
    }
    const cudaError_t ei = cudaGraphInstantiate(&c->rebuild_graph, g, 0);
    cudaGraphDestroy(g);
    if (ei != cudaSuccess) {  // no memory for a graph: without it
      cudaGetLastError();
      c->rebuild_graph = nullptr;
    }
  }
  if (!c->rebuild_graph) return enqueue_rebuild(c);
  MD_CUDA(cudaGraphLaunch(c->rebuild_graph, c->stream));
  c->launches += c->rebuild_kernels;
  return MD_OK;
}

static int rebuild(md_ctx* c) {
  cudaStream_t s = c->stream;
  if (!c->nbr) MD_TRY(grow_list(c, c->maxneigh));  // (an earlier growth found no memory)
  MD_TRY(run_rebuild(c));
  for (int attempt = 0; attempt < 4; attempt++) {
    if (attempt > 0) MD_TRY(enqueue_build(c));
    MD_CUDA(cudaStreamSynchronize(s));
    unsigned int before[6];
    memcpy(before, (const char*)(c->h_pinned + 12), sizeof(before));
    if (before[5]) return MD_ETIMEOUT;
    unsigned int mc;
    memcpy(&mc, (const char*)(c->h_pinned + 9), sizeof(mc));
    c->max_count = (int32_t)mc;
    uint32_t kmax;
    memcpy(&kmax, (const char*)(c->h_pinned + 9) + sizeof(mc), sizeof(kmax));
    c->kmax = kmax;
    if (c->xq && md_fx_dense(kmax) != c->fx_d) MD_TRY(md_upload_fx(c));
    if ((int)mc <= c->maxneigh) {
      float disp2;
      memcpy(&disp2, &before[0], sizeof(disp2));
      double half = 0.5 * c->skin;
      // with check_disp the list is rebuilt before any force evaluation at
      // positions beyond skin/2, so no build is dangerous
      if (c->builds > 0 && !c->check_disp && (double)disp2 > half * half) c->dangerous++;
      c->builds++;
      return MD_OK;
    }
    int grown = (int)(mc + mc / 8 + 8);
    grown = (grown + 7) & ~7;
    MD_TRY(grow_list(c, grown));
  }
  return MD_ENEIGH;
}

// Until a rebuild succeeds again, rows hold stale entries or there are none:
// list_rc keeps them from being read.
int md_rebuild(md_ctx* c) {
  c->list_rc = MD_OK;
  c->list_rc = rebuild(c);
  return c->list_rc;
}

int md_list_entries(md_ctx* c, int64_t* total) {
  MD_TRY(c->list_rc);
  unsigned long long* d = reinterpret_cast<unsigned long long*>(c->i64_tmp);
  MD_CUDA(cudaMemsetAsync(d, 0, sizeof(unsigned long long), c->stream));
  k_sum_counts<<<(unsigned)md_blocks(2 * c->n), MD_BLOCK, 0, c->stream>>>(c->numneigh, 2 * c->n, d);
  c->launches++;
  MD_CUDA(cudaGetLastError());
  MD_CUDA(cudaMemcpyAsync(c->h_pinned + 10, d, sizeof(unsigned long long), cudaMemcpyDeviceToHost,
                          c->stream));
  MD_CUDA(cudaStreamSynchronize(c->stream));
  unsigned long long t;
  memcpy(&t, (const char*)(c->h_pinned + 10), sizeof(t));
  *total = (int64_t)t;
  return MD_OK;
}

int md_list_to_csr(md_ctx* c, int64_t* offsets, int32_t* idx) {
  MD_TRY(c->list_rc);
  const unsigned nb = (unsigned)md_blocks(c->n);
  int32_t* cnt_orig = c->rank;  // rebuild scratch, free between rebuilds
  k_csr_counts<<<nb, MD_BLOCK, 0, c->stream>>>(c->numneigh, c->id, c->n, cnt_orig);
  c->launches++;
  MD_TRY(md_scan_i64(c, cnt_orig, offsets, c->n));
  k_csr_fill<<<nb, MD_BLOCK, 0, c->stream>>>(c->numneigh, c->nbr, c->id, c->n, c->maxneigh,
                                             offsets, idx);
  c->launches++;
  MD_CUDA(cudaGetLastError());
  return MD_OK;
}
