// md_pair_fix.cu -- launches of the FP64 contexts' fixed-point pair kernel
// (md_pair_fx.cuh).
#include "md_pair.cuh"
#include "md_pair_fx.cuh"

namespace {

template <bool HALF, bool EV, bool SINGLE, int T, int U>
cudaError_t launch(const PairArgs& a, float cut1, const float* cut_tab, cudaStream_t s,
                   int carve) {
  int occ = 1;
  cudaError_t e =
      md_prepare_kernel((const void*)k_pair_fx<HALF, EV, SINGLE, T, U>, carve, &occ);
  if (e != cudaSuccess) return e;
  unsigned blocks = (unsigned)md_blocks(a.n * T);
  if (a.tile_ctr) {
    const unsigned cap = (unsigned)(a.nslots * occ);
    if (blocks > cap) blocks = cap;
  }
  k_pair_fx<HALF, EV, SINGLE, T, U><<<blocks, MD_BLOCK, 0, s>>>(a, cut1, cut_tab);
  return cudaGetLastError();
}

template <bool HALF, bool EV, bool SINGLE>
cudaError_t launch_t(const PairArgs& a, int t, int u, float cut1, const float* cut_tab,
                     cudaStream_t s, int carve) {
  constexpr int U1 = EV ? 2 : 1;
  if (u == 1) {
    switch (t) {
      case 1: return launch<HALF, EV, SINGLE, 1, U1>(a, cut1, cut_tab, s, carve);
      case 2: return launch<HALF, EV, SINGLE, 2, U1>(a, cut1, cut_tab, s, carve);
      case 4: return launch<HALF, EV, SINGLE, 4, U1>(a, cut1, cut_tab, s, carve);
      case 8: return launch<HALF, EV, SINGLE, 8, U1>(a, cut1, cut_tab, s, carve);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (t) {
    case 1: return launch<HALF, EV, SINGLE, 1, 2>(a, cut1, cut_tab, s, carve);
    case 2: return launch<HALF, EV, SINGLE, 2, 2>(a, cut1, cut_tab, s, carve);
    case 4: return launch<HALF, EV, SINGLE, 4, 2>(a, cut1, cut_tab, s, carve);
    case 8: return launch<HALF, EV, SINGLE, 8, 2>(a, cut1, cut_tab, s, carve);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t md_pair_fx_launch(const PairArgs& a, bool half, bool ev, bool single, int t, int u,
                              float cut1, const float* cut_tab, cudaStream_t s, int carve) {
  if (half) {
    if (ev) return single ? launch_t<true, true, true>(a, t, u, cut1, cut_tab, s, carve)
                          : launch_t<true, true, false>(a, t, u, cut1, cut_tab, s, carve);
    return single ? launch_t<true, false, true>(a, t, u, cut1, cut_tab, s, carve)
                  : launch_t<true, false, false>(a, t, u, cut1, cut_tab, s, carve);
  }
  if (ev) return single ? launch_t<false, true, true>(a, t, u, cut1, cut_tab, s, carve)
                        : launch_t<false, true, false>(a, t, u, cut1, cut_tab, s, carve);
  return single ? launch_t<false, false, true>(a, t, u, cut1, cut_tab, s, carve)
                : launch_t<false, false, false>(a, t, u, cut1, cut_tab, s, carve);
}
