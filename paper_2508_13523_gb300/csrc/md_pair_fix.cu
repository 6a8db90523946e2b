// md_pair_fix.cu -- launches of the FP64 contexts' fixed-point pair kernel
// (md_pair_fx.cuh), Eq. 1 alone.
#include "md_pair.cuh"
#include "md_pair_fx.cuh"

cudaError_t md_pair_fx_launch(const PairArgs& a, bool half, bool ev, bool single, int t, int u,
                              float cut1, const float* cut_tab, cudaStream_t s, int carve) {
  if (half)
    return single ? md_pair_fx_launch_t<true, true>(a, ev, t, u, cut1, cut_tab, s, carve)
                  : md_pair_fx_launch_t<true, false>(a, ev, t, u, cut1, cut_tab, s, carve);
  return single ? md_pair_fx_launch_t<false, true>(a, ev, t, u, cut1, cut_tab, s, carve)
                : md_pair_fx_launch_t<false, false>(a, ev, t, u, cut1, cut_tab, s, carve);
}
