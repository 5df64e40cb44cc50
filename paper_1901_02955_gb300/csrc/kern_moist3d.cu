// kern_moist3d.cu -- stage kernels for two vapours with cloud and precipitation, 3-D.
#include "snap_march.cuh"

namespace snap {

bool find_kernels_moist3d(int f32, int visc, int micro, KernelSet *out) {
  using L = Lay<2, 2, true>;
  // FP32: 8 x 8 x 4 cells, 256 threads, registers capped for 3 CTAs per SM (the compact
  // shared-memory cross fits three); 16 x 8 x 2 for two; FP64 uncapped
  using A = TileT<8, 8, 4, 256, 3>;
  using A64 = TileT<8, 8, 4>;
  using B = TileT<16, 8, 2, 256, 2>;
  // the march along z first, by 16 warps per SM in either shape: 32 x 16 columns convert and
  // reconstruct less halo per cell (Jovian column 256 x 256 x 128 4.19 -> 4.03 ms per step); two
  // CTAs of 32 x 8 wait less at their barriers where grids are small (100 x 90 x 100 678 against 691
  // us) and with the microphysics (radiative-convective 128 x 96 x 128 1051 against 1057 us)
  using M = MarchT<32, 8, 32, 2>;
  using M2 = MarchT<32, 16, 32, 1>;
  using M64 = MarchT<32, 8, 32, 1>;
  if (visc) return false;
  if (micro)  // sedimentation and the Kessler scheme compiled in: the march and one one-shot tile
    *out = f32 ? Family<float, L>::set_micro<M, A>() : Family<double, L>::set_micro<M64, A64>();
  else
    *out = f32 ? Family<float, L>::set<false, M2, M, A, B>() : Family<double, L>::set<false, M64, A64>();
  return true;
}

}  // namespace snap
