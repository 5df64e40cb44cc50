// kern_dry3d.cu -- stage kernels for a dry gas in three dimensions (optional viscosity).
#include "snap_adjoint.cuh"
#include "snap_march.cuh"

namespace snap {

bool find_kernels_dry3d(int f32, int visc, KernelSet *out) {
  using L = Lay<0, 0, true>;
  using A = TileT<8, 8, 4, 256, 2>;  // FP32: 2 CTAs per SM (128 registers)
  using B = TileT<16, 8, 2, 256, 2>;
  using A64 = TileT<8, 8, 4>;
  // inviscid: the march along z first (3 CTAs of 256 threads per SM in FP32), the one-shot tiles
  // for grids too small to fill the SMs with columns
  using M = MarchT<32, 8, 32, 3>;
  using M64 = MarchT<32, 8, 32, 1>;
  if (f32)
    *out = visc ? Family<float, L>::set<true, A, B>() : Family<float, L>::set<false, M, A, B>();
  else
    *out = visc ? Family<double, L>::set<true, A64>() : Family<double, L>::set<false, M64, A64>();
  return true;
}

bool find_adjoint_kernels_dry3d(int f32, AdjKernels *out) {
  using L = Lay<0, 0, true>;
  *out = f32 ? AdjFamily<float, L>::get() : AdjFamily<double, L>::get();
  return true;
}

}  // namespace snap
