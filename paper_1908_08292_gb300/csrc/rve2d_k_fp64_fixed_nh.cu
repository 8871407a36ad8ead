// 2D RVE kernel instantiations: FP64, neo-Hookean, arrays indexed by quadrature point (grids up to 16), multigrid where
// the grid has a hierarchy and block-Jacobi.
#include "rve2d_fp64.cuh"

namespace fehmm {
cudaError_t rve2d_launch_fp64_fixed_nh(const Rve2dArgs& a, int n_blocks, cudaStream_t stream) {
  if (a.mg && mg_levels(a.fixed_n) > 0) return rve2d_launch_fp64<true, true, 0, 1>(a, n_blocks, stream);
  return rve2d_launch_fp64<true, false, 0, 1>(a, n_blocks, stream);
}
}  // namespace fehmm
