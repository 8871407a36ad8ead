// 2D RVE kernel instantiations: FP64, block-Jacobi, neo-Hookean, arrays indexed by quadrature point (grids up to 16).
#include "rve2d_fp64.cuh"

namespace fehmm {
cudaError_t rve2d_launch_fp64_fixed_nh(const Rve2dArgs& a, int n_blocks, cudaStream_t stream) {
  return rve2d_launch_fp64<true, false, 0, 1>(a, n_blocks, stream);
}
}  // namespace fehmm
