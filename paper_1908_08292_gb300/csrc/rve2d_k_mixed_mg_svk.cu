// 2D RVE kernel instantiations: mixed precision, multigrid, St. Venant-Kirchhoff, grids 24 and 32.
#include "rve2d.cuh"

namespace fehmm {
cudaError_t rve2d_launch_mixed_mg_svk(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream) {
  if (a.nn_max == 24 * 24) return rve2d_launch_instance<float, true, 1, 24>(a, n_blocks, smem, stream);
  return rve2d_launch_instance<float, true, 1, 32>(a, n_blocks, smem, stream);
}
}  // namespace fehmm
