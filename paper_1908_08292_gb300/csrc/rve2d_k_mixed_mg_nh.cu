// 2D RVE kernel instantiations: mixed precision, multigrid, neo-Hookean, grids 24 and 32.
#include "rve2d.cuh"

namespace fehmm {
cudaError_t rve2d_launch_mixed_mg_nh(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream) {
  if (a.nn_max == 24 * 24) return rve2d_launch_instance<float, true, 0, 24>(a, n_blocks, smem, stream);
  return rve2d_launch_instance<float, true, 0, 32>(a, n_blocks, smem, stream);
}
}  // namespace fehmm
