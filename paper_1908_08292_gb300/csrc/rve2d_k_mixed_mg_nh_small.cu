// 2D RVE kernel instantiations: mixed precision, multigrid, neo-Hookean, grids 6 to 16.
#include "rve2d.cuh"

namespace fehmm {
cudaError_t rve2d_launch_mixed_mg_nh_small(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream) {
  switch (a.nn_max) {
    case 6 * 6: return rve2d_launch_instance<float, true, 0, 6>(a, n_blocks, smem, stream);
    case 8 * 8: return rve2d_launch_instance<float, true, 0, 8>(a, n_blocks, smem, stream);
    case 12 * 12: return rve2d_launch_instance<float, true, 0, 12>(a, n_blocks, smem, stream);
    default: return rve2d_launch_instance<float, true, 0, 16>(a, n_blocks, smem, stream);
  }
}
}  // namespace fehmm
