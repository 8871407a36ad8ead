// 2D RVE kernel instantiations: FP64, multigrid, St. Venant-Kirchhoff.
#include "rve2d_fp64.cuh"

namespace fehmm {
cudaError_t rve2d_launch_fp64_mg_svk(const Rve2dArgs& a, int n_blocks, cudaStream_t stream) {
  switch (dofs_per_thread_d2(a.nn_max)) {
    case 1: return rve2d_launch_fp64<false, true, 1, 1>(a, n_blocks, stream);
    case 2: return rve2d_launch_fp64<false, true, 1, 2>(a, n_blocks, stream);
    default: return rve2d_launch_fp64<false, true, 1, 4>(a, n_blocks, stream);
  }
}
}  // namespace fehmm
