// Host side of the 2D batched periodic-RVE solver: shared-memory and scratch sizes and the
// dispatch to the kernel instantiations.  Each instantiation is compiled in a translation unit
// of its own (rve2d_k_*.cu) so that the builds run in parallel; the device code is rve2d.cuh.
#include "rve2d_fp64.cuh"

#include <algorithm>

namespace fehmm {

cudaError_t rve2d_launch_mixed_mg_nh(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream);
cudaError_t rve2d_launch_mixed_mg_nh_small(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream);
cudaError_t rve2d_launch_mixed_mg_svk(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream);
cudaError_t rve2d_launch_mixed_mg_svk_small(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream);
cudaError_t rve2d_launch_mixed_bj_nh(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream);
cudaError_t rve2d_launch_mixed_bj_svk(const Rve2dArgs& a, int n_blocks, size_t smem, cudaStream_t stream);
cudaError_t rve2d_launch_fp64_mg_nh(const Rve2dArgs& a, int n_blocks, cudaStream_t stream);
cudaError_t rve2d_launch_fp64_mg_svk(const Rve2dArgs& a, int n_blocks, cudaStream_t stream);
cudaError_t rve2d_launch_fp64_bj_nh(const Rve2dArgs& a, int n_blocks, cudaStream_t stream);
cudaError_t rve2d_launch_fp64_bj_svk(const Rve2dArgs& a, int n_blocks, cudaStream_t stream);
cudaError_t rve2d_launch_fp64_fixed_nh(const Rve2dArgs& a, int n_blocks, cudaStream_t stream);

size_t rve2d_smem_bytes(int nn_max, bool mixed) {
  return mixed ? offsets2d<float>(nn_max).total : offsets_d2(nn_max, true).total;
}

long long rve2d_scratch_stride(int nn_max, bool mixed) {
  // mixed: staged element tangents [36][nn_max] and the coarse element matrices of the multigrid
  return mixed ? 36LL * nn_max + mg_slow_max(nn_max) : scratch_d2(nn_max, true);
}

size_t rve2d_scratch_bytes(int nn_max, bool mixed, int n_blocks) {
  return (mixed ? sizeof(float) : sizeof(double)) * (size_t)rve2d_scratch_stride(nn_max, mixed) * n_blocks;
}

// Blocks of RVEs with nn nodes that one SM holds: 128 registers per thread, the shared memory of the
// layout plus 1 KB the driver takes per block.
int rve2d_blocks_per_sm(int nn, bool mixed) {
  const int regs = 65536 / (128 * (mixed ? threads2d<float>(nn) : threads_d2(nn)));
  const int smem = (int)((228 * 1024) / (rve2d_smem_bytes(nn, mixed) + 1024));
  return std::max(1, std::min(regs, smem));
}

// The multigrid and block-Jacobi paths and the two laws are separate instantiations, so each is
// register-allocated on its own.  Only six grids have a multigrid hierarchy (n = 2^k m, m = 3 or 4): in
// mixed precision each is an instantiation with the grid size known when compiling, which makes every
// level's offsets, row and column indices constants.  Any other grid takes the block-Jacobi kernel.
cudaError_t rve2d_launch(const Rve2dArgs& a, bool mixed, int n_blocks, cudaStream_t stream) {
  const size_t smem = rve2d_smem_bytes(a.nn_max, mixed);
  const bool svk = a.law == 1;
  int n = 2;
  while (n * n < a.nn_max) ++n;
  const bool mg = a.mg && mg_levels(n) > 0;
  if (mixed) {
    if (mg && n <= 16) return svk ? rve2d_launch_mixed_mg_svk_small(a, n_blocks, smem, stream) : rve2d_launch_mixed_mg_nh_small(a, n_blocks, smem, stream);
    if (mg) return svk ? rve2d_launch_mixed_mg_svk(a, n_blocks, smem, stream) : rve2d_launch_mixed_mg_nh(a, n_blocks, smem, stream);
    return svk ? rve2d_launch_mixed_bj_svk(a, n_blocks, smem, stream) : rve2d_launch_mixed_bj_nh(a, n_blocks, smem, stream);
  }
  if (mg) return svk ? rve2d_launch_fp64_mg_svk(a, n_blocks, stream) : rve2d_launch_fp64_mg_nh(a, n_blocks, stream);
  return svk ? rve2d_launch_fp64_bj_svk(a, n_blocks, stream) : rve2d_launch_fp64_bj_nh(a, n_blocks, stream);
}

cudaError_t rve2d_launch_fixed_fp64(const Rve2dArgs& a, int n_blocks, cudaStream_t stream) {
  return rve2d_launch_fp64_fixed_nh(a, n_blocks, stream);
}

}  // namespace fehmm
