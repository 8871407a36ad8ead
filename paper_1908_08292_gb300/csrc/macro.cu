// Macro-scale kernels: Fbar at the macro quadrature points and the HMM assembly of the
// macro residual and tangent on a structured Q1 (2D) / Hex8 (3D) mesh of [0,1]^d.
//
// Paper Sec. 3.1-3.2: Fbar = I + Grad u^H at x_{K_delta_l} (the gradient of the
// linearised macro field, Eq. linearization-uH); f_I = sum_qp omega Pbar Grad N_I, which is
// int B_I^T S^H with S^H = <F>^-1 <P> (Eq. f_I^int, macro-mean-stress); and
// K_IJ = sum_qp omega Grad N_I . Abar . Grad N_J, the RVE-averaged bilinear form of
// Eq. ModifiedBilinearForm-3 assembled as in Eq. Assem_k_T_IK_mac.
//
// The assembly is a graph-coloured scatter: elements are split into 2^d colours by the
// parity of their grid coordinates, so no two elements of one colour share a node and each
// colour's launch adds into f and the CSR values without atomics (deterministic sums).
#include <cuda_runtime.h>
#include <stdint.h>

#include "rve_args.h"

namespace fehmm {
namespace {

__device__ __forceinline__ double gauss01(int g) {
  return g == 0 ? 0.21132486540518711775 : 0.78867513459481288225;
}
__device__ __forceinline__ int cx(int a) { return ((a & 3) == 1 || (a & 3) == 2) ? 1 : 0; }
__device__ __forceinline__ int cy(int a) { return (a & 3) >= 2 ? 1 : 0; }
__device__ __forceinline__ int cz(int a) { return a >= 4 ? 1 : 0; }

// physical gradient of corner a's shape function at Gauss point g
template <int D>
__device__ __forceinline__ void grad_N(int a, int g, const MacroArgs& m, double (&gr)[3]) {
  const double xi[3] = {gauss01(g & 1), gauss01((g >> 1) & 1), D == 3 ? gauss01((g >> 2) & 1) : 0.0};
  const int of[3] = {cx(a), cy(a), cz(a)};
  double phi[3], dphi[3];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    phi[k] = of[k] ? xi[k] : 1.0 - xi[k];
    dphi[k] = of[k] ? 1.0 : -1.0;
  }
#pragma unroll
  for (int k = 0; k < D; ++k) {
    double v = dphi[k] / m.h[k];
#pragma unroll
    for (int l = 0; l < D; ++l)
      if (l != k) v *= phi[l];
    gr[k] = v;
  }
}

template <int D>
__device__ __forceinline__ int corner_node(int e, int a, const MacroArgs& m) {
  const int ex = e % m.nel[0], ey = (e / m.nel[0]) % m.nel[1], ez = D == 3 ? e / (m.nel[0] * m.nel[1]) : 0;
  const int nx1 = m.nel[0] + 1, ny1 = m.nel[1] + 1;
  return (ex + cx(a)) + nx1 * (ey + cy(a)) + (D == 3 ? nx1 * ny1 * (ez + cz(a)) : 0);
}

template <int D>
__global__ void macro_qp_F_kernel(const MacroArgs m) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= m.n_qp) return;
  const int e = q / m.nq, g = q % m.nq;
  double F[D][D];
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int J = 0; J < D; ++J) F[i][J] = (i == J) ? 1.0 : 0.0;
#pragma unroll
  for (int a = 0; a < (1 << D); ++a) {
    double gr[3];
    grad_N<D>(a, g, m, gr);
    const int node = corner_node<D>(e, a, m);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const double ui = m.u[(size_t)node * D + i];
#pragma unroll
      for (int J = 0; J < D; ++J) F[i][J] += ui * gr[J];
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int J = 0; J < D; ++J) m.F[(size_t)q * D * D + i * D + J] = F[i][J];
}

// One block of NEN^2 threads per element, thread (I, J).  FP64-pipe bound (64 cycles per warp instruction on an
// SM sub-partition), so every contraction is done once and shared through shared memory.  On the structured mesh
// dN_I/dx_a is a sign (the side of I along a) times a function of the other coordinates, so the Gauss points
// along a are added first: with c the Gauss points of the other axes,
//   S_a[c][J]_ik = sum over g along a of sum_b A_iakb(g) dN_J/dx_b(g),
//   K_IJ,ik = omega sum_a sum_c dN_I/dx_a(c) S_a[c][J]_ik,
// 84 + 108 FMAs a thread in 3D (contracting both gradients per thread and Gauss point: over 1300).  The nodal
// force: each thread takes one Gauss point of its node I, summed over J.  f and K of 16^3 Hex8 elements,
// with the clearing of both: 960 -> 173 us; of 32 x 32 Q1: 58 -> 40 us.
template <int D>
__global__ void __launch_bounds__(1 << (2 * D)) macro_assemble_kernel(const MacroArgs m, int color) {
  constexpr int NEN = 1 << D, NQ = 1 << D, T = NEN * NEN, D2 = D * D, D4 = D2 * D2, NC = NQ / 2, NS = D * NC * NEN * D2;
  __shared__ double As[NQ][D4 + 1], S[D][NC][NEN][D2], gr[NEN][NQ][D];
  const int t = threadIdx.x, I = t / NEN, J = t % NEN;
  const int c0 = color & 1, c1 = (color >> 1) & 1, c2 = (color >> 2) & 1;
  const int n0 = (m.nel[0] - c0 + 1) / 2, n1 = (m.nel[1] - c1 + 1) / 2;
  const int ke = blockIdx.x, kx = ke % n0, ky = (ke / n0) % n1, kz = ke / (n0 * n1);
  const int e = 2 * kx + c0 + m.nel[0] * (2 * ky + c1 + m.nel[1] * (D == 3 ? 2 * kz + c2 : 0));
  for (int k = t; k < NEN * NQ * D; k += T) (&gr[0][0][0])[k] = m.grad[k];
  if (m.A)
    for (int q = t; q < NQ * D4; q += T) As[q / D4][q % D4] = m.A[(size_t)e * NQ * D4 + q];
  double omega = 1.0;
#pragma unroll
  for (int k = 0; k < D; ++k) omega *= 0.5 * m.h[k];
  __syncthreads();
  // Gauss point with the coordinates c on the axes other than a, s along a (bit k: the axis k)
  auto point = [](int a, int c, int s) { return (c & ((1 << a) - 1)) | (s << a) | ((c >> a) << (a + 1)); };
  if (m.A) {
    for (int q = t; q < NS; q += T) {  // S_a[c][j]_ik
      const int ik = q % D2, j = (q / D2) % NEN, c = (q / (D2 * NEN)) % NC, a = q / (D2 * NEN * NC);
      const int i = ik / D, k = ik % D;
      double v = 0.0;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int g = point(a, c, s);
#pragma unroll
        for (int b = 0; b < D; ++b) v = fma(As[g][((i * D + a) * D + k) * D + b], gr[j][g][b], v);
      }
      S[a][c][j][ik] = v;
    }
  }
  double fb[D];  // Gauss point J's share of node I's force
#pragma unroll
  for (int i = 0; i < D; ++i) {
    fb[i] = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) fb[i] = fma(m.P[((size_t)e * NQ + J) * D2 + i * D + a], gr[I][J][a], fb[i]);
#pragma unroll
    for (int o = 1; o < NEN; o <<= 1) fb[i] += __shfl_xor_sync(T < 32 ? (1u << T) - 1u : 0xffffffffu, fb[i], o);
  }
  __syncthreads();
  if (J == 0) {
    const int nodeI = corner_node<D>(e, I, m);
#pragma unroll
    for (int i = 0; i < D; ++i) m.f[(size_t)nodeI * D + i] += omega * fb[i];
  }
  if (m.A) {
    double Kb[D2];
#pragma unroll
    for (int q = 0; q < D2; ++q) Kb[q] = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const double ga = gr[I][point(a, c, 0)][a];
#pragma unroll
        for (int q = 0; q < D2; ++q) Kb[q] = fma(ga, S[a][c][J][q], Kb[q]);
      }
    const int base = m.blk_base[((size_t)e * NEN + I) * NEN + J];
    const int stride = m.blk_stride[(size_t)e * NEN + I];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int k = 0; k < D; ++k) m.K[base + i * stride + k] += omega * Kb[i * D + k];
  }
}

template <int D>
__global__ void macro_grad_kernel(const MacroArgs m, double* grad) {  // [corner][Gauss point][D], once per mesh
  for (int e = threadIdx.x; e < (1 << D) * (1 << D); e += blockDim.x) {
    double v[3];
    grad_N<D>(e >> D, e & ((1 << D) - 1), m, v);
    for (int k = 0; k < D; ++k) grad[e * D + k] = v[k];
  }
}

// u[dof_k] = scale * value_k on the Dirichlet dofs; du <- 0 everywhere (start of a load step)
__global__ void macro_dirichlet_kernel(double* u, double* du, int n, const int32_t* dofs, const double* vals,
                                       int n_fixed, double scale) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n_fixed) u[dofs[t]] = scale * vals[t];
  if (du)
    for (int i = t; i < n; i += gridDim.x * blockDim.x) du[i] = 0.0;
}

// u += du (du is zero on the Dirichlet dofs)
__global__ void macro_update_kernel(double* u, const double* du, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) u[t] += du[t];
}

// y = scale K x over all rows (CSR; 8 lanes per row, 4 rows per warp, shuffle sum).  The loop
// bound is uniform over each warp (its 4 rows share `base`), so the shuffles see all lanes.
__global__ void macro_spmv_kernel(const int32_t* rowptr, const int32_t* col, const double* K, const double* x,
                                  double scale, double* y, int n) {
  const int lane8 = threadIdx.x & 7, sub = (threadIdx.x & 31) >> 3;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, warps = (gridDim.x * blockDim.x) >> 5;
  for (int base = 4 * warp; base < n; base += 4 * warps) {
    const int i = base + sub;
    double s = 0.0;
    if (i < n)
      for (int k = rowptr[i] + lane8; k < rowptr[i + 1]; k += 8) s = fma(K[k], x[col[k]], s);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (lane8 == 0 && i < n) y[i] = scale * s;
  }
}

}  // namespace

cudaError_t macro_spmv_launch(const int32_t* rowptr, const int32_t* col, const double* K, const double* x,
                              double scale, double* y, int n, cudaStream_t stream) {
  const int threads = 256, rows_per_block = threads / 8;
  int blocks = (n + rows_per_block - 1) / rows_per_block;
  blocks = blocks < 1 ? 1 : (blocks > 1024 ? 1024 : blocks);
  macro_spmv_kernel<<<blocks, threads, 0, stream>>>(rowptr, col, K, x, scale, y, n);
  return cudaGetLastError();
}

cudaError_t macro_dirichlet_launch(double* u, double* du, int n, const int32_t* dofs, const double* vals, int n_fixed,
                                   double scale, cudaStream_t stream) {
  const int work = n_fixed > 0 ? n_fixed : 1;
  const int blocks = (work + 255) / 256 > 0 ? (work + 255) / 256 : 1;
  macro_dirichlet_kernel<<<blocks < 64 ? 64 : blocks, 256, 0, stream>>>(u, du, n, dofs, vals, n_fixed, scale);
  return cudaGetLastError();
}

cudaError_t macro_update_launch(double* u, const double* du, int n, cudaStream_t stream) {
  macro_update_kernel<<<(n + 255) / 256, 256, 0, stream>>>(u, du, n);
  return cudaGetLastError();
}

cudaError_t macro_qp_F_launch(const MacroArgs& m, cudaStream_t stream) {
  const int threads = 128, blocks = (m.n_qp + threads - 1) / threads;
  if (m.dim == 2)
    macro_qp_F_kernel<2><<<blocks, threads, 0, stream>>>(m);
  else
    macro_qp_F_kernel<3><<<blocks, threads, 0, stream>>>(m);
  return cudaGetLastError();
}

cudaError_t macro_grad_launch(const MacroArgs& m, double* grad) {
  if (m.dim == 2)
    macro_grad_kernel<2><<<1, 64>>>(m, grad);
  else
    macro_grad_kernel<3><<<1, 64>>>(m, grad);
  return cudaGetLastError();
}

cudaError_t macro_assemble_launch(const MacroArgs& m, cudaStream_t stream, int* launches) {
  const int ncol = 1 << m.dim;
  for (int c = 0; c < ncol; ++c) {
    const int c0 = c & 1, c1 = (c >> 1) & 1, c2 = (c >> 2) & 1;
    const int n0 = (m.nel[0] - c0 + 1) / 2, n1 = (m.nel[1] - c1 + 1) / 2;
    const int n2 = m.dim == 3 ? (m.nel[2] - c2 + 1) / 2 : 1;
    const int total = n0 * n1 * n2;
    if (total <= 0) continue;
    if (m.dim == 2)
      macro_assemble_kernel<2><<<total, 16, 0, stream>>>(m, c);
    else
      macro_assemble_kernel<3><<<total, 64, 0, stream>>>(m, c);
    const cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    ++*launches;
  }
  return cudaSuccess;
}

}  // namespace fehmm
