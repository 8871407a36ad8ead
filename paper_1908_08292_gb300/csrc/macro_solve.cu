// Macro Newton correction: K_ff du_f = -f_f with du = 0 on the Dirichlet dofs (the linearised
// macro problem, Eq. L(GH) with the tangent of Eq. ModifiedBilinearForm-3 assembled as in
// Eq. Assem_k_T_IK_mac).  Jacobi-preconditioned CG in FP64 over the CSR tangent.
//
// One cooperative launch, one block per SM at most, all co-resident.  The CG is the single-
// reduction form of Chronopoulos and Gear: per iteration the vector updates and u = M^-1 r, the
// exchange of u, the sparse product w = K u together with the partial inner products gamma = r.u and
// delta = w.u, and their sum over the blocks, added in the same order by every block: identical
// decisions in every block.  Fixed rows carry M^-1 = 0 and no product, which keeps their r, u, p, x
// at zero.  The first output is |f_free|_2, the macro convergence measure.
//
// Two kernels.  macro_pcg_resident_kernel (meshes whose rows fit the registers of one block per SM, up to
// 128 rows a block) holds its rows of K and of every vector in registers for the whole solve; blocks
// exchange only u at the block boundaries and the partial sums, both as 16-byte {value, sequence number}
// words that the reader polls, so an exchange is one store and one load through the L2.  An iteration was
// bound by its two grid barriers and by reading K again after each (9 us at 2178 rows); now by those two
// hops (about 0.6 us each) and by the FP64 pipe (64 cycles per warp instruction on an SM sub-partition),
// which the split of the rows over all SMs, the order of the updates (p and x beside the exchange) and
// one lane per inner product keep short.  Per iteration on a GB300: 50 rows 9.0 -> 2.3 us, 2178 rows (2D)
// 9.6 -> 3.5, 9894 rows (2D) 11.3 -> 3.9, 14739 rows (3D) 15.4 -> 8.0.  macro_pcg_kernel: any larger mesh,
// vectors in global memory, two grid barriers per iteration.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "fehmm_device.cuh"
#include "rve_args.h"

namespace cg = cooperative_groups;

namespace fehmm {
namespace {

constexpr int kSolveThreads = 256;
constexpr int kRowLanes = 8;                              // lanes per matrix row in the product
constexpr int kRowsPerBlock = kSolveThreads / kRowLanes;  // 32

// Sum (a, b) over the grid: block sums -> partial[2*block], grid barrier, every block adds the
// partials in index order (warp 0, fixed shuffle tree), so all blocks get identical totals.
// Consecutive calls must use alternate partial buffers: a block may write the next call's
// partials while a slower block still reads this call's, and only a grid barrier of the call
// in between (every call has one) orders the reads of call k before the writes of call k + 2.
__device__ void grid_sum2(double& a, double& b, double* partial, double (*sbuf)[2], cg::grid_group& grid) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    sbuf[warp][0] = a;
    sbuf[warp][1] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0.0, s1 = 0.0;
    for (int k = 0; k < kSolveThreads / 32; ++k) {
      s0 += sbuf[k][0];
      s1 += sbuf[k][1];
    }
    partial[2 * blockIdx.x] = s0;
    partial[2 * blockIdx.x + 1] = s1;
  }
  grid.sync();
  if (warp == 0) {
    double t0 = 0.0, t1 = 0.0;
    for (int j = lane; j < (int)gridDim.x; j += 32) {
      t0 += partial[2 * j];
      t1 += partial[2 * j + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      t0 += __shfl_xor_sync(0xffffffffu, t0, o);
      t1 += __shfl_xor_sync(0xffffffffu, t1, o);
    }
    if (lane == 0) {
      sbuf[0][0] = t0;
      sbuf[0][1] = t1;
    }
  }
  __syncthreads();
  a = sbuf[0][0];
  b = sbuf[0][1];
  __syncthreads();  // sbuf is reused by the next call
}

// w = K u over this block's rows (8 lanes per row); returns this thread's share of w.u.  The
// loop bound is uniform over each warp (its 4 rows share `base`), so the shuffles see all lanes.
__device__ __forceinline__ double spmv_rows(const MacroSolveArgs& a, const double* dinv, const double* u, double* w,
                                            int n) {
  const int lane8 = threadIdx.x % kRowLanes;
  const int warp_rows = (blockIdx.x * kSolveThreads + (threadIdx.x & ~31)) / kRowLanes;  // first row of the warp
  const int sub = (threadIdx.x & 31) / kRowLanes;
  const int n_rows_grid = gridDim.x * kRowsPerBlock;
  double wu = 0.0;
  for (int base = warp_rows; base < n; base += n_rows_grid) {
    const int i = base + sub;
    double s = 0.0;
    if (i < n && dinv[i] != 0.0) {
      const int k1 = a.rowptr[i + 1];
      for (int k = a.rowptr[i] + lane8; k < k1; k += kRowLanes) s = fma(a.K[k], u[a.col[k]], s);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (lane8 == 0 && i < n) {
      w[i] = s;
      wu = fma(s, u[i], wu);
    }
  }
  return wu;
}

__global__ void __launch_bounds__(kSolveThreads) macro_pcg_kernel(const MacroSolveArgs a) {
  cg::grid_group grid = cg::this_grid();
  __shared__ double sbuf[kSolveThreads / 32][2];
  const int n = a.n;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  double* x = a.du;
  double* r = a.work;
  double* u = r + n;
  double* w = u + n;
  double* p = w + n;
  double* s = p + n;
  double* dinv = s + n;
  double* partials = dinv + n;  // two buffers of [2 * gridDim.x], alternated between grid sums
  int parity = 0;
  auto next_partial = [&]() {
    double* buf = partials + (size_t)parity * 2 * gridDim.x;
    parity ^= 1;
    return buf;
  };
  // Jacobi diagonal, r = -f on free rows, u = M^-1 r
  double ff = 0.0, ru = 0.0;
  for (int i = tid; i < n; i += stride) {
    const bool fixed = a.fixed[i] != 0;
    double d = 1.0;
    for (int k = a.rowptr[i]; k < a.rowptr[i + 1]; ++k)
      if (a.col[k] == i) d = a.K[k];
    const double di = fixed ? 0.0 : 1.0 / d;
    const double ri = fixed ? 0.0 : -a.f[i];
    dinv[i] = di;
    x[i] = 0.0;
    r[i] = ri;
    u[i] = ri * di;
    p[i] = 0.0;
    s[i] = 0.0;
    ff = fma(ri, ri, ff);
    ru = fma(ri, ri * di, ru);
  }
  grid_sum2(ff, ru, next_partial(), sbuf, grid);  // its grid barrier also publishes u and dinv
  if (tid == 0) a.out[0] = sqrt(ff);
  double gamma = ru;
  const double stop = a.rtol * a.rtol * gamma;
  int it = 0, status = 0;
  if (gamma > 0.0) {
    double delta = spmv_rows(a, dinv, u, w, n), unused = 0.0;
    grid_sum2(delta, unused, next_partial(), sbuf, grid);
    double alpha = gamma / delta, beta = 0.0;
    if (!(delta > 0.0)) status = 2;
    while (status == 0) {
      // p = u + beta p, s = w + beta s, x += alpha p, r -= alpha s, u = M^-1 r, gamma' = r.u
      double g = 0.0;
      for (int i = tid; i < n; i += stride) {
        const double pi = fma(beta, p[i], u[i]);
        const double si = fma(beta, s[i], w[i]);
        p[i] = pi;
        s[i] = si;
        x[i] = fma(alpha, pi, x[i]);
        const double ri = fma(-alpha, si, r[i]);
        r[i] = ri;
        const double ui = ri * dinv[i];
        u[i] = ui;
        g = fma(ri, ui, g);
      }
      ++it;
      grid.sync();  // u complete before the product
      double d = spmv_rows(a, dinv, u, w, n);
      grid_sum2(g, d, next_partial(), sbuf, grid);
      if (g <= stop) break;
      if (it >= a.max_it) {
        status = 1;
        break;
      }
      beta = g / gamma;
      const double den = d - beta * g / alpha;
      if (!(den > 0.0)) {
        status = 2;
        break;
      }
      alpha = g / den;
      gamma = g;
    }
  }
  if (tid == 0) {
    a.out[1] = (double)it;
    a.out[2] = (double)status;
  }
}

// ------------------------------------------------------------------ rows resident in registers
constexpr int kResMaxThreads = 256, kResMaxRows = 128;

__device__ __forceinline__ double fp64_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// *p = max(*p, v) over the blocks that call it, for values that are not negative; NaN is above every number
__device__ __forceinline__ void raise_to(double* p, double v) {
  atomicMax(reinterpret_cast<unsigned long long*>(p), (unsigned long long)__double_as_longlong(v));
}

// {value, sequence number} as one 16-byte word: a reader sees both or neither
__device__ __forceinline__ void put(ulonglong2* p, double v, unsigned long long seq) {
  asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p),
               "l"(__double_as_longlong(v)), "l"(seq)
               : "memory");
}

// Calls take(e, value) for e = t, t + blockDim.x, ... < count with the words at word(e) once they carry seq; four
// loads are in flight at a time (one after the other their latencies add up).  False if a word has not come within
// `limit` cycles.
template <typename Word, typename Take>
__device__ __forceinline__ bool get_all(int count, unsigned long long seq, long long limit, Word word, Take take) {
  constexpr int M = 4;
  bool ok = true;
  for (int e0 = threadIdx.x; e0 < count; e0 += M * blockDim.x) {
    unsigned long long b[M], s[M];
    const long long t0 = clock64();
    for (;;) {
      bool all = true;
#pragma unroll
      for (int j = 0; j < M; ++j) {
        const int e = e0 + j * blockDim.x;
        s[j] = seq;
        if (e < count)
          asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                       : "=l"(b[j]), "=l"(s[j])
                       : "l"(word(e))
                       : "memory");
      }
#pragma unroll
      for (int j = 0; j < M; ++j) all = all && s[j] == seq;
      if (all) break;
      if (clock64() - t0 > limit) {
        ok = false;
        break;
      }
    }
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (e0 + j * blockDim.x < count) take(e0 + j * blockDim.x, __longlong_as_double((long long)b[j]));
  }
  return ok;
}

// L lanes per row, at most PER nonzeros per lane.
template <int L, int PER>
__global__ void __launch_bounds__(kResMaxThreads, 1) macro_pcg_resident_kernel(const MacroSolveArgs a) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ __align__(16) double us[];  // u of this block's rows, then of the rows around them
  __shared__ double part[2][32], total[4];      // total: alpha, beta, first sum, second sum
  __shared__ int action;                        // 0: go on, 1: converged, 2: cap, 3: breakdown, 4: gave up
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5, nb = gridDim.x;
  const int R = blockDim.x / L, lr = t / L, ll = t % L;
  const int r0 = blockIdx.x * R, i = r0 + lr;
  const bool mine = i < a.n;
  const int h0 = a.halo_ptr[blockIdx.x], nh = a.halo_ptr[blockIdx.x + 1] - h0;
  ulonglong2* pub = reinterpret_cast<ulonglong2*>(a.pub);
  // Partial sums, two alternating buffers of 2 per block: a block may publish its next sums while a slower one
  // still reads these, but the ones after that only when every block has read these (it needs their next).
  // u needs one buffer: a block publishes its next u after sums that every reader of this u contributed to.
  ulonglong2* slots = pub + a.n;  // [2][2 * nb]
  // this lane's nonzeros, the row's diagonal and right-hand side
  const bool fixed = !mine || a.fixed[i] != 0;
  constexpr int PL = (PER + 1) / 2;
  double k[PER], d = 0.0;
  uint32_t lc[PL];  // two 16-bit places each
  {
    const int k0 = mine ? a.rowptr[i] : 0, k1 = mine ? a.rowptr[i + 1] : 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int e = k0 + ll + j * L;
      const bool in = e < k1;
      const uint32_t c = in ? a.lcol[e] : 0u;
      k[j] = in ? a.K[e] : 0.0;
      lc[j / 2] = (j & 1) ? lc[j / 2] | (c << 16) : c;
      if (in && (int)c == lr) d = k[j];
      if (fixed) k[j] = 0.0;
    }
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  }
  const double di = fixed ? 0.0 : 1.0 / (d != 0.0 ? d : 1.0);
  double r = fixed ? 0.0 : -a.f[i], u = r * di, x = 0.0, p = 0.0, s = 0.0, w = 0.0;
  if (mine && ll == 0) pub[i] = make_ulonglong2(0ull, 0ull);
  if (t < 4) slots[(t >> 1) * 2 * nb + 2 * blockIdx.x + (t & 1)] = make_ulonglong2(0ull, 0ull);
  if (t == 0) action = 0;
  if (blockIdx.x == 0 && t < 3) a.out[t] = 0.0;
  grid.sync();  // every word carries sequence number 0
  unsigned long long useq = 0, sseq = 0;
  bool lost = false;

  auto publish = [&]() {
    ++useq;
    if (ll == 0) {
      us[lr] = u;
      if (mine && nb > 1) put(pub + i, u, useq);
    }
  };
  auto product = [&]() {  // the surrounding rows' u, then w = K u (the same in all lanes of a row)
    lost |= !get_all(nh, useq, a.wait_limit, [&](int h) { return pub + a.halo[h0 + h]; }, [&](int h, double v) { us[R + h] = v; });
    __syncthreads();
    w = lost ? fp64_nan() : 0.0;  // a block that gave up spoils the sums it still publishes
#pragma unroll
    for (int j = 0; j < PER; ++j) w = fma(k[j], us[(j & 1) ? lc[j / 2] >> 16 : lc[j / 2] & 0xffffu], w);
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  };
  // Sums over the grid of the values v of lanes ll == 0 (first) and ll == 1 (second), the others zero, into
  // total[2], total[3] of warp 0; `decide` runs in warp 0 with them before the closing barrier.
  auto reduce = [&](double v, auto decide) {
#pragma unroll
    for (int o = L; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane < 2) part[0][2 * warp + lane] = v;
    __syncthreads();
    ++sseq;
    ulonglong2* slot = slots + (sseq & 1) * 2 * nb;
    double acc = 0.0;
    if (warp == 0) {
      acc = lane < 2 * nw ? part[0][lane] : 0.0;
      for (int o = 2; o < 2 * nw; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane < 2 && nb > 1) put(slot + 2 * blockIdx.x + lane, acc, sseq);
    }
    if (nb > 1) {
      acc = 0.0;
      lost |= !get_all(2 * nb, sseq, a.wait_limit, [&](int e) { return slot + e; }, [&](int, double q) { acc += q; });
#pragma unroll
      for (int o = 2; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane < 2) part[1][2 * warp + lane] = acc;
      if (__syncthreads_or(lost) && t == 0) action = 4;
      if (warp == 0) {
        acc = lane < 2 * nw ? part[1][lane] : 0.0;
        for (int o = 2; o < 2 * nw; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      }
    }
    if (warp == 0) {
      const double q0 = __shfl_sync(0xffffffffu, acc, 0), q1 = __shfl_sync(0xffffffffu, acc, 1);
      __syncwarp();
      if (lane == 0 && action == 0) decide(q0, q1);
    }
    __syncthreads();
  };
  // scalars of the iteration, thread 0 only
  double gamma = 0.0, rgamma = 0.0, den = 0.0, stop = 0.0;
  int it = 0;
  reduce(ll < 2 ? r * (ll ? u : r) : 0.0, [&](double ff, double ru) {
    if (blockIdx.x == 0) raise_to(a.out, sqrt(ff));
    gamma = ru;
    stop = a.rtol * a.rtol * gamma;
    if (!(gamma > 0.0)) action = 1;
  });
  if (action == 0) {
    publish();
    product();
    reduce(ll == 1 ? w * u : 0.0, [&](double, double delta) {
      if (!(delta > 0.0)) {
        action = 3;
        return;
      }
      den = delta;
      total[0] = div_d(gamma, delta);
      total[1] = 0.0;
    });
  }
  while (action == 0) {
    const double alpha = total[0], beta = total[1], u_old = u;
    s = fma(beta, s, w);
    r = fma(-alpha, s, r);
    u = r * di;
    publish();
    p = fma(beta, p, u_old);  // off the path of u: while it travels
    x = fma(alpha, p, x);
    if (t == 0) rgamma = recip_d(gamma);
    product();
    reduce(ll < 2 ? u * (ll ? w : r) : 0.0, [&](double g, double dl) {
      ++it;
      if (g <= stop) {
        action = 1;
        return;
      }
      if (it >= a.max_it) {
        action = 2;
        return;
      }
      // infinite: gamma is subnormal (g / gamma may be an ordinary number)
      const double b = __double2hiint(rgamma) == 0x7ff00000 ? g / gamma : g * rgamma;
      den = fma(-b * b, den, dl);  // d - beta g / alpha, with alpha = gamma / (the last) den
      if (!(den > 0.0)) {
        action = 3;
        return;
      }
      total[0] = div_d(g, den);
      total[1] = b;
      gamma = g;
    });
  }
  if (mine && ll == 0) a.du[i] = x;
  if (t == 0) {
    if (blockIdx.x == 0) {
      a.out[1] = (double)it;
      raise_to(a.out + 2, (double)(action - 1));  // 0 converged, 1 cap, 2 breakdown
    }
    // A block that gave up makes this the outcome, whatever the others made of its words; the norm may be one that
    // block 0 never formed.
    if (action == 4) {
      raise_to(a.out, fp64_nan());
      raise_to(a.out + 2, 3.0);
    }
  }
}

}  // namespace

size_t macro_solve_work_doubles(int n, int blocks) { return 6 * (size_t)n + 4 * (size_t)blocks; }

// One block per 32 rows (one pass of the product), at most one per SM.
int macro_solve_blocks(int num_sms, long long n_rows) {
  long long b = (n_rows + kRowsPerBlock - 1) / kRowsPerBlock;
  if (b < 1) b = 1;
  return (int)(b < num_sms ? b : num_sms);
}

// Lanes per row, rows and blocks of the resident kernel for a mesh of n rows (0 lanes: not resident).  An FP64
// warp instruction takes 64 cycles of an SM sub-partition however many of its lanes are active, so an iteration
// counts (instructions of a warp) x (warps per sub-partition): with L lanes a row, 8 + nnz / L + ... instructions
// and R L / 128 warps.  R <= 16 rows: 8 lanes fill the four sub-partitions with one warp each; up to 32 rows 4
// lanes, above that 2.  A mesh of up to 128 rows (3D, with 81 nonzeros a row: 64) is solved by one block, which
// exchanges nothing.
MacroResident macro_resident_plan(int dim, int n, int num_sms) {
  MacroResident m{};
  const int rows = n <= (dim == 2 ? 128 : 64) ? n : std::max(16, (n + num_sms - 1) / num_sms);
  if (rows > kResMaxRows) return m;
  m.lanes = rows <= 16 ? 8 : rows <= 32 ? 4 : 2;
  const int per_warp = 32 / m.lanes;
  m.rows = (rows + per_warp - 1) / per_warp * per_warp;
  m.blocks = (n + m.rows - 1) / m.rows;
  return m;
}

// Per block the distinct columns outside its rows (in the order met), and per nonzero its column's place among the
// block's rows and those.  The d rows of a node have the same columns.  False if a block needs more places than
// the shared memory for u holds.
bool macro_resident_columns(MacroResident& m, int dim, int n, const std::vector<int32_t>& rowptr,
                            const std::vector<int32_t>& col, std::vector<int32_t>& halo_ptr, std::vector<int32_t>& halo,
                            std::vector<uint16_t>& lcol) {
  halo_ptr.assign(1, 0);
  halo.clear();
  lcol.resize(col.size());
  std::vector<int32_t> block(n, -1);  // the block that last met this column
  std::vector<uint16_t> place(n);
  int most = 0;
  for (int b = 0; b < m.blocks; ++b) {
    const int r0 = b * m.rows, r1 = std::min(n, r0 + m.rows);
    int places = m.rows;
    for (int i = r0; i < r1; ++i) {
      block[i] = b;
      place[i] = (uint16_t)(i - r0);
    }
    for (int i = r0; i < r1; ++i) {
      if (i > r0 && i % dim != 0) {
        std::copy(lcol.begin() + rowptr[i - 1], lcol.begin() + rowptr[i], lcol.begin() + rowptr[i]);
        continue;
      }
      for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        const int32_t c = col[e];
        if (block[c] != b) {
          block[c] = b;
          place[c] = (uint16_t)places++;
          halo.push_back(c);
        }
        lcol[e] = place[c];
      }
    }
    if (places > 4096) return false;
    most = std::max(most, places);
    halo_ptr.push_back((int32_t)halo.size());
  }
  m.smem = sizeof(double) * most;
  return true;
}

cudaError_t macro_solve_resident_launch(const MacroSolveArgs& a, int dim, const MacroResident& m, cudaStream_t stream) {
  void* args[] = {(void*)&a};
  const void* kernel;
  if (dim == 2)
    kernel = m.lanes == 8   ? (const void*)macro_pcg_resident_kernel<8, 3>
             : m.lanes == 4 ? (const void*)macro_pcg_resident_kernel<4, 5>
                            : (const void*)macro_pcg_resident_kernel<2, 9>;
  else
    kernel = m.lanes == 8   ? (const void*)macro_pcg_resident_kernel<8, 11>
             : m.lanes == 4 ? (const void*)macro_pcg_resident_kernel<4, 21>
                            : (const void*)macro_pcg_resident_kernel<2, 41>;
  return cudaLaunchCooperativeKernel(kernel, dim3(m.blocks), dim3(m.rows * m.lanes), args, m.smem, stream);
}

cudaError_t macro_solve_launch(const MacroSolveArgs& a, int blocks, cudaStream_t stream) {
  void* args[] = {(void*)&a};
  return cudaLaunchCooperativeKernel((void*)macro_pcg_kernel, dim3(blocks), dim3(kSolveThreads), args, 0, stream);
}

}  // namespace fehmm
