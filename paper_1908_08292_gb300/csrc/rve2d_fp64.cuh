// The 2D RVE solve in FP64 mode: the method of rve2d.cuh (same levels, same PCG, same recovery) in a thread layout
// of its own.
//
// On a GB300 an FP64 warp instruction occupies one of an SM's four sub-partitions for 64 cycles, however many of
// its lanes are active, so a solve's time is (FP64 instructions of a warp) x (warps per sub-partition) x 64 cycles
// and everything else hides behind it.  Hence:
//  * one thread per degree of freedom (node, component), and two per element (one line of Gauss points each, which
//    exchange partial sums): the same work in fewer instructions per warp, spread over all four sub-partitions;
//  * a row of the stencil (18 values) stays in the thread's registers up to 22 x 22, beyond that in the block's
//    scratch (32 x 32 has four dofs per thread);
//  * the step scalars are formed by one thread (division and comparison are FP64 instructions too) with a refined
//    reciprocal (a division is about nine), and both inner products go through one shuffle tree;
//  * the part of the neo-Hookean tangent that is the same matrix for every element is added once, scaled by mu.
// Measured on a GB300, one pass from a committed state, against the node-pair layout of rve2d.cuh with TA = double:
// at 512 threads (first figure) and at one thread per node pair (second).  64 RVEs of 8 x 8: 3.18, 2.45 -> 0.71 ms;
// 100 of 32 x 32: 18.3, 18.3 -> 12.4 ms; 150 of 16 x 16 through the no-allocation entry, block-Jacobi: 16.3, 8.6 -> 5.2 ms
// (3.3 with multigrid).
#pragma once
#include "rve2d.cuh"

namespace fehmm {

namespace {

constexpr int kThreadsD2 = 512;
// Threads: one per degree of freedom, at least four warps, at most 512 (then DPT dofs per thread).
__host__ __device__ constexpr int threads_d2(int nn) {
  const int t = (2 * nn + 31) / 32 * 32;
  return t < 128 ? 128 : t > kThreadsD2 ? kThreadsD2 : t;
}
__host__ __device__ constexpr int dofs_per_thread_d2(int nn) { return nn <= 256 ? 1 : nn <= 512 ? 2 : 4; }

// Byte offsets in shared memory.  The multigrid's fast region follows where it fits (n <= 24).
struct OffsetsD2 {
  size_t w, p, x, stage, red, lame, misc, fast, total;
  bool fast_in_smem;
};
__host__ __device__ constexpr OffsetsD2 offsets_d2(int NN, bool mg) {
  OffsetsD2 o{};
  size_t off = 0;
  const auto take = [&off](size_t bytes) {
    const size_t at = off;
    off += (bytes + 15) & ~size_t(15);
    return at;
  };
  o.w = take(sizeof(double) * 2 * NN);
  o.p = take(sizeof(double) * 4 * NN);       // two alternating exchange buffers
  o.x = take(sizeof(double) * 2 * NN);
  o.stage = take(sizeof(double) * 16 * NN);  // element forces [8][NN]; condensation X [4][2 NN], L [4][2 NN]
  o.red = take(sizeof(double) * (kBlockSumDoubles + 40));
  o.lame = take(sizeof(double) * (2 * kMaxPhase + kResidualTable));
  o.misc = take(sizeof(double) * 16);
  int n = 2;
  while (n * n < NN) ++n;
  const size_t fast = sizeof(double) * (size_t)(mg ? mg_fast_elems(n) : 0);
  o.fast_in_smem = off + fast <= 200 * 1024;
  o.fast = o.fast_in_smem ? take(fast) : 0;
  o.total = off;
  return o;
}
__host__ __device__ constexpr size_t most_smem_d2(bool mg) {  // over the grids
  size_t most = 0;
  for (int n = 2; n <= 32; n += 2) most = offsets_d2(n * n, mg).total > most ? offsets_d2(n * n, mg).total : most;
  return most;
}
// Block scratch (doubles): staged element tangents [36][NN], the stencil [18][2 NN] (grids that do not hold it in
// registers), then the multigrid: fast region (where not in shared memory) and slow region.  The slow region takes the
// stencil's place where that is in registers: it has a third of its size.
__host__ __device__ constexpr long long scratch_d2(int NN, bool mg) {
  int n = 2;
  while (n * n < NN) ++n;
  return 72LL * NN + (mg ? mg_fast_elems(n) + mg_slow_elems(n) : 0);
}

__device__ __forceinline__ double other(double v) { return __shfl_xor_sync(0xffffffffu, v, 1); }  // the pair's lane

template <int DPT, int LAW>
struct D2 {
  int n, NN, ND, T, bc;
  const uint8_t* phase;
  // shared memory
  double *w, *p, *x, *stage, *red, *lame, *restab, *misc;
  // block scratch
  double *ke;     // staged element tangents [36][NN]
  double *st;     // stencil [18][2 NN] (DPT = 4)
  MgCtx<double> mg;
  // this thread's degrees of freedom
  bool act[DPT], pin[DPT];
  int dof[DPT], col[DPT][3], row[DPT][3];
};

template <int DPT>
constexpr bool kRowInRegs = DPT <= 2;
template <int DPT>
struct Row {
  double k[kRowInRegs<DPT> ? DPT : 1][18];
};

// sum of two values over the block in one shuffle tree; valid in warp 0 before the caller's barrier
__device__ __forceinline__ void dot2(double g, double d, double* buf, double& sg, double& sd) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double a = lane < 16 ? g : d;
  const double b = lane < 16 ? d : g;
  a += __shfl_xor_sync(0xffffffffu, b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((lane & 15) == 0) buf[(lane & 16) + warp] = a;
  __syncthreads();
  if (warp == 0) {
    double v = (lane & 15) < nw ? buf[lane] : 0.0;
    for (int o = 1; o < nw; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    sg = __shfl_sync(0xffffffffu, v, 0);
    sd = __shfl_sync(0xffffffffu, v, 16);
  }
}

// ------------------------------------------------------------------ element work, two lanes per element
// Lane pair (2k, 2k + 1): element e, Gauss line t = g01(lane & 1) of two points each.
struct Elem2 {
  bool in;
  int e, nd[4];
};
__device__ __forceinline__ Elem2 elem2(int k, int n, int NN) {
  Elem2 q;
  q.in = k < NN;
  q.e = q.in ? k : 0;
  const int i = q.e % n, j = q.e / n, ip = wrap_inc(i, n), jp = wrap_inc(j, n);
  q.nd[0] = q.e;
  q.nd[1] = ip + n * j;
  q.nd[2] = ip + n * jp;
  q.nd[3] = i + n * jp;
  return q;
}

// Element tangents (36 upper-triangle entries) into ke[tri][e]; each lane adds its line's two points, then the
// lanes of a pair exchange halves.
template <int DPT, int LAW>
__device__ __forceinline__ void element_tangents_d2(const D2<DPT, LAW>& s) {
  const int half = threadIdx.x & 1;
  const double ih = (double)s.n, t = gauss01(half);
  const double2* w = reinterpret_cast<const double2*>(s.w);
  for (int k0 = 0; k0 < s.NN; k0 += s.T / 2) {
    const Elem2 q = elem2(k0 + (threadIdx.x >> 1), s.n, s.NN);
    const int ph = s.phase[q.e];
    const double lam = s.lame[2 * ph], mu = s.lame[2 * ph + 1];
    const double2 w0 = w[q.nd[0]], w1 = w[q.nd[1]], w2 = w[q.nd[2]], w3 = w[q.nd[3]];
    const double F00 = s.misc[0] + ih * ((w1.x - w0.x) + t * ((w2.x - w3.x) - (w1.x - w0.x)));
    const double F10 = s.misc[2] + ih * ((w1.y - w0.y) + t * ((w2.y - w3.y) - (w1.y - w0.y)));
    double Ke[36];
#pragma unroll
    for (int k = 0; k < 36; ++k) Ke[k] = 0.0;
    // natural shape gradients; the factors 1 / h cancel against the area: 1/4 per point
    const double gx[4] = {-(1 - t), 1 - t, t, -t};
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const double sg = gauss01(g);
      const double F01 = s.misc[1] + ih * ((w3.x - w0.x) + sg * ((w2.x - w1.x) - (w3.x - w0.x)));
      const double F11 = s.misc[3] + ih * ((w3.y - w0.y) + sg * ((w2.y - w1.y) - (w3.y - w0.y)));
      const double gy[4] = {-(1 - sg), -sg, sg, 1 - sg};
      double vx[4], vy[4];
      if constexpr (LAW == kLawNH) {
        const double J = F00 * F11 - F01 * F10, iJ = recip_d(J), J2 = J * J;
        const double hb = 0.5 * lam * (J2 - 1.0) - mu, gm = lam * J2;
        const double i00 = F11 * iJ, i01 = -F10 * iJ, i10 = -F01 * iJ, i11 = F00 * iJ;
        const double cg = 0.25 * gm, ch = 0.25 * hb, cd = cg - ch;
        double gvx[4], gvy[4], hvx[4], hvy[4], dvx[4], dvy[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          vx[a] = i00 * gx[a] + i01 * gy[a];
          vy[a] = i10 * gx[a] + i11 * gy[a];
          gvx[a] = cg * vx[a];
          gvy[a] = cg * vy[a];
          hvx[a] = -ch * vx[a];
          hvy[a] = -ch * vy[a];
          dvx[a] = cd * vx[a];
          dvy[a] = cd * vy[a];
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int c = r; c < 8; ++c) {
            const int a = r >> 1, ii = r & 1, b = c >> 1, kk = c & 1;
            double& K = Ke[tri8(r, c)];
            if (ii == kk) {  // (cg - ch) v_a,i v_b,i
              K = fma(ii ? dvy[a] : dvx[a], ii ? vy[b] : vx[b], K);
            } else {  // cg v_a,i v_b,k - ch v_b,i v_a,k
              K = fma(ii ? gvy[a] : gvx[a], kk ? vy[b] : vx[b], K);
              K = fma(kk ? hvy[a] : hvx[a], ii ? vy[b] : vx[b], K);
            }
          }
      } else {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          vx[a] = F00 * gx[a] + F01 * gy[a];
          vy[a] = F10 * gx[a] + F11 * gy[a];
        }
        const double c00 = F00 * F00 + F10 * F10, c01 = F00 * F01 + F10 * F11, c11 = F01 * F01 + F11 * F11;
        const double trE = 0.5 * (c00 + c11) - 1.0;
        const double S00 = 0.25 * (lam * trE + mu * (c00 - 1.0)), S11 = 0.25 * (lam * trE + mu * (c11 - 1.0)), S01 = 0.25 * mu * c01;
        const double b00 = F00 * F00 + F01 * F01, b01 = F00 * F10 + F01 * F11, b11 = F10 * F10 + F11 * F11;
        const double cl = 0.25 * lam, cm = 0.25 * mu;
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int c = r; c < 8; ++c) {
            const int a = r >> 1, ii = r & 1, b = c >> 1, kk = c & 1;
            const double va_i = ii ? vy[a] : vx[a], va_k = kk ? vy[a] : vx[a];
            const double vb_i = ii ? vy[b] : vx[b], vb_k = kk ? vy[b] : vx[b];
            const double gg = gx[a] * gx[b] + gy[a] * gy[b];
            const double bik = (ii == kk) ? (ii ? b11 : b00) : b01;
            double val = cl * va_i * vb_k + cm * (gg * bik + vb_i * va_k);
            if (ii == kk) val += gx[a] * (S00 * gx[b] + S01 * gy[b]) + gy[a] * (S01 * gx[b] + S11 * gy[b]);
            Ke[tri8(r, c)] += val;
          }
      }
    }
    // lane 0 keeps entries 0 .. 17, lane 1 the rest
    double mine[18];
#pragma unroll
    for (int k = 0; k < 18; ++k) mine[k] = (half ? Ke[18 + k] : Ke[k]) + other(half ? Ke[k] : Ke[18 + k]);
    if constexpr (LAW == kLawNH) {  // + mu sum_points g_a . g_b / 4, the same matrix for every element
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = r; c < 8; ++c) {
          if ((r & 1) != (c & 1)) continue;
          constexpr double third = 1.0 / 3.0, sixth = 1.0 / 6.0;
          const int a = r >> 1, b = c >> 1;
          // Q1 Laplacian on a square: 2/3 on the diagonal, -1/6 along an edge, -1/3 across
          const double L = a == b ? 2.0 * third : ((a ^ b) == 2 ? -third : -sixth);
          const int tri = tri8(r, c);
          if (half == (tri >= 18)) mine[tri % 18] = fma(mu, L, mine[tri % 18]);
        }
    }
    if (q.in) {
#pragma unroll
      for (int k = 0; k < 18; ++k) s.ke[(size_t)(18 * half + k) * s.NN + q.e] = mine[k];
    }
  }
}

// The stencil rows of this thread's dofs from the staged element tangents, the inverted nodal block's rows, and
// (withL) minus the rows of the operator applied to the unit gradients, Lb[c][dof].
template <int DPT, int LAW>
__device__ __forceinline__ void gather_rows_d2(const D2<DPT, LAW>& s, Row<DPT>& R, double (&Mi)[DPT][2], bool withL, double* Lb) {
  const int n = s.n, NN = s.NN, c = threadIdx.x & 1;
  const double h = 1.0 / n;
#pragma unroll
  for (int q = 0; q < DPT; ++q) {
    double K[18], L[4] = {0.0, 0.0, 0.0, 0.0};
    const int v = s.dof[q] >> 1, i = v % n, j = v / n;
    const int ei[2] = {i, wrap_dec(i, n)}, ej[2] = {j, wrap_dec(j, n)};
    bool seen[9] = {false, false, false, false, false, false, false, false, false};
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int slot = ei[offx(l)] + n * ej[offy(l)];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int nb = (offy(m) - offy(l) + 1) * 3 + (offx(m) - offx(l) + 1);
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          const double a = s.ke[(size_t)tri8(2 * l, 2 * m + kk) * NN + slot], b = s.ke[(size_t)tri8(2 * l + 1, 2 * m + kk) * NN + slot];
          const double e = c ? b : a;
          K[2 * nb + kk] = seen[nb] ? K[2 * nb + kk] + e : e;
          if (withL) {
            if (offx(m)) L[2 * kk] = fma(e, h, L[2 * kk]);
            if (offy(m)) L[2 * kk + 1] = fma(e, h, L[2 * kk + 1]);
          }
        }
        seen[nb] = true;
      }
    }
    const double k0 = K[8], k1 = K[9], o0 = other(k0), o1 = other(k1);  // rows of the nodal block
    const double det = c ? o0 * k1 - o1 * k0 : k0 * o1 - k1 * o0;
    const double id = !s.act[q] || s.pin[q] ? 0.0 : 1.0 / det;
    // inverse [[d, -b], [-c, a]] / det of [[a, b], [c, d]]: row 0 from row 1's second entry, ...
    Mi[q][0] = c ? -k0 * id : o1 * id;
    Mi[q][1] = c ? o0 * id : -k1 * id;
    if constexpr (kRowInRegs<DPT>) {
#pragma unroll
      for (int k = 0; k < 18; ++k) R.k[q][k] = s.act[q] ? K[k] : 0.0;
    } else {
      if (s.act[q])
#pragma unroll
        for (int k = 0; k < 18; ++k) s.st[(size_t)k * s.ND + s.dof[q]] = K[k];
    }
    if (withL && s.act[q])
#pragma unroll
      for (int k = 0; k < 4; ++k) Lb[(size_t)k * s.ND + s.dof[q]] = s.pin[q] ? 0.0 : -L[k];
  }
}

// ------------------------------------------------------------------ multigrid, one thread per dof
__device__ __forceinline__ double2 block_row(const Block2<double>& b, int c) {
  return reinterpret_cast<const double2*>(&b)[c];
}

// (K z)[d] on a coarse level (zero at a pinned node)
__device__ __forceinline__ double mg_apply_d2(const MgLevel<double>& L, const double2* z, int d) {
  const int n = L.n, v = d >> 1, c = d & 1, i = v % n, j = v / n;
  const int cols[3] = {wrap_dec(i, n), i, wrap_inc(i, n)};
  const int rows[3] = {wrap_dec(j, n) * n, j * n, wrap_inc(j, n) * n};
  double y = 0.0;
#pragma unroll
  for (int nb = 0; nb < 9; ++nb) {
    const double2 zn = z[rows[nb / 3] + cols[nb % 3]], k = block_row(L.st[nb * L.NN + v], c);
    y = fma(k.x, zn.x, y);
    y = fma(k.y, zn.y, y);
  }
  return pinned2(i, j, L.bc) ? 0.0 : y;
}

// omega M^-1 applied to the nodal pair this lane and its neighbour hold
__device__ __forceinline__ double smooth_d2(const Block2<double>& m, int c, double r, double omega) {
  const double2 k = block_row(m, c);
  const double o = other(r);
  return omega * (k.x * (c ? o : r) + k.y * (c ? r : o));
}

// restriction of t (dofs of grid nf) to dof d of the grid half as fine
__device__ __forceinline__ double restrict_d2(const double* t, int nf, int d, int bc) {
  const int nc = nf >> 1, v = d >> 1, c = d & 1, I = v % nc, J = v / nc, ix = 2 * I, jy = 2 * J;
  const int cols[3] = {wrap_dec(ix, nf), ix, ix + 1};
  const int rows[3] = {wrap_dec(jy, nf) * nf, jy * nf, (jy + 1) * nf};
  auto at = [&](int y, int x) { return t[2 * (rows[y] + cols[x]) + c]; };
  const double corners = (at(0, 0) + at(0, 2)) + (at(2, 0) + at(2, 2)), edges = (at(0, 1) + at(2, 1)) + (at(1, 0) + at(1, 2));
  return pinned2(I, J, bc) ? 0.0 : fma(0.25, corners, fma(0.5, edges, at(1, 1)));
}

// prolongation of zc (grid nf / 2) to component c of node (i, j): the mean of the four coarse nodes around it
__device__ __forceinline__ double prolong_d2(const double* zc, int nf, int i, int j, int c) {
  const int nc = nf >> 1, i0 = i >> 1, j0 = j >> 1;
  const int i1 = (i & 1) ? wrap_inc(i0, nc) : i0, j1 = (j & 1) ? wrap_inc(j0, nc) : j0;
  auto at = [&](int x, int y) { return zc[2 * (x + nc * y) + c]; };
  return 0.25 * ((at(i0, j0) + at(i1, j0)) + (at(i0, j1) + at(i1, j1)));
}

// restricted residual of level l and, on a smoothing level, its pre-smoothed correction
__device__ __forceinline__ void restrict_smooth_d2(const MgCtx<double>& mg, int l, const double* tf, int nf) {
  const MgLevel<double> c = mg.level(l);
  for (int d0 = 0; d0 < 2 * c.NN; d0 += blockDim.x) {  // whole warps: smooth_d2 exchanges within a pair
    const int d = d0 + threadIdx.x;
    const bool in = d < 2 * c.NN;
    const double r = in ? restrict_d2(tf, nf, d, mg.bc) : 0.0;
    if (in) reinterpret_cast<double*>(c.r)[d] = r;
    if (l < mg.levels) {
      const double z = smooth_d2(c.mi[in ? d >> 1 : 0], d & 1, r, mg.omega);
      if (in) reinterpret_cast<double*>(c.z)[d] = z;
    }
  }
}

__device__ void coarse_cycle_d2(const MgCtx<double>& mg) {
  const int tid = threadIdx.x, T = blockDim.x;
  for (int l = 1; l < mg.levels; ++l) {
    const MgLevel<double> v = mg.level(l);
    const double* r = reinterpret_cast<const double*>(v.r);
    double* t = reinterpret_cast<double*>(v.t);
    for (int d = tid; d < 2 * v.NN; d += T) t[d] = r[d] - mg_apply_d2(v, v.z, d);
    __syncthreads();
    restrict_smooth_d2(mg, l + 1, t, v.n);
    __syncthreads();
  }
  {  // coarsest: z = A^-1 r, four lanes per row
    const MgLevel<double> c = mg.level(mg.levels);
    const double z = coarsest_row<double>(mg.coarsest_inverse(), reinterpret_cast<const double*>(c.r), 2 * c.NN);
    const int row = tid >> 2;
    if (row < 2 * c.NN && (tid & 3) == 0) reinterpret_cast<double*>(c.z)[row] = pinned2((row >> 1) % c.n, (row >> 1) / c.n, c.bc) ? 0.0 : z;
    __syncthreads();
  }
  for (int l = mg.levels - 1; l >= 1; --l) {
    const MgLevel<double> v = mg.level(l);
    const double* zc = reinterpret_cast<const double*>(mg_result<double>(mg, l + 1));
    double* z = reinterpret_cast<double*>(v.z);
    for (int d = tid; d < 2 * v.NN; d += T) z[d] += prolong_d2(zc, v.n, (d >> 1) % v.n, (d >> 1) / v.n, d & 1);
    __syncthreads();
    for (int d0 = 0; d0 < 2 * v.NN; d0 += T) {
      const int d = d0 + tid;
      const bool in = d < 2 * v.NN;
      const double t = in ? reinterpret_cast<const double*>(v.r)[d] - mg_apply_d2(v, v.z, d) : 0.0;
      const double dz = smooth_d2(v.mi[in ? d >> 1 : 0], d & 1, t, mg.omega);
      if (in) reinterpret_cast<double*>(v.t)[d] = z[d] + dz;
    }
    __syncthreads();
  }
}

// Galerkin element matrices of the coarse grid nf / 2, one thread per column: K_E = sum over the four fine elements
// of W^T K_e W (see mg_coarse_element).
__device__ __forceinline__ void coarse_elements_d2(const double* kf, int nf, double* kc) {
  const int nc = nf >> 1, nnc = nc * nc, NNf = nf * nf;
  for (int task = threadIdx.x; task < 8 * nnc; task += blockDim.x) {
    const int E = task >> 3, col = task & 7, I = E % nc, J = E / nc;
    double acc[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = 0.0;
#pragma unroll 1
    for (int ab = 0; ab < 4; ++ab) {
      const int a = ab & 1, b = ab >> 1, e = (2 * I + a) + nf * (2 * J + b);
      auto weight = [&](int k, int c) {  // of coarse corner c at fine corner k
        const double x2 = 0.5 * (a + offx(k)), y2 = 0.5 * (b + offy(k));
        return (offx(c) ? x2 : 1.0 - x2) * (offy(c) ? y2 : 1.0 - y2);
      };
      double wc[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) wc[m] = 0.0;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c == (col >> 1))
#pragma unroll
          for (int m = 0; m < 4; ++m) wc[m] = weight(m, c);
      double t[8];  // column col of K_e W
#pragma unroll
      for (int row = 0; row < 8; ++row) {
        double v = 0.0;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const double k0 = kf[(size_t)tri8(row, 2 * m) * NNf + e], k1 = kf[(size_t)tri8(row, 2 * m + 1) * NNf + e];
          v = fma((col & 1) ? k1 : k0, wc[m], v);
        }
        t[row] = v;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        double wk[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) wk[k] = weight(k, c);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[2 * c + i] = fma(wk[k], t[2 * k + i], acc[2 * c + i]);
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r <= col) {
        const int tri = r * 8 - (r * (r - 1)) / 2 + (col - r);
        kc[(size_t)tri * nnc + E] = acc[r];
      }
  }
}

// All coarse levels below the staged element tangents.  Ends with a barrier.
__device__ void mg_build_d2(const MgCtx<double>& mg, const double* ke) {
  const int tid = threadIdx.x, T = blockDim.x;
  const double* kf = ke;
  int nf = mg.n;
  for (int l = 1; l <= mg.levels; ++l) {
    const MgLevel<double> c = mg.level(l);
    coarse_elements_d2(kf, nf, c.ke);
    __syncthreads();
    kf = c.ke;
    nf = c.n;
  }
  for (int l = 1; l < mg.levels; ++l) {  // stencils and inverted blocks of the smoothing levels, a block per thread
    const MgLevel<double> v = mg.level(l);
    for (int task = tid; task < 9 * v.NN; task += T) {
      const int nb = task / v.NN, node = task % v.NN, i = node % v.n, j = node / v.n;
      double blk[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if (q == nb) mg_stencil_block<double>(v.ke, v.n, i, j, q, blk);
      v.st[nb * v.NN + node] = {blk[0], blk[1], blk[2], blk[3]};
      if (nb == 4) {
        double m[4];
        invert_block<double>(blk, pinned2(i, j, v.bc), m);
        v.mi[node] = {m[0], m[1], m[2], m[3]};
      }
    }
  }
  mg_invert_coarsest<double>(mg);
}

// ------------------------------------------------------------------ PCG
// As pcg_pair (Chronopoulos-Gear, truncated on negative curvature, warm start relative to the right-hand side's
// reference); b and x0 / x per dof.  The result x goes to xs (x0 is read from there).
template <int DPT, int LAW, bool kMG>
__device__ int pcg_d2(const D2<DPT, LAW>& s, const Row<DPT>& R, const double (&Mi)[DPT][2], const double (&b)[DPT], double* xs,
                      double rtol, int max_it, int* status, bool truncate, bool warm) {
  const int c = threadIdx.x & 1;
  double r[DPT], u[DPT], w[DPT], p[DPT], sv[DPT], x[DPT];
#pragma unroll
  for (int q = 0; q < DPT; ++q) {
    r[q] = s.act[q] ? b[q] : 0.0;
    x[q] = 0.0;
  }
  int pb = 0;
  auto exchange_apply = [&]() {  // w = K u
    double* buf = s.p + pb * s.ND;
    pb ^= 1;
#pragma unroll
    for (int q = 0; q < DPT; ++q)
      if (s.act[q]) buf[s.dof[q]] = u[q];
    __syncthreads();
    const double2* z = reinterpret_cast<const double2*>(buf);
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
      double y = 0.0;
#pragma unroll
      for (int nb = 0; nb < 9; ++nb) {
        const double2 zn = z[s.row[q][nb / 3] + s.col[q][nb % 3]];
        if constexpr (kRowInRegs<DPT>) {
          y = fma(R.k[q][2 * nb], zn.x, y);
          y = fma(R.k[q][2 * nb + 1], zn.y, y);
        } else {
          y = fma(s.st[(size_t)(2 * nb) * s.ND + s.dof[q]], zn.x, y);
          y = fma(s.st[(size_t)(2 * nb + 1) * s.ND + s.dof[q]], zn.y, y);
        }
      }
      w[q] = s.act[q] && !s.pin[q] ? y : 0.0;
    }
  };
  auto jacobi = [&](int q, double v) {  // row of M^-1 applied to the node's pair
    const double o = other(v);
    return fma(Mi[q][0], c ? o : v, Mi[q][1] * (c ? v : o));
  };
  auto precond = [&]() {
    if (!kMG || !s.mg.levels) {
#pragma unroll
      for (int q = 0; q < DPT; ++q) u[q] = jacobi(q, r[q]);
      return;
    }
    const double om = s.mg.omega;
#pragma unroll
    for (int q = 0; q < DPT; ++q) u[q] = om * jacobi(q, r[q]);
    exchange_apply();
    double* ft = reinterpret_cast<double*>(s.mg.fine_t());
#pragma unroll
    for (int q = 0; q < DPT; ++q)
      if (s.act[q]) ft[s.dof[q]] = r[q] - w[q];
    __syncthreads();
    restrict_smooth_d2(s.mg, 1, ft, s.n);
    __syncthreads();
    coarse_cycle_d2(s.mg);
    const double* zc = reinterpret_cast<const double*>(mg_result<double>(s.mg, 1));
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
      const double z = prolong_d2(zc, s.n, s.col[q][1], s.row[q][1] / s.n, c);
      if (s.act[q]) u[q] += z;
    }
    exchange_apply();
#pragma unroll
    for (int q = 0; q < DPT; ++q) u[q] = fma(om, jacobi(q, r[q] - w[q]), u[q]);
  };
  double* red = s.red + kBlockSumDoubles;
  double* out = red + 32;  // alpha, beta; [2] the decision
  auto dots = [&](bool both, double& g, double& d) {  // valid in warp 0
    double a = 0.0, e = 0.0;
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
      a = fma(r[q], u[q], a);
      if (both) e = fma(w[q], u[q], e);
    }
    dot2(a, e, red, g, d);
  };
  // The scalars live in thread 0; every thread reads the step and the decision (0 go on, 1 converged, 2 cap,
  // 3 breakdown, 4 negative curvature: truncate, 5 negative curvature at the first direction).
  double gref = -1.0, stop = 0.0, gamma = 0.0, den = 0.0;
  int it = 0, phase = warm ? 0 : 1;
  for (;;) {
    precond();
    if (phase == 0) {  // u = M^-1 b: the stopping reference, then r = b - K x0
      double g = 0.0, d = 0.0;
      dots(false, g, d);
      gref = g;
#pragma unroll
      for (int q = 0; q < DPT; ++q) u[q] = x[q] = s.act[q] ? xs[s.dof[q]] : 0.0;
      exchange_apply();
#pragma unroll
      for (int q = 0; q < DPT; ++q) r[q] -= w[q];
      it = 1;
      phase = 1;
      continue;
    }
    exchange_apply();
    double g = 0.0, d = 0.0;
    dots(true, g, d);
    if (threadIdx.x == 0) {
      int code = 0;
      if (phase == 1) {
        stop = rtol * rtol * (warm ? gref : g);
        if (!isfinite(g) || g < 0.0 || (warm && !(gref >= 0.0))) {
          code = 3;
        } else if (!(g > 0.0) || (warm && g <= stop)) {
          code = 1;
        } else if (!(d > 0.0)) {
          code = truncate && d < 0.0 ? 5 : 3;
          out[0] = g / -d;
        } else {
          den = d;
          out[0] = div_d(g, d);
          out[1] = 0.0;
          if (it >= max_it) code = 2;
        }
      } else if (!(g >= 0.0)) {  // preconditioner not positive definite (or non-finite)
        code = 3;
      } else if (g <= stop) {
        code = 1;
      } else {
        const double beta = div_d(g, gamma), dn = fma(-beta * beta, den, d);  // p_new^T K p_new
        if (!(dn > 0.0)) {
          code = truncate && dn < 0.0 ? 4 : 3;
        } else {
          den = dn;
          out[0] = div_d(g, dn);
          out[1] = beta;
          if (it + 1 >= max_it) code = 2;
        }
      }
      gamma = g;
      reinterpret_cast<int*>(out + 2)[0] = code;
    }
    __syncthreads();
    const int code = reinterpret_cast<const int*>(out + 2)[0];
    const double alpha = out[0], beta = out[1];
    if (phase == 2) ++it;
    if (code) {
      if (code == 5) {
#pragma unroll
        for (int q = 0; q < DPT; ++q) x[q] = fma(alpha, u[q], x[q]);
      }
      *status = code == 1 ? kStatusOk : code == 2 ? kStatusPcgCap : code == 3 ? kStatusPcgBreakdown : kStatusNegCurv;
      break;
    }
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
      p[q] = phase == 1 ? u[q] : fma(beta, p[q], u[q]);
      sv[q] = phase == 1 ? w[q] : fma(beta, sv[q], w[q]);
      x[q] = fma(alpha, p[q], x[q]);
      r[q] = fma(-alpha, sv[q], r[q]);
    }
    phase = 2;
  }
#pragma unroll
  for (int q = 0; q < DPT; ++q)
    if (s.act[q]) xs[s.dof[q]] = x[q];
  return it;
}

// Tangent at the current w: staged element tangents, coarse levels (build_mg), stencil rows.
template <int DPT, int LAW, bool kMG>
__device__ __forceinline__ void build_d2(const D2<DPT, LAW>& s, Row<DPT>& R, double (&Mi)[DPT][2], bool withL, double* Lb,
                                         bool build_mg) {
  element_tangents_d2(s);
  __syncthreads();
  if (kMG && s.mg.levels && build_mg) mg_build_d2(s.mg, s.ke);
  gather_rows_d2(s, R, Mi, withL, Lb);
  __syncthreads();
}

// Energy form of the tangent transfer on this lane's Gauss line of its elements (see element_transfer).
template <int DPT, int LAW>
__device__ __forceinline__ void transfer_d2(const D2<DPT, LAW>& s, const double* X, double (&Q)[10]) {
  const int half = threadIdx.x & 1;
  const double ih = (double)s.n, wq = 0.25 / (ih * ih), t = gauss01(half);
  const double2* w = reinterpret_cast<const double2*>(s.w);
  for (int k0 = 0; k0 < s.NN; k0 += s.T / 2) {
    const Elem2 el = elem2(k0 + (threadIdx.x >> 1), s.n, s.NN);
    if (!el.in) continue;
    const int ph = s.phase[el.e];
    const double lam = s.lame[2 * ph], mu = s.lame[2 * ph + 1];
    const double2 w0 = w[el.nd[0]], w1 = w[el.nd[1]], w2 = w[el.nd[2]], w3 = w[el.nd[3]];
    const double F00 = s.misc[0] + ih * ((w1.x - w0.x) + t * ((w2.x - w3.x) - (w1.x - w0.x)));
    const double F10 = s.misc[2] + ih * ((w1.y - w0.y) + t * ((w2.y - w3.y) - (w1.y - w0.y)));
#pragma unroll 1
    for (int g = 0; g < 2; ++g) {
      const double sg = gauss01(g);
      const double F01 = s.misc[1] + ih * ((w3.x - w0.x) + sg * ((w2.x - w1.x) - (w3.x - w0.x)));
      const double F11 = s.misc[3] + ih * ((w3.y - w0.y) + sg * ((w2.y - w1.y) - (w3.y - w0.y)));
      double k00, k01, k10, k11, hb = 0.0, gm = 0.0, S00 = 0.0, S01 = 0.0, S11 = 0.0;
      if constexpr (LAW == kLawNH) {
        const double J = F00 * F11 - F01 * F10, iJ = recip_d(J);
        k00 = F11 * iJ;
        k01 = -F10 * iJ;
        k10 = -F01 * iJ;
        k11 = F00 * iJ;
        hb = 0.5 * lam * (J * J - 1.0) - mu;
        gm = lam * J * J;
      } else {
        k00 = F00;
        k01 = F01;
        k10 = F10;
        k11 = F11;
        const double c00 = F00 * F00 + F10 * F10, c01 = F00 * F01 + F10 * F11, c11 = F01 * F01 + F11 * F11;
        const double trE = 0.5 * (c00 + c11) - 1.0;
        S00 = lam * trE + mu * (c00 - 1.0);
        S11 = lam * trE + mu * (c11 - 1.0);
        S01 = mu * c01;
      }
      double G[4][4], M[4][4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double2* Xc = reinterpret_cast<const double2*>(X + (size_t)c * s.ND);
        const double2 a0 = Xc[el.nd[0]], a1 = Xc[el.nd[1]], a2 = Xc[el.nd[2]], a3 = Xc[el.nd[3]];
        G[c][0] = ih * ((a1.x - a0.x) + t * ((a2.x - a3.x) - (a1.x - a0.x)));
        G[c][2] = ih * ((a1.y - a0.y) + t * ((a2.y - a3.y) - (a1.y - a0.y)));
        G[c][1] = ih * ((a3.x - a0.x) + sg * ((a2.x - a1.x) - (a3.x - a0.x)));
        G[c][3] = ih * ((a3.y - a0.y) + sg * ((a2.y - a1.y) - (a3.y - a0.y)));
        G[c][c] += 1.0;
        M[c][0] = k00 * G[c][0] + k10 * G[c][2];
        M[c][1] = k00 * G[c][1] + k10 * G[c][3];
        M[c][2] = k01 * G[c][0] + k11 * G[c][2];
        M[c][3] = k01 * G[c][1] + k11 * G[c][3];
      }
      int k = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int d = c; d < 4; ++d) {
          const double tm = M[c][0] * M[d][0] + M[c][1] * M[d][2] + M[c][2] * M[d][1] + M[c][3] * M[d][3];
          const double ac = M[c][0] + M[c][3], ad = M[d][0] + M[d][3];
          if constexpr (LAW == kLawNH) {
            const double gg = G[c][0] * G[d][0] + G[c][1] * G[d][1] + G[c][2] * G[d][2] + G[c][3] * G[d][3];
            Q[k] += wq * (mu * gg - hb * tm + gm * ac * ad);
          } else {
            const double mm = M[c][0] * M[d][0] + M[c][1] * M[d][1] + M[c][2] * M[d][2] + M[c][3] * M[d][3];
            const double gs = (G[c][0] * S00 + G[c][1] * S01) * G[d][0] + (G[c][0] * S01 + G[c][1] * S11) * G[d][1] +
                              (G[c][2] * S00 + G[c][3] * S01) * G[d][2] + (G[c][2] * S01 + G[c][3] * S11) * G[d][3];
            Q[k] += wq * (gs + lam * ac * ad + mu * (mm + tm));
          }
          ++k;
        }
    }
  }
}

// Whether a PCG that ended so is tried again with another preconditioner (fresh levels, less damping, block-Jacobi): a
// breakdown, and a cap that tells of one.  The no-allocation entry's callers may cap the PCG to truncate it: multigrid
// takes 10 to 25 iterations to the default tolerances (stiffness ratios up to 1000), so a cap below kTellingCap that
// binds is a truncation, whose step is taken as it is.  (Tried six times, 40 RVEs of 6^2 to 16^2 with caps of 2 to 20
// took 6.0 to 10.8 times as long as with block-Jacobi, which that entry ran before it had multigrid.)
constexpr int kTellingCap = 64;
template <bool kFixed>
__device__ __forceinline__ bool mends(int pst, int cap) {
  return pst == kStatusPcgBreakdown || (pst == kStatusPcgCap && (!kFixed || cap >= kTellingCap));
}

template <bool kFixed, bool kMG, int LAW, int DPT>
__device__ void solve_item_d2(const Rve2dArgs& a, int qp, unsigned char* smem, double* scr) {
  const int tid = threadIdx.x;
  const int rv = kFixed ? (a.phase_per_qp ? qp : 0) : a.qp_rve[qp];
  const int n = kFixed ? a.fixed_n : a.rve_n[rv];
  const int NN = n * n, ND = 2 * NN;
  const OffsetsD2 off = offsets_d2(NN, kMG);
  D2<DPT, LAW> s;
  s.n = n;
  s.NN = NN;
  s.ND = ND;
  s.T = blockDim.x;
  s.bc = a.bc;
  s.phase = a.phase + (kFixed ? (size_t)rv * NN : (size_t)a.rve_phase_off[rv]);
  s.w = reinterpret_cast<double*>(smem + off.w);
  s.p = reinterpret_cast<double*>(smem + off.p);
  s.x = reinterpret_cast<double*>(smem + off.x);
  s.stage = reinterpret_cast<double*>(smem + off.stage);
  s.red = reinterpret_cast<double*>(smem + off.red);
  s.lame = reinterpret_cast<double*>(smem + off.lame);
  s.restab = s.lame + 2 * kMaxPhase;
  s.misc = reinterpret_cast<double*>(smem + off.misc);
  s.ke = scr;
  s.st = scr + 36 * (size_t)NN;
  s.mg.n = n;
  s.mg.levels = kMG ? mg_levels(n) : 0;
  s.mg.bc = a.bc;
  s.mg.omega = (double)a.mg_omega;
  s.mg.fast = off.fast_in_smem ? reinterpret_cast<double*>(smem + off.fast) : scr + 72 * (size_t)NN;
  s.mg.slow = scr + (kRowInRegs<DPT> ? 36 * (size_t)NN : 72 * (size_t)NN + (kMG ? mg_fast_elems(n) : 0));
#pragma unroll
  for (int q = 0; q < DPT; ++q) {
    const int d = tid + q * s.T;
    s.act[q] = d < ND;
    s.dof[q] = s.act[q] ? d : (tid & 1);
    const int v = s.dof[q] >> 1, i = v % n, j = v / n;
    s.pin[q] = pinned2(i, j, a.bc);
    s.col[q][0] = wrap_dec(i, n);
    s.col[q][1] = i;
    s.col[q][2] = wrap_inc(i, n);
    s.row[q][0] = wrap_dec(j, n) * n;
    s.row[q][1] = j * n;
    s.row[q][2] = wrap_inc(j, n) * n;
  }
  if constexpr (kFixed) {  // device-supplied phase ids are checked before any table read
    int badp = 0;
    for (int e = tid; e < NN; e += s.T) badp |= s.phase[e] >= kMaxPhase;
    if (__syncthreads_or(badp)) {
      if (tid == 0) a.status[qp] = kStatusBadPhase;
      return;
    }
  }
  const size_t w_off = kFixed ? (size_t)qp * ND : (size_t)a.qp_w_off[qp];
  const double* w_in = a.w_in + w_off;
  double* w_out = a.w_out + w_off;
  if (tid < 4) s.misc[tid] = a.F[(size_t)qp * 4 + tid];
  const double* lame_g = a.rve_lame + (size_t)rv * 2 * kMaxPhase;
  if (tid < 2 * kMaxPhase) s.lame[tid] = lame_g[tid];
  residual_table(n, lame_g, s.restab);
#pragma unroll
  for (int q = 0; q < DPT; ++q)
    if (s.act[q]) s.w[s.dof[q]] = s.pin[q] ? 0.0 : w_in[s.dof[q]];
  __shared__ int s_ctl[4];  // stages, stage, Newton iterations of the earlier stages, newton_code
  if (tid == 0) {
    s_ctl[0] = 1;
    s_ctl[1] = 1;
    s_ctl[2] = 0;
  }
  __syncthreads();
  double* Xs = s.stage;            // [4][ND]
  double* Lb = s.stage + 4 * ND;   // [4][ND]
  Row<DPT> R;
  double Mi[DPT][2];
  int status = kStatusNewtonCap, it = 0, cg_total = 0;
  double Psum[4];
  // Newton with step halving, rebuild-and-retry and load continuation exactly as solve_item_2d (the reasons stand
  // there)
  for (;;) {
    int nhalf = 0;
    double r0 = 0.0, step = 1.0;
    it = 0;
    status = kStatusNewtonCap;
    for (;;) {
      Psum[0] = Psum[1] = Psum[2] = Psum[3] = 0.0;
      int nbad = 0;
      block_residual<LAW>(n, reinterpret_cast<const double2*>(s.w), s.misc, s.restab, s.phase, s.stage, Psum, nbad);
      const bool bad = __syncthreads_or(nbad);
      double Rv[DPT], v2[1] = {0.0};
#pragma unroll
      for (int q = 0; q < DPT; ++q) {
        const int c = tid & 1, i = s.col[q][1], im = s.col[q][0], jr = s.row[q][1], jm = s.row[q][0];
        const double* f = s.stage + c * NN;
        Rv[q] = (f[i + jr] + f[2 * NN + im + jr]) + (f[4 * NN + im + jm] + f[6 * NN + i + jm]);
        if (!s.act[q] || s.pin[q]) Rv[q] = 0.0;
        v2[0] = fma(Rv[q], Rv[q], v2[0]);
      }
      block_sum_fp64<1>(v2, s.red);
      const int code = newton_code(bad, v2[0], it, nhalf, r0, a.newton_rtol, a.newton_atol,
                                   s_ctl[0] > 1 ? max(a.max_newton, kRetryNewtonCap) : a.max_newton, s_ctl + 3);
      if (code == kNewtonHalve) {
        ++nhalf;
        step *= 0.5;
#pragma unroll
        for (int q = 0; q < DPT; ++q)
          if (s.act[q]) s.w[s.dof[q]] -= step * s.x[s.dof[q]];
        __syncthreads();
        continue;
      }
      if (code >= 0) {
        status = code;
        break;
      }
      bool reuse = kMG && s.mg.levels && a.mg_reuse && it > 0;
      double b[DPT];
#pragma unroll
      for (int q = 0; q < DPT; ++q) b[q] = -Rv[q];
      int pst = kStatusOk;
      const double omega0 = s.mg.omega;
      for (;;) {
        build_d2<DPT, LAW, kMG>(s, R, Mi, false, nullptr, !reuse);
        cg_total += pcg_d2<DPT, LAW, kMG>(s, R, Mi, b, s.x, a.cg_rtol, a.max_cg, &pst, true, false);
        __syncthreads();
        const bool mended = mends<kFixed>(pst, a.max_cg);
        if (reuse && (mended || pst == kStatusNegCurv)) {
          reuse = false;
        } else if (kMG && s.mg.levels && mended && s.mg.omega > 0.2 * omega0) {
          s.mg.omega *= 0.5;
        } else if (kFixed && kMG && s.mg.levels && mended) {
          s.mg.levels = 0;  // block-Jacobi, the entry's preconditioner for grids without a hierarchy
        } else {
          break;
        }
        pst = kStatusOk;
      }
      s.mg.omega = omega0;
      if (kFixed && kMG) s.mg.levels = mg_levels(n);
      if (pst == kStatusPcgBreakdown) {
        status = kStatusPcgBreakdown;
        break;
      }
      step = 1.0;
      nhalf = 0;
#pragma unroll
      for (int q = 0; q < DPT; ++q)
        if (s.act[q]) s.w[s.dof[q]] += s.x[s.dof[q]];
      __syncthreads();
      ++it;
    }
    const bool failed = !(status == kStatusOk || status == kStatusNewtonCap);
    int stages = s_ctl[0], stage = s_ctl[1];
    if (failed && stages == 1 && a.retry_stages > 1) {
      stages = a.retry_stages;
      stage = 0;
#pragma unroll
      for (int q = 0; q < DPT; ++q)
        if (s.act[q]) s.w[s.dof[q]] = 0.0;
    } else if (failed || stage >= stages) {
      break;
    }
    ++stage;
    __syncthreads();  // every thread has read s_ctl and finished with this stage's Fbar
    if (tid < 4) {
      const double Ft = a.F[(size_t)qp * 4 + tid], id = (tid == 0 || tid == 3) ? 1.0 : 0.0;
      s.misc[tid] = stage == stages ? Ft : id + (Ft - id) * stage / stages;
    }
    if (tid == 0) {
      s_ctl[0] = stages;
      s_ctl[1] = stage;
      s_ctl[2] += it;
    }
    __syncthreads();
  }
  const int it_total = s_ctl[2] + it;

  double Pv[5] = {Psum[0], Psum[1], Psum[2], Psum[3], 0.0};
  const bool usable = (status == kStatusOk || status == kStatusNewtonCap);
  const bool want_W = usable && (a.flags & kFlagEnergy) && a.W != nullptr;
  if (want_W)
    for (int e = tid; e < NN; e += s.T) {
      const int ph = s.phase[e];
      Pv[4] += element_energy<LAW>(e, n, reinterpret_cast<const double2*>(s.w), s.misc, s.lame[2 * ph], s.lame[2 * ph + 1]);
    }
  block_sum_fp64<5>(Pv, s.red);

  int cond_total = 0, cond_max = 0;
  double Q[10];
  const bool want_A = usable && !(a.flags & kFlagNoTangent) && a.A != nullptr;
  if (want_A) {
    const bool warm = a.X_in != nullptr;
    const double* X0 = warm ? reinterpret_cast<const double*>(a.X_in) + 4 * w_off : nullptr;
    const double omega0 = s.mg.omega;
    bool reuse_t = kMG && s.mg.levels && a.mg_reuse && it > 0;
    for (;;) {
      __syncthreads();  // the element forces in the stage have been read
      build_d2<DPT, LAW, kMG>(s, R, Mi, true, Lb, !reuse_t);
      bool redo = false;
      int t_total = 0, t_max = 0, t_status = kStatusOk;
      for (int k = 0; k < 4; ++k) {
        double b[DPT];
#pragma unroll
        for (int q = 0; q < DPT; ++q) b[q] = s.act[q] ? Lb[(size_t)k * ND + s.dof[q]] : 0.0;
        int pst = kStatusOk, ci = 0;
        bool kept = warm;
        for (;;) {
          if (kept) {
#pragma unroll
            for (int q = 0; q < DPT; ++q)
              if (s.act[q]) Xs[(size_t)k * ND + s.dof[q]] = s.pin[q] ? 0.0 : X0[(size_t)k * ND + s.dof[q]];
          }
          ci += pcg_d2<DPT, LAW, kMG>(s, R, Mi, b, Xs + (size_t)k * ND, a.cond_rtol, a.max_cond_cg, &pst, false, kept);
          __syncthreads();
          const bool mended = mends<kFixed>(pst, a.max_cond_cg);
          if (reuse_t && mended) {
            redo = true;
            break;
          }
          if (kMG && s.mg.levels && mended && (kFixed || s.mg.omega > 0.2 * omega0)) {
            if (s.mg.omega > 0.2 * omega0) s.mg.omega *= 0.5;
            else s.mg.levels = 0;
          } else if (kept && pst == kStatusPcgBreakdown) {  // from zero (see solve_item_2d)
            kept = false;
            s.mg.omega = omega0;
          } else {
            break;
          }
          pst = kStatusOk;
        }
        s.mg.omega = omega0;
        if (kFixed && kMG) s.mg.levels = mg_levels(n);
        t_total += ci;
        t_max = ci > t_max ? ci : t_max;
        if (redo) break;
        if (pst != kStatusOk && t_status == kStatusOk) t_status = pst;
      }
      cond_total += t_total;
      cond_max = t_max > cond_max ? t_max : cond_max;
      if (!redo) {
        if (t_status != kStatusOk && status == kStatusOk) status = t_status;
        break;
      }
      reuse_t = false;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 10; ++k) Q[k] = 0.0;
    transfer_d2(s, Xs, Q);
    block_sum_fp64<10>(Q, s.red);
  }

#pragma unroll
  for (int q = 0; q < DPT; ++q)
    if (s.act[q]) w_out[s.dof[q]] = s.w[s.dof[q]];
  if (want_A && a.X_out) {
    double* Xo = reinterpret_cast<double*>(a.X_out) + 4 * w_off;
    for (int v = tid; v < 4 * ND; v += s.T) Xo[v] = Xs[v];
  }
  if (tid == 0) {
    a.status[qp] = status;
    if (a.iters) {
      a.iters[(size_t)qp * 4 + 0] = it_total;
      a.iters[(size_t)qp * 4 + 1] = cg_total;
      a.iters[(size_t)qp * 4 + 2] = cond_total;
      a.iters[(size_t)qp * 4 + 3] = cond_max;
    }
    if (usable) {
      const double wq = 0.25 / ((double)n * n);  // Gauss weight x det J; |Omega| = 1
#pragma unroll
      for (int k = 0; k < 4; ++k) a.P[(size_t)qp * 4 + k] = Pv[k] * wq;
      if (want_W) a.W[qp] = Pv[4] * wq;
      if (want_A) {
        int k = 0;
        for (int c = 0; c < 4; ++c)
          for (int d = c; d < 4; ++d) {
            a.A[(size_t)qp * 16 + c * 4 + d] = Q[k];
            a.A[(size_t)qp * 16 + d * 4 + c] = Q[k];
            ++k;
          }
      }
    }
  }
  __syncthreads();
}

template <bool kFixed, bool kMG, int LAW, int DPT>
__global__ void __launch_bounds__(kThreadsD2, 1) rve2d_fp64_kernel(const Rve2dArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_item;
  double* scr = reinterpret_cast<double*>(a.scratch) + (size_t)blockIdx.x * a.scratch_stride;
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(a.queue, 1);
    __syncthreads();
    const int item = s_item;
    __syncthreads();
    if (item >= (a.n_dev ? *a.n_dev : a.n_qp)) break;
    const int qp = kFixed ? item : a.order[item];
    if (!kFixed && a.only_n && a.rve_n[a.qp_rve[qp]] != a.only_n) continue;  // another launch's grid
    solve_item_d2<kFixed, kMG, LAW, DPT>(a, qp, smem_raw, scr);
  }
}

}  // namespace

template <bool kFixed, bool kMG, int LAW, int DPT>
inline cudaError_t rve2d_launch_fp64(const Rve2dArgs& a, int n_blocks, cudaStream_t stream) {
  const size_t smem = offsets_d2(a.nn_max, kMG).total;
  constexpr size_t most = most_smem_d2(kMG);  // the kernel's limit for every thread that launches it
  const cudaError_t err = cudaFuncSetAttribute(rve2d_fp64_kernel<kFixed, kMG, LAW, DPT>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (err != cudaSuccess) return err;
  rve2d_fp64_kernel<kFixed, kMG, LAW, DPT><<<n_blocks, threads_d2(a.nn_max), smem, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace fehmm
