// The whole-network kernels: value, input gradient and input Hessian (eval_hess_kernel), and value and input
// gradient or a whole loss gradient (grad_kernel).  Included by mlp.cu behind the layer functions.
#pragma once

#include "mlp_fused.cuh"

namespace fehmm {
namespace fused {

struct Net {
  const bf16* W1;    // [128][8]
  const bf16* W[3];  // W2..W4 [128][128]
  const bf16* W1T;   // [8][128]
  const bf16* w5;    // [128]
  const float* b[4];
  const float* b5;
};

// ------------------------------------------------------------------ value, gradient, Hessian
// A tile is 16 samples x 8 rows: row d * 16 + s is the forward tangent of sample s along input d (d < 6), the
// sample itself (d = 6), or unused (d = 7).  The forward products of samples and tangents are the same product
// (a_l and silu'(z_l) dz_l times W^T), and so are the backward ones (delta_l and its tangent times W), so a
// tile needs six 128^3 products; tensor memory keeps the tangents dz_2..dz_4 of the forward pass for the
// backward one.  silu and its derivatives are evaluated once per sample and unit by all threads together, and
// passed to the tangent rows through shared memory.  Bound by that exchange (four barriers a layer), not by
// the tensor pipe: 32768 points 1.26 ms layer by layer, 0.191 ms here (0.228 with 256 threads); 1000 points
// 21 us.
constexpr int kEvalThreads = 512, kEvalSamples = 16, kLd = 132;  // kLd: padded row (bank-conflict free float4)

struct EvalSmem {
  uint8_t w[3 * kTileBytes];
  uint8_t a[kTileBytes];
  float z[3][kEvalSamples][kLd];  // z_1..z_3
  float buf[kEvalSamples][kLd], sd[kEvalSamples][kLd], aux[kEvalSamples][kLd];
  float bias[4][128], w5[128];
  bf16 w1[128 * 8], w1t[8 * 128], x[16 * 8];
  uint64_t bar;
  uint32_t slot;
};

__global__ void __launch_bounds__(kEvalThreads, 1)
eval_hess_kernel(const Net net, const float* x, int B, float* y, float* g, float* H, int* err) {
  extern __shared__ __align__(1024) uint8_t fused_smem[];
  EvalSmem& sm = *reinterpret_cast<EvalSmem*>(fused_smem);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int quad = warp & 3, col0 = (warp >> 2) * 32;  // TMEM lanes 32 quad .., columns col0 .. + 31
  const int row = 32 * quad + lane, d = row >> 4, s = row & 15;
  const int es = t >> 5, ej = (t & 31) * 4;  // elementwise: sample es, units ej .. ej + 3
  load_weights(sm.w, net.W[0], net.W[1], net.W[2]);
  for (int e = t; e < 128; e += kEvalThreads) {
    for (int l = 0; l < 4; ++l) sm.bias[l][e] = net.b[l][e];
    sm.w5[e] = __bfloat162float(net.w5[e]);
  }
  for (int e = t; e < 1024; e += kEvalThreads) {
    sm.w1[e] = net.W1[e];
    sm.w1t[e] = net.W1T[e];
  }
  {  // the unused rows stay zero
    const float zero[4] = {0.f, 0.f, 0.f, 0.f};
    store4(sm.a, 112 + es, ej, zero);
  }
  tc::cp_async_wait<0>();
  const uint32_t tmem = block_begin(&sm.bar, &sm.slot);
  const uint32_t my_lanes = tmem + ((uint32_t)(32 * quad) << 16);
  const uint32_t wa = tc::smem_u32(sm.w), aa = tc::smem_u32(sm.a);
  uint32_t parity = 0;
  bool failed = false;
  // operand tile complete -> one product into TMEM columns c, waited for
  auto forward_or_back = [&](int l, bool back, uint32_t c) {
    fence_smem();
    fence_before();
    __syncthreads();
    if (t == 0) {
      fence_after();
      const uint32_t w = wa + (l - 2) * kTileBytes;
      if (back)
        product<false, true, 128>(tmem + c, aa, w, 8, false);
      else
        product<false, false, 128>(tmem + c, aa, w, 8, false);
      tc::mma_commit(tc::smem_u32(&sm.bar));
    }
    failed = __syncthreads_or(!tc::mbar_wait(tc::smem_u32(&sm.bar), parity));  // every thread takes the same way
    parity ^= 1;
    fence_after();
  };
  // the samples' rows of a product -> buf
  auto samples_to_buf = [&](uint32_t c) {
    if (quad == 3) {
      float v[32];
      tmem_load<32>(my_lanes + c + col0, v);
      if (lane < 16) {
#pragma unroll
        for (int k = 0; k < 32; k += 4)
          *reinterpret_cast<float4*>(&sm.buf[lane][col0 + k]) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
      }
    }
    __syncthreads();
  };
  const int tiles = (B + kEvalSamples - 1) / kEvalSamples;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int b0 = tile * kEvalSamples;
    if (t < 128) {
      const int q = b0 + (t >> 3), k = t & 7;
      sm.x[t] = __float2bfloat16(q < B && k < 6 ? x[(size_t)q * 6 + k] : 0.f);
    }
    __syncthreads();
    {  // z_1 without its bias, 8 units a warp
      float v[4];
      input_layer(reinterpret_cast<const uint8_t*>(sm.x), 128, sm.w1, warp, v);
      const int r = lane >> 2, c = 8 * warp + 2 * (lane & 3);
      sm.buf[r][c] = v[0];
      sm.buf[r][c + 1] = v[1];
      sm.buf[r + 8][c] = v[2];
      sm.buf[r + 8][c + 1] = v[3];
    }
    __syncthreads();
    for (int l = 1; l <= 4 && !failed; ++l) {  // buf holds z_l without its bias
      {
        float a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float z = sm.buf[es][ej + k] + sm.bias[l - 1][ej + k];
          const float dz = silu_d(z);
          if (l < 4) {
            sm.z[l - 1][es][ej + k] = z;
            sm.sd[es][ej + k] = dz;
            a[k] = silu_f(z);
          } else {  // the output layer and delta_4 = w5 silu'(z_4)
            const float w = sm.w5[ej + k];
            sm.buf[es][ej + k] = __bfloat162float(__float2bfloat16(silu_f(z)));
            sm.aux[es][ej + k] = w * silu_dd(z);
            a[k] = w * dz;
          }
        }
        store4(sm.a, 96 + es, ej, a);
      }
      __syncthreads();
      if (l == 4 && y) {  // y = w5 . a_4 + b5, one warp per sample
        float v = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) v += sm.w5[lane + 32 * j] * sm.buf[warp][lane + 32 * j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && b0 + warp < B) y[b0 + warp] = v + net.b5[0];
      }
      if (quad < 3) {  // tangents: silu'(z_l) dz_l, at the top w5 silu''(z_4) dz_4
        const float(*f)[kLd] = l < 4 ? sm.sd : sm.aux;
        float v[32];
        if (l == 1) {
#pragma unroll
          for (int k = 0; k < 32; ++k) v[k] = __bfloat162float(sm.w1t[d * 128 + col0 + k]);
        } else {
          tmem_load<32>(my_lanes + (l - 2) * 128 + col0, v);
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] *= f[s][col0 + k];
#pragma unroll
        for (int k = 0; k < 32; k += 8) store8(sm.a, row, col0 + k, v + k);
      }
      if (l < 4) {
        forward_or_back(l + 1, false, (l - 1) * 128);
        if (!failed) samples_to_buf((l - 1) * 128);
      }
    }
    for (int l = 3; l >= 1 && !failed; --l) {  // delta_l = (delta_{l+1} W_{l+1}) silu'(z_l), and its tangents
      forward_or_back(l + 1, true, 384);
      if (failed) break;
      samples_to_buf(384);
      {
        float a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float z = sm.z[l - 1][es][ej + k], c = sm.buf[es][ej + k], dz = silu_d(z);
          sm.sd[es][ej + k] = dz;
          sm.aux[es][ej + k] = c * silu_dd(z);
          a[k] = c * dz;
        }
        store4(sm.a, 96 + es, ej, a);
      }
      __syncthreads();
      if (quad < 3) {
        float v[32], zd[32];
        tmem_load<32>(my_lanes + 384 + col0, v);
        if (l == 1) {
#pragma unroll
          for (int k = 0; k < 32; ++k) zd[k] = __bfloat162float(sm.w1t[d * 128 + col0 + k]);
        } else {
          tmem_load<32>(my_lanes + (l - 2) * 128 + col0, zd);
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = __fmaf_rn(v[k], sm.sd[s][col0 + k], __fmul_rn(sm.aux[s][col0 + k], zd[k]));
#pragma unroll
        for (int k = 0; k < 32; k += 8) store8(sm.a, row, col0 + k, v + k);
      }
    }
    if (failed) break;
    __syncthreads();
    if (warp < 7) {  // through the input layer: rows 16 warp .. are direction `warp`, or the gradient
      float v[4];
      times_w1(sm.a, warp, sm.w1t, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int q = b0 + (lane >> 2) + (e >> 1) * 8, j = 2 * (lane & 3) + (e & 1);
        if (q >= B || j >= 6) continue;
        if (warp < 6)
          H[(size_t)q * 36 + j * 6 + warp] = v[e];
        else if (g)
          g[(size_t)q * 6 + j] = v[e];
      }
    }
  }
  if (failed && t == 0) atomicExch(err, 1);
  block_end(tmem);
}

// ------------------------------------------------------------------ value and gradient; loss gradient
// A tile is ROWS samples (32, 64 or 128).  The products always have 128 rows; with fewer samples they are
// repeated 128 / ROWS times down the operand, so that every warp finds all samples in the tensor-memory lanes
// it can read, and a thread has 32 ROWS / 128 columns of one sample: a step's elementwise work (silu and its
// derivatives, the longest part of it) shrinks with the tile, and a batch of 4096 spreads over 128 SMs in place
// of 32.  kTrain: then the loss residuals and the reverse pass through the gradient and the forward pass,
// with the weight gradients' products (K = the tile's samples) accumulated in tensor memory over all tiles of
// the block and added to the gradient once.  z_l, C_l = delta_{l+1} W_{l+1} and q_l wait in global memory (a
// private [column / 4][row] layout, coalesced), the BF16 operands of the weight gradients as tile images that
// return by cp.async one step ahead.  Twelve products in a row per tile: bound by their latency and the
// elementwise steps between them.  A training step (loss, gradient, AdamW) of 4096 samples: 505 us layer by
// layer, 122 us with 128 samples a tile, 60 us with 32; of 16384: 142 us (128 samples a tile).
constexpr int kGradThreads = 512, kGradMaxRows = 128;

struct GradSmem {
  uint8_t w[3 * kTileBytes];
  uint8_t t[3][kTileBytes];
  uint8_t x[4096], rg[4096];  // 128 x 16 BF16 (features 8 .. 15 zero), row groups 256 bytes apart
  float g[128][8];
  float y[128], ry[128];
  float bias[4][128], w5[128];
  bf16 w1[128 * 8], w1t[8 * 128];
  uint64_t bar;
  uint32_t slot;
};

struct GradArgs {
  Net net;
  const float *x, *ty, *tg;
  int B;
  float cy, cg;
  float *y, *g;         // outputs of the evaluation (null: not wanted)
  float *G, *loss;      // training: gradient (zeroed) and loss (zeroed)
  float *Z[4], *C[3], *Q[3];  // [tiles][ROWS * 128]: z_1..z_4, C_1..C_3, q_1..q_3
  uint8_t *A[3], *D[3];       // tile images of a_1..a_3, delta_2..delta_4
  int off_w[5], off_b[5];     // offsets of W_l, b_l in G (index 4: w5, b5)
  int* err;
};

__device__ __forceinline__ uint32_t narrow_off(int r, int c) {
  return (uint32_t)(r >> 3) * 256 + (uint32_t)(c >> 3) * 128 + (uint32_t)(r & 7) * 16 + (uint32_t)(c & 7) * 2;
}

// v[k] summed over the warp's 32 lanes; the lanes whose index is a multiple of 32 / NC receive column
// lane / (32 / NC) (each step halves the columns a lane still carries)
template <int NC>
__device__ __forceinline__ float column_sum(float (&v)[NC]) {
  const int lane = threadIdx.x & 31;
  int n = NC;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = lane & o;
#pragma unroll
      for (int k = 0; k < NC / 2; ++k) {
        if (k >= n) break;
        const float send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}

template <bool kTrain, int ROWS>
__global__ void __launch_bounds__(kGradThreads, 1) grad_kernel(const __grid_constant__ GradArgs p) {
  extern __shared__ __align__(1024) uint8_t fused_smem[];
  GradSmem& sm = *reinterpret_cast<GradSmem*>(fused_smem);
  const Net& net = p.net;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  constexpr int COPIES = 128 / ROWS, NC = 32 / COPIES;  // columns of a thread
  const int quad = warp & 3, tl = 32 * quad + lane;    // TMEM lane
  const int row = tl % ROWS, c0 = (warp >> 2) * 32 + tl / ROWS * NC;
  load_weights(sm.w, net.W[0], net.W[1], net.W[2]);
  for (int e = t; e < 1024; e += kGradThreads) {
    sm.w1[e] = net.W1[e];
    sm.w1t[e] = net.W1T[e];
    reinterpret_cast<uint32_t*>(sm.x)[e] = 0u;
    reinterpret_cast<uint32_t*>(sm.rg)[e] = 0u;
  }
  for (int e = t; e < 128; e += kGradThreads) {
    for (int l = 0; l < 4; ++l) sm.bias[l][e] = net.b[l][e];
    sm.w5[e] = __bfloat162float(net.w5[e]);
  }
  tc::cp_async_wait<0>();
  const uint32_t tmem = block_begin(&sm.bar, &sm.slot);
  const uint32_t my_lanes = tmem + ((uint32_t)(32 * quad) << 16), work = 384;
  const uint32_t bar = tc::smem_u32(&sm.bar);
  const uint32_t wa = tc::smem_u32(sm.w);
  const uint32_t ta[3] = {tc::smem_u32(sm.t[0]), tc::smem_u32(sm.t[1]), tc::smem_u32(sm.t[2])};
  uint32_t parity = 0;
  bool failed = false;
  float sum_b[4] = {0.f, 0.f, 0.f, 0.f}, sum_w5 = 0.f, sum_b5 = 0.f;  // column sums of this lane's column
  auto ready = [&]() {  // operands complete
    fence_smem();
    fence_before();
    __syncthreads();
    if (t == 0) fence_after();
  };
  auto done = [&]() {  // the products of this step (committed by thread 0); every thread takes the same way after
    failed = __syncthreads_or(!tc::mbar_wait(bar, parity));
    parity ^= 1;
    fence_after();
  };
  auto image_out = [&](uint8_t* img, int c, const float* v) {
    *reinterpret_cast<uint4*>(img + core_off(row, c)) = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
  };
  auto image_in = [&](int k, const uint8_t* img) {
    for (int e = t; e < ROWS * 16; e += kGradThreads) tc::cp_async16(ta[k] + 16 * e, img + 16 * e, 16);
    tc::cp_async_commit();
  };
  auto save = [&](float* m, const float (&v)[NC]) {
    float4* q = reinterpret_cast<float4*>(m) + (c0 / 4) * ROWS + row;
#pragma unroll
    for (int k = 0; k < NC / 4; ++k) q[k * ROWS] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
  };
  auto load = [&](const float* m, float (&v)[NC]) {
    const float4* q = reinterpret_cast<const float4*>(m) + (c0 / 4) * ROWS + row;
#pragma unroll
    for (int k = 0; k < NC / 4; ++k) {
      const float4 f = q[k * ROWS];
      v[4 * k] = f.x;
      v[4 * k + 1] = f.y;
      v[4 * k + 2] = f.z;
      v[4 * k + 3] = f.w;
    }
  };
  auto at = [&](float* m, int r, int c) { return reinterpret_cast<float2*>(m + ((c >> 2) * ROWS + r) * 4 + (c & 3)); };
  auto to_tile = [&](int k, const float (&v)[NC]) {
#pragma unroll
    for (int j = 0; j < NC; j += 8)
#pragma unroll
      for (int c = 0; c < COPIES; ++c) store8(sm.t[k], row + c * ROWS, c0 + j, v + j);
  };
  const int tiles = (p.B + ROWS - 1) / ROWS;
  bool more = false;  // a weight gradient of an earlier tile is in tensor memory
  for (int tile = blockIdx.x; tile < tiles && !failed; tile += gridDim.x) {
    const int b0 = tile * ROWS;
    const size_t mat = (size_t)tile * ROWS * 128, img = (size_t)tile * ROWS * 256;
    for (int e = t; e < ROWS * 6; e += kGradThreads) {
      const int r = e / 6, k = e % 6;
      *reinterpret_cast<bf16*>(sm.x + narrow_off(r, k)) = __float2bfloat16(b0 + r < p.B ? p.x[(size_t)(b0 + r) * 6 + k] : 0.f);
    }
    __syncthreads();
    constexpr int RT = ROWS / 16;  // 16-row tiles of the mma.sync products, dealt to the warps by units of 16 x 8
    const int g4 = lane >> 2, t4 = 2 * (lane & 3);
#pragma unroll 1
    for (int u = warp; u < 16 * RT; u += kGradThreads / 32) {  // input layer
      float v[4];
      const int r = 16 * (u % RT) + g4, nt = u / RT, c = 8 * nt + t4;
      input_layer(sm.x + narrow_off(16 * (u % RT), 0), 256, sm.w1, nt, v);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float z0 = v[2 * h] + sm.bias[0][c], z1 = v[2 * h + 1] + sm.bias[0][c + 1];
        *at(p.Z[0] + mat, r + 8 * h, c) = make_float2(z0, z1);
        const uint32_t a = pack2(silu_f(z0), silu_f(z1));
#pragma unroll
        for (int q = 0; q < COPIES; ++q) *reinterpret_cast<uint32_t*>(sm.t[0] + core_off(r + 8 * h + q * ROWS, c)) = a;
        if (kTrain) *reinterpret_cast<uint32_t*>(p.A[0] + img + core_off(r + 8 * h, c)) = a;
      }
    }
    for (int l = 2; l <= 4; ++l) {  // forward
      ready();
      if (t == 0) {
        product<false, false, 128>(tmem + work, ta[0], wa + (l - 2) * kTileBytes, 8, false);
        tc::mma_commit(bar);
      }
      done();
      if (failed) break;
      float v[NC], a[NC];
      tmem_load<NC>(my_lanes + work + c0, v);
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        v[k] += sm.bias[l - 1][c0 + k];
        a[k] = silu_f(v[k]);
      }
      save(p.Z[l - 1] + mat, v);
      to_tile(0, a);
      if (kTrain && l < 4)
#pragma unroll
        for (int k = 0; k < NC; k += 8) image_out(p.A[l - 1] + img, c0 + k, a + k);
      if (l == 4) {  // y = w5 . a_4 + b5 (one warp per sample), then delta_4 in the place of a_4
        __syncthreads();
        for (int q = warp; q < ROWS; q += kGradThreads / 32) {
          float y = 0.f;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            y += sm.w5[lane + 32 * j] *
                 __bfloat162float(*reinterpret_cast<const bf16*>(sm.t[0] + core_off(q, lane + 32 * j)));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
          if (lane == 0) {
            y += net.b5[0];
            sm.y[q] = y;
            if (p.y && b0 + q < p.B) p.y[b0 + q] = y;
          }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NC; ++k) a[k] = sm.w5[c0 + k] * silu_d(v[k]);
        to_tile(0, a);
        if (kTrain)
#pragma unroll
          for (int k = 0; k < NC; k += 8) image_out(p.D[2] + img, c0 + k, a + k);
      }
    }
    for (int l = 3; l >= 1 && !failed; --l) {  // delta_l = C_l silu'(z_l), C_l = delta_{l+1} W_{l+1}
      float z[NC], v[NC];
      load(p.Z[l - 1] + mat, z);  // of l = 1: other threads' values, behind the barriers since
      ready();
      if (t == 0) {
        product<false, true, 128>(tmem + work, ta[0], wa + (l - 1) * kTileBytes, 8, false);
        tc::mma_commit(bar);
      }
      done();
      if (failed) break;
      tmem_load<NC>(my_lanes + work + c0, v);
      if (kTrain) save(p.C[l - 1] + mat, v);
#pragma unroll
      for (int k = 0; k < NC; ++k) v[k] *= silu_d(z[k]);
      to_tile(0, v);
      if (kTrain && l > 1)
#pragma unroll
        for (int k = 0; k < NC; k += 8) image_out(p.D[l - 2] + img, c0 + k, v + k);
    }
    if (failed) break;
    __syncthreads();
    if (warp < RT) {  // g = delta_1 W_1
      float v[4];
      times_w1(sm.t[0], warp, sm.w1t, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) sm.g[16 * warp + (lane >> 2) + 8 * (e >> 1)][2 * (lane & 3) + (e & 1)] = v[e];
    }
    __syncthreads();
    if (p.g)
      for (int e = t; e < ROWS * 6; e += kGradThreads)
        if (b0 + e / 6 < p.B) p.g[(size_t)b0 * 6 + e] = sm.g[e / 6][e % 6];
    if constexpr (kTrain) {
      image_in(2, p.D[0] + img);  // delta_2
      float l_sum = 0.f;
      if (t < ROWS) {  // loss residuals of sample t
        const bool in = b0 + t < p.B;
        const float e = in ? sm.y[t] - p.ty[b0 + t] : 0.f;
        sm.ry[t] = p.cy * e;
        sum_b5 += p.cy * e;
        l_sum += p.cy * e * e;
        float r[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const float eg = in ? sm.g[t][k] - p.tg[(size_t)(b0 + t) * 6 + k] : 0.f;
          r[k] = p.cg * eg;
          l_sum += p.cg * eg * eg;
        }
        *reinterpret_cast<uint4*>(sm.rg + narrow_off(t, 0)) = make_uint4(pack2(r[0], r[1]), pack2(r[2], r[3]), pack2(r[4], r[5]), 0u);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l_sum += __shfl_xor_sync(0xffffffffu, l_sum, o);
        if (lane == 0) atomicAdd(p.loss, 0.5f * l_sum);
      }
      // units x features: delta^T rg (or dz_1^T x) into 16 work columns, then added to the gradient of W_1
      auto narrow_product = [&](uint32_t a, const uint8_t* b) {
        constexpr uint32_t idesc = tc::idesc_bf16_f32(128, 16) | (1u << 15) | (1u << 16);
        const uint32_t bb = tc::smem_u32(b);
        for (int k = 0; k < RT; ++k)
          tc::mma_bf16(tmem + work, desc(a + k * 2 * kRowGroup, kRowGroup, kColGroup), desc(bb + k * 512, 256, 128), idesc, k > 0);
      };
      auto narrow_add = [&]() {
        if (warp < 4) {  // lane = unit
          float v[8];
          tmem_load<8>(my_lanes + work, v);
#pragma unroll
          for (int k = 0; k < 6; ++k) atomicAdd(p.G + p.off_w[0] + tl * 8 + k, v[k]);
        }
      };
      ready();
      if (t == 0) {
        narrow_product(ta[0], sm.rg);
        tc::mma_commit(bar);
      }
#pragma unroll 1
      for (int u = warp; u < 16 * RT; u += kGradThreads / 32) {  // e_1 = rg W_1^T, es_1 = e_1 silu'(z_1), q_1 = e_1 C_1 silu''(z_1)
        float v[4];
        const int r = 16 * (u % RT) + g4, nt = u / RT, c = 8 * nt + t4;
        input_layer(sm.rg + narrow_off(16 * (u % RT), 0), 256, sm.w1, nt, v);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 z = *at(p.Z[0] + mat, r + 8 * h, c), cc = *at(p.C[0] + mat, r + 8 * h, c);
          const float e0 = v[2 * h], e1 = v[2 * h + 1];
          *at(p.Q[0] + mat, r + 8 * h, c) = make_float2(e0 * cc.x * silu_dd(z.x), e1 * cc.y * silu_dd(z.y));
          const uint32_t es = pack2(e0 * silu_d(z.x), e1 * silu_d(z.y));
#pragma unroll
          for (int q = 0; q < COPIES; ++q) *reinterpret_cast<uint32_t*>(sm.t[1] + core_off(r + 8 * h + q * ROWS, c)) = es;
        }
      }
      done();
      if (!failed) {
        narrow_add();
        image_in(0, p.D[1] + img);  // delta_3
      }
      for (int l = 1; l <= 3 && !failed; ++l) {  // e_{l+1} = es_l W_{l+1}^T; gradient of W_{l+1} += delta_{l+1}^T es_l
        float z[NC], v[NC], c[NC];
        load(p.Z[l] + mat, z);
        if (l < 3) load(p.C[l] + mat, c);
        tc::cp_async_wait<1>();
        const uint32_t dt = ta[l == 2 ? 0 : 2];
        ready();
        if (t == 0) {
          product<false, false, 128>(tmem + work, ta[1], wa + (l - 1) * kTileBytes, 8, false);
          product<true, true, 128>(tmem + (l - 1) * 128, dt, ta[1], RT, more);
          tc::mma_commit(bar);
        }
        done();
        if (failed) break;
        // one step ahead: delta_4, then a_3, a_2
        if (l == 1) image_in(2, p.D[2] + img);
        if (l == 2) image_in(0, p.A[2] + img);
        if (l == 3) image_in(2, p.A[1] + img);
        tmem_load<NC>(my_lanes + work + c0, v);
        if (l < 3) {
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            c[k] = v[k] * c[k] * silu_dd(z[k]);
            v[k] *= silu_d(z[k]);
          }
          save(p.Q[l] + mat, c);
          to_tile(1, v);
        } else {  // dz_4 = ry w5 silu'(z_4) + e_4 w5 silu''(z_4); gradient of w5: e_4 silu'(z_4) + a_4 ry
          const float ry = sm.ry[row];
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            const float w = sm.w5[c0 + k], sd = silu_d(z[k]);
            const float q = v[k] * w * silu_dd(z[k]);
            c[k] = __fmaf_rn(v[k], sd, __bfloat162float(__float2bfloat16(silu_f(z[k]))) * ry);
            v[k] = __fmaf_rn(ry * w, sd, q);
          }
          to_tile(1, v);
          sum_w5 += column_sum(c);
          sum_b[3] += column_sum(v);
        }
      }
      for (int l = 4; l >= 1 && !failed; --l) {  // gradient of W_l += dz_l^T a_{l-1}; dz_{l-1} = (dz_l W_l) silu' + q
        float z[NC], v[NC], q[NC];
        if (l > 1) {
          load(p.Z[l - 2] + mat, z);
          load(p.Q[l - 2] + mat, q);
          if (l > 2)
            tc::cp_async_wait<1>();
          else
            tc::cp_async_wait<0>();
        }
        ready();
        if (t == 0) {
          if (l > 1) {
            product<false, true, 128>(tmem + work, ta[1], wa + (l - 2) * kTileBytes, 8, false);
            product<true, true, 128>(tmem + (l - 2) * 128, ta[1], ta[l == 3 ? 2 : 0], RT, true);
          } else {
            narrow_product(ta[1], sm.x);
          }
          tc::mma_commit(bar);
        }
        done();
        if (failed) break;
        if (l == 1) {
          narrow_add();
          break;
        }
        if (l == 4) image_in(0, p.A[0] + img);
        tmem_load<NC>(my_lanes + work + c0, v);
#pragma unroll
        for (int k = 0; k < NC; ++k) v[k] = __fmaf_rn(v[k], silu_d(z[k]), q[k]);
        to_tile(1, v);
        sum_b[l - 2] += column_sum(v);
      }
      more = true;
      fence_before();
    }
    __syncthreads();
  }
  tc::cp_async_wait<0>();
  if (failed) {
    if (t == 0) atomicExch(p.err, 1);
  } else if (kTrain && more) {
    fence_after();
#pragma unroll 1
    for (int m = 0; m < 3; ++m) {  // W_{m+2}: this thread's unit, 32 inputs
      float v[32];
      tmem_load<32>(my_lanes + m * 128 + (warp >> 2) * 32, v);
      float* dst = p.G + p.off_w[m + 1] + tl * 128 + (warp >> 2) * 32;
#pragma unroll
      for (int k = 0; k < 32; k += 4)
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + k), "f"(v[k]), "f"(v[k + 1]), "f"(v[k + 2]),
                     "f"(v[k + 3])
                     : "memory");
    }
    if (lane % COPIES == 0) {
      const int c = c0 + lane / COPIES;
#pragma unroll
      for (int l = 0; l < 4; ++l) atomicAdd(p.G + p.off_b[l] + c, sum_b[l]);
      atomicAdd(p.G + p.off_w[4] + c, sum_w5);
    }
    if (t < ROWS) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum_b5 += __shfl_xor_sync(0xffffffffu, sum_b5, o);
      if (lane == 0) atomicAdd(p.G + p.off_b[4], sum_b5);
    }
  }
  block_end(tmem);
}

}  // namespace fused
}  // namespace fehmm
