// Whole-network kernels of the surrogate MLP: one launch takes a tile of samples through every layer, with
// the three 128 x 128 weight matrices (BF16, 96 KB) resident in shared memory, the operand of each product
// built there by the epilogue of the one before, and the FP32 products in tensor memory.
//
// The layer-by-layer form (a tcgen05 product, a stored FP32 matrix, an elementwise launch, ...) was bound by
// launches and by the traffic between them: 20 launches and 1.26 ms for value, input gradient and Hessian of
// 32768 points, 42 launches and 0.50 ms for a training step of 4096 samples, at 1 % tensor-pipe activity.
//
// Products: 128 x 128 x 128 as eight tcgen05.mma of K = 16 in ascending order, the same instruction and
// order as layer by layer, so that every activation is bit for bit what the layer-by-layer form gave; the
// 6-wide input layer (K or N = 8) runs on mma.sync, K ascending.
//
// Shared-memory operands are in 8 x 8 core matrices of 128 bytes: block (r / 8, c / 8) of a 128 x 128 matrix
// at (r / 8) * 2048 + (c / 8) * 128.  With rows as M or N and columns as K that is the K-major layout (128
// bytes from one K group to the next, 2048 from one row group to the next); with columns as M or N and rows
// as K it is the M/N-major one (the strides change places), so one copy of a weight matrix serves a layer's
// forward and backward product, and one copy of an activation serves the next layer and the weight gradient.
//
// Every mbarrier wait is bounded (tc::mbar_wait); one that runs out sets *err, and the block frees its
// tensor memory and returns.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fehmm {
namespace tc {

constexpr long long kWaitCycles = 1ll << 32;

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9, 10-12 = 1),
// both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// 16 bytes global -> shared, the bytes past src_bytes (0 or 16) zero-filled
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > kWaitCycles) return false;
  }
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

}  // namespace tc

namespace fused {

using bf16 = __nv_bfloat16;

constexpr int kTileBytes = 128 * 128 * 2;
constexpr uint32_t kRowGroup = 2048, kColGroup = 128;  // bytes between 8-row groups and between 8-column groups

__device__ __forceinline__ uint32_t core_off(int r, int c) {  // byte offset of element (r, c)
  return (uint32_t)(r >> 3) * kRowGroup + (uint32_t)(c >> 3) * kColGroup + (uint32_t)(r & 7) * 16 + (uint32_t)(c & 7) * 2;
}

// Descriptor of an operand whose K groups are lbo bytes apart and whose M/N groups are sbo bytes apart.
__device__ __forceinline__ uint64_t desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}

// D (128 x N FP32 at TMEM address d) (+)= A B over K = 16 * steps.  AT / BT: the operand's K runs over the
// rows of its matrix (M/N-major), else over its columns.
template <bool AT, bool BT, int N>
__device__ __forceinline__ void product(uint32_t d, uint32_t a, uint32_t b, int steps, bool accumulate) {
  constexpr uint32_t idesc = tc::idesc_bf16_f32(128, N) | (AT ? 1u << 15 : 0u) | (BT ? 1u << 16 : 0u);
#pragma unroll 1
  for (int k = 0; k < steps; ++k) {
    const uint64_t da = AT ? desc(a + k * 2 * kRowGroup, kRowGroup, kColGroup) : desc(a + k * 2 * kColGroup, kColGroup, kRowGroup);
    const uint64_t db = BT ? desc(b + k * 2 * kRowGroup, kRowGroup, kColGroup) : desc(b + k * 2 * kColGroup, kColGroup, kRowGroup);
    tc::mma_bf16(d, da, db, idesc, (accumulate || k > 0) ? 1u : 0u);
  }
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// N columns of this warp's 32 TMEM lanes (thread = lane)
template <int N>
__device__ __forceinline__ void tmem_load(uint32_t addr, float (&v)[N]) {
  static_assert(N == 8 || N == 16 || N == 32, "columns of one load");
  uint32_t* u = reinterpret_cast<uint32_t*>(v);
  if constexpr (N == 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7])
                 : "r"(addr));
  } else if constexpr (N == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
          "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
        : "r"(addr));
  } else {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
          "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]),
          "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]),
          "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
        : "r"(addr));
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 p(__float2bfloat16(lo), __float2bfloat16(hi));
  return *reinterpret_cast<uint32_t*>(&p);
}

// 8 values of row r, columns c .. c + 7 (c a multiple of 8) into a 128 x 128 BF16 tile
__device__ __forceinline__ void store8(uint8_t* tile, int r, int c, const float* v) {
  *reinterpret_cast<uint4*>(tile + core_off(r, c)) = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}

// the same of 4 values (c a multiple of 4)
__device__ __forceinline__ void store4(uint8_t* tile, int r, int c, const float* v) {
  *reinterpret_cast<uint2*>(tile + core_off(r, c)) = make_uint2(pack2(v[0], v[1]), pack2(v[2], v[3]));
}

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Rows 16 * tile16 .. + 15 of (128 x 128 BF16 tile) x W1 (K = 128, N = 8; w1t = W1^T [8][128]): d[0], d[1] at
// row lane / 4, columns 2 (lane % 4) + {0, 1}; d[2], d[3] eight rows below.
__device__ __forceinline__ void times_w1(const uint8_t* tile, int tile16, const bf16* w1t, float (&d)[4]) {
  const int lane = threadIdx.x & 31;
  d[0] = d[1] = d[2] = d[3] = 0.f;
  const uint32_t base = tc::smem_u32(tile) + core_off(16 * tile16 + (lane & 15), 8 * (lane >> 4));
  const bf16* b = w1t + (lane >> 2) * 128 + 2 * (lane & 3);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    uint32_t a[4];
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(base + k * 2 * kColGroup));
    mma_16816(d, a, *reinterpret_cast<const uint32_t*>(b + 16 * k), *reinterpret_cast<const uint32_t*>(b + 16 * k + 8));
  }
}

// 16 rows x 8 features (BF16 in shared memory: rows of 16 bytes, the upper eight `up` bytes behind the lower)
// times W1^T for units 8 nt .. 8 nt + 7: the input layer's product (K = 8, the upper half of the
// instruction's K is zero)
__device__ __forceinline__ void input_layer(const uint8_t* x, int up, const bf16* w1, int nt, float (&d)[4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  d[0] = d[1] = d[2] = d[3] = 0.f;
  const uint32_t a[4] = {*reinterpret_cast<const uint32_t*>(x + g * 16 + 4 * t),
                         *reinterpret_cast<const uint32_t*>(x + up + g * 16 + 4 * t), 0u, 0u};
  mma_16816(d, a, *reinterpret_cast<const uint32_t*>(w1 + (8 * nt + g) * 8 + 2 * t), 0u);
}

// W2..W4 (row-major [out][in] BF16 in global memory, ld 128) into three tiles
__device__ __forceinline__ void load_weights(uint8_t* tiles, const bf16* w2, const bf16* w3, const bf16* w4) {
  for (int e = threadIdx.x; e < 3 * 2048; e += blockDim.x) {
    const int m = e >> 11, r = (e >> 4) & 127, c = (e & 15) * 8;
    const bf16* w = (m == 0 ? w2 : m == 1 ? w3 : w4) + r * 128 + c;
    tc::cp_async16(tc::smem_u32(tiles + m * kTileBytes + core_off(r, c)), w, 16);
  }
  tc::cp_async_commit();
}

// Block set-up: one mbarrier, 512 columns of tensor memory.  Ends with a barrier; returns the TMEM address.
__device__ __forceinline__ uint32_t block_begin(uint64_t* bar, uint32_t* slot) {
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(bar));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  return *slot;
}

__device__ __forceinline__ void block_end(uint32_t tmem) {
  fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

}  // namespace fused
}  // namespace fehmm
