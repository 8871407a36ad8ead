// Energy-surrogate MLP on BF16 tensor cores (the learned part of the workload; the paper has
// no counterpart).  x in R^6 -> 4 hidden layers of 128 SiLU units -> scalar y.
//   z1 = W1 x + b1, a_l = silu(z_l), z_{l+1} = W_{l+1} a_l + b_{l+1}, y = w5 . a4 + b5
// Provided: forward, input gradient dy/dx (reverse mode), input Hessian (forward mode over the
// reverse pass, the 6 input directions batched as extra rows), the Sobolev training loss
// L = 1/2 sum_b [cy (y_b - ty_b)^2 + cg |dy/dx_b - tg_b|^2] with its exact parameter gradient
// (reverse mode through both the forward and the input-gradient pass), and a fused AdamW step
// on FP32 master weights that refreshes the BF16 copies.
//
// One launch takes a tile of samples through the whole network (mlp_kernels.cuh): BF16 operands in shared
// memory, tcgen05 products with FP32 accumulators in tensor memory.  BF16 rounding happens exactly where an
// operand of a product is stored.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <vector>

#include "fehmm.h"

namespace fehmm {
namespace {

using bf16 = __nv_bfloat16;

constexpr int W = 128;   // hidden width
constexpr int NIN = 6;   // inputs
constexpr int NINP = 8;  // inputs padded to a 16-byte row
// packed FP32 parameter layout
constexpr int OFF_W1 = 0;                     // [128][8]
constexpr int OFF_B1 = OFF_W1 + W * NINP;     // [128]
constexpr int OFF_W2 = OFF_B1 + W;            // [128][128]
constexpr int OFF_B2 = OFF_W2 + W * W;
constexpr int OFF_W3 = OFF_B2 + W;
constexpr int OFF_B3 = OFF_W3 + W * W;
constexpr int OFF_W4 = OFF_B3 + W;
constexpr int OFF_B4 = OFF_W4 + W * W;
constexpr int OFF_W5 = OFF_B4 + W;            // [128]
constexpr int OFF_B5 = OFF_W5 + W;            // [1]
constexpr int N_PARAMS = OFF_B5 + 4;          // padded

__host__ __device__ constexpr int off_W(int l) { return l == 1 ? OFF_W1 : l == 2 ? OFF_W2 : l == 3 ? OFF_W3 : OFF_W4; }
__host__ __device__ constexpr int off_b(int l) { return l == 1 ? OFF_B1 : l == 2 ? OFF_B2 : l == 3 ? OFF_B3 : OFF_B4; }

// --------------------------------------------------------------- elementwise
__device__ __forceinline__ float sig(float z) { return 1.f / (1.f + __expf(-z)); }
__device__ __forceinline__ float silu_f(float z) { return z * sig(z); }
__device__ __forceinline__ float silu_d(float z) {
  const float s = sig(z);
  return s * (1.f + z * (1.f - s));
}
__device__ __forceinline__ float silu_dd(float z) {
  const float s = sig(z);
  return s * (1.f - s) * (2.f + z * (1.f - 2.f * s));
}

#define GRID_STRIDE(i, n) for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)(n); i += (size_t)gridDim.x * blockDim.x)

// ------------------------------------------------------------ parameters
// bf16 copies of parameter i: row-major [out][in] in Wb, and W1^T padded [8][128]
__device__ __forceinline__ void refresh_bf16(int i, float v, bf16* Wb, bf16* W1T) {
  const bf16 b = __float2bfloat16(v);
  Wb[i] = b;
  if (i < OFF_B1) W1T[(i % NINP) * W + i / NINP] = b;
}

__global__ void refresh_kernel(const float* P, bf16* Wb, bf16* W1T) {
  GRID_STRIDE(i, N_PARAMS) refresh_bf16((int)i, P[i], Wb, W1T);
}

__global__ void zero_kernel(float* G, float* loss) {
  GRID_STRIDE(i, N_PARAMS) G[i] = 0.f;
  if (blockIdx.x == 0 && threadIdx.x == 0) *loss = 0.f;
}

// AdamW (decoupled weight decay on weight matrices only) and the bf16 copies of the new values, in one pass
// (one launch in place of six); padded input columns of W1 stay zero
__global__ void adamw_kernel(float* P, const float* G, float* m, float* v, int n, float lr, float b1, float b2,
                             float eps, float wd, float bc1, float bc2, bf16* Wb, bf16* W1T) {
  GRID_STRIDE(i, n) {
    const int ii = (int)i;
    if (ii < OFF_B1 && (ii % NINP) >= NIN) continue;
    if (ii >= OFF_B5 + 1) continue;
    const bool is_weight = (ii < OFF_B1) || (ii >= OFF_W2 && ii < OFF_B2) || (ii >= OFF_W3 && ii < OFF_B3) ||
                           (ii >= OFF_W4 && ii < OFF_B4) || (ii >= OFF_W5 && ii < OFF_B5);
    const float g = G[i];
    const float mm = b1 * m[i] + (1.f - b1) * g;
    const float vv = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mm;
    v[i] = vv;
    float p = P[i];
    if (is_weight) p -= lr * wd * p;
    p -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
    P[i] = p;
    refresh_bf16(ii, p, Wb, W1T);
  }
}

}  // namespace
}  // namespace fehmm

#include "mlp_kernels.cuh"

using namespace fehmm;

struct fehmm_mlp {
  int max_batch = 0;
  float* P = nullptr;   // FP32 masters [N_PARAMS]
  float* G = nullptr;   // gradient
  float* m = nullptr;
  float* v = nullptr;
  bf16* Wb = nullptr;   // bf16 copy of P (row-major weights)
  bf16* W1T = nullptr;  // W1^T [8][128]
  float* loss = nullptr;
  int num_sms = 0;
  // workspace of the whole-network kernels, [tiles of 128 samples][128 * 128] each (mlp_kernels.cuh)
  float* Z[4] = {};
  float* C[3] = {};
  float* Q[3] = {};
  bf16* A[3] = {};
  bf16* D[3] = {};
  int step = 0;
  int* err = nullptr;     // set by a kernel whose mbarrier wait ran out
  std::vector<void*> allocs;
  long long launches = 0;
};

namespace {

template <typename T>
int alloc(fehmm_mlp* m, T*& p, size_t count) {
  void* q = nullptr;
  if (cudaMalloc(&q, sizeof(T) * count) != cudaSuccess) {
    cudaGetLastError();
    return FEHMM_ERR_OOM;
  }
  m->allocs.push_back(q);
  p = static_cast<T*>(q);
  return FEHMM_OK;
}

int blocks_for(size_t n) {
  size_t b = (n + 255) / 256;
  if (b > 4096) b = 4096;
  return (int)(b ? b : 1);
}

void refresh(fehmm_mlp* m, cudaStream_t s) {
  refresh_kernel<<<blocks_for(N_PARAMS), 256, 0, s>>>(m->P, m->Wb, m->W1T);
  m->launches += 1;
}

fused::Net net(const fehmm_mlp* m) {
  fused::Net n{};
  n.W1 = m->Wb + OFF_W1;
  for (int l = 2; l <= 4; ++l) n.W[l - 2] = m->Wb + off_W(l);
  n.W1T = m->W1T;
  n.w5 = m->Wb + OFF_W5;
  for (int l = 1; l <= 4; ++l) n.b[l - 1] = m->P + off_b(l);
  n.b5 = m->P + OFF_B5;
  return n;
}

// Persistent launch of a whole-network kernel: at most one block per SM (its weights and tiles fill the
// shared memory, its accumulators the tensor memory).
template <typename Kernel, typename... Args>
int launch(fehmm_mlp* m, Kernel kernel, int tiles, int threads, size_t smem, cudaStream_t s, Args... args) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return FEHMM_ERR_CUDA;
  }
  kernel<<<tiles < m->num_sms ? tiles : m->num_sms, threads, smem, s>>>(args...);
  m->launches += 1;
  return cudaGetLastError() == cudaSuccess ? FEHMM_OK : FEHMM_ERR_CUDA;
}

// The smallest tile that still needs one round of blocks: a step's latency grows with the tile's samples.
template <bool kTrain>
int launch_grad(fehmm_mlp* m, const fused::GradArgs& a, cudaStream_t s) {
  const size_t smem = sizeof(fused::GradSmem);
  if (a.B <= 32 * m->num_sms) return launch(m, fused::grad_kernel<kTrain, 32>, (a.B + 31) / 32, fused::kGradThreads, smem, s, a);
  if (a.B <= 64 * m->num_sms) return launch(m, fused::grad_kernel<kTrain, 64>, (a.B + 63) / 64, fused::kGradThreads, smem, s, a);
  return launch(m, fused::grad_kernel<kTrain, 128>, (a.B + 127) / 128, fused::kGradThreads, smem, s, a);
}

fused::GradArgs grad_args(fehmm_mlp* m, const float* x, int B) {
  fused::GradArgs a{};
  a.net = net(m);
  a.x = x;
  a.B = B;
  for (int l = 0; l < 4; ++l) a.Z[l] = m->Z[l];
  for (int l = 0; l < 3; ++l) {
    a.C[l] = m->C[l];
    a.Q[l] = m->Q[l];
    a.A[l] = reinterpret_cast<uint8_t*>(m->A[l]);
    a.D[l] = reinterpret_cast<uint8_t*>(m->D[l]);
  }
  a.err = m->err;
  return a;
}

}  // namespace

extern "C" {

int fehmm_mlp_num_params(void) { return N_PARAMS; }

int fehmm_mlp_create(fehmm_mlp** out, int max_batch) {
  if (!out || max_batch <= 0) return FEHMM_ERR_ARG;
  *out = nullptr;
  fehmm_mlp* m = new (std::nothrow) fehmm_mlp();
  if (!m) return FEHMM_ERR_OOM;
  m->max_batch = max_batch;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    delete m;
    return FEHMM_ERR_CUDA;
  }
  const size_t BW = ((size_t)max_batch + fused::kGradMaxRows - 1) / fused::kGradMaxRows * fused::kGradMaxRows * W;
  int rc = FEHMM_OK;
  rc |= alloc(m, m->P, N_PARAMS);
  rc |= alloc(m, m->G, N_PARAMS);
  rc |= alloc(m, m->m, N_PARAMS);
  rc |= alloc(m, m->v, N_PARAMS);
  rc |= alloc(m, m->Wb, N_PARAMS);
  rc |= alloc(m, m->W1T, (size_t)NINP * W);
  rc |= alloc(m, m->loss, 4);
  for (int l = 0; l < 4; ++l) rc |= alloc(m, m->Z[l], BW);
  for (int l = 0; l < 3; ++l) {
    rc |= alloc(m, m->C[l], BW);
    rc |= alloc(m, m->Q[l], BW);
    rc |= alloc(m, m->A[l], BW);
    rc |= alloc(m, m->D[l], BW);
  }
  rc |= alloc(m, m->err, 1);
  if (rc != FEHMM_OK) {
    for (void* p : m->allocs) cudaFree(p);
    delete m;
    return FEHMM_ERR_OOM;
  }
  cudaMemset(m->P, 0, sizeof(float) * N_PARAMS);
  cudaMemset(m->err, 0, sizeof(int));
  cudaMemset(m->m, 0, sizeof(float) * N_PARAMS);
  cudaMemset(m->v, 0, sizeof(float) * N_PARAMS);
  *out = m;
  return FEHMM_OK;
}

int fehmm_mlp_destroy(fehmm_mlp* m) {
  if (!m) return FEHMM_ERR_ARG;
  for (void* p : m->allocs) cudaFree(p);
  delete m;
  return FEHMM_OK;
}

int fehmm_mlp_set_params(fehmm_mlp* m, const float* host_params) {
  if (!m || !host_params) return FEHMM_ERR_ARG;
  if (cudaMemcpy(m->P, host_params, sizeof(float) * N_PARAMS, cudaMemcpyHostToDevice) != cudaSuccess)
    return FEHMM_ERR_CUDA;
  cudaMemset(m->m, 0, sizeof(float) * N_PARAMS);
  cudaMemset(m->v, 0, sizeof(float) * N_PARAMS);
  m->step = 0;
  refresh(m, 0);
  return cudaDeviceSynchronize() == cudaSuccess ? FEHMM_OK : FEHMM_ERR_CUDA;
}

int fehmm_mlp_get_params(fehmm_mlp* m, float* host_params, float* host_grad) {
  if (!m || (!host_params && !host_grad)) return FEHMM_ERR_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return FEHMM_ERR_CUDA;
  if (host_params && cudaMemcpy(host_params, m->P, sizeof(float) * N_PARAMS, cudaMemcpyDeviceToHost) != cudaSuccess)
    return FEHMM_ERR_CUDA;
  if (host_grad && cudaMemcpy(host_grad, m->G, sizeof(float) * N_PARAMS, cudaMemcpyDeviceToHost) != cudaSuccess)
    return FEHMM_ERR_CUDA;
  return FEHMM_OK;
}

int fehmm_mlp_eval(fehmm_mlp* m, const float* x, int B, float* y, float* g, float* H, void* stream) {
  if (!m || !x || B <= 0 || B > m->max_batch) return FEHMM_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (H)
    return launch(m, fused::eval_hess_kernel, (B + fused::kEvalSamples - 1) / fused::kEvalSamples, fused::kEvalThreads,
                  sizeof(fused::EvalSmem), s, net(m), x, B, y, g, H, m->err);
  fused::GradArgs a = grad_args(m, x, B);
  a.y = y;
  a.g = g;
  return launch_grad<false>(m, a, s);
}

int fehmm_mlp_loss_grad(fehmm_mlp* m, const float* x, const float* ty, const float* tg, int B, float cy, float cg,
                        float* loss_out, void* stream) {
  if (!m || !x || !ty || !tg || B <= 0 || B > m->max_batch) return FEHMM_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  fused::GradArgs a = grad_args(m, x, B);
  a.ty = ty;
  a.tg = tg;
  a.cy = cy;
  a.cg = cg;
  a.G = m->G;
  a.loss = loss_out ? loss_out : m->loss;
  for (int l = 1; l <= 4; ++l) {
    a.off_w[l - 1] = off_W(l);
    a.off_b[l - 1] = off_b(l);
  }
  a.off_w[4] = OFF_W5;
  a.off_b[4] = OFF_B5;
  zero_kernel<<<blocks_for(N_PARAMS), 256, 0, s>>>(a.G, a.loss);
  m->launches += 1;
  return launch_grad<true>(m, a, s);
}

int fehmm_mlp_adamw(fehmm_mlp* m, float lr, float beta1, float beta2, float eps, float weight_decay, void* stream) {
  if (!m || !(lr > 0)) return FEHMM_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  m->step += 1;
  const float bc1 = 1.f - powf(beta1, (float)m->step), bc2 = 1.f - powf(beta2, (float)m->step);
  adamw_kernel<<<blocks_for(N_PARAMS), 256, 0, s>>>(m->P, m->G, m->m, m->v, N_PARAMS, lr, beta1, beta2, eps,
                                                   weight_decay, bc1, bc2, m->Wb, m->W1T);
  m->launches += 1;
  return cudaGetLastError() == cudaSuccess ? FEHMM_OK : FEHMM_ERR_CUDA;
}

long long fehmm_mlp_launch_count(const fehmm_mlp* m) { return m ? m->launches : -1; }

int fehmm_mlp_check(fehmm_mlp* m, int* flag) {
  if (!m || !flag) return FEHMM_ERR_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return FEHMM_ERR_CUDA;
  if (cudaMemcpy(flag, m->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return FEHMM_ERR_CUDA;
  if (*flag != 0 && cudaMemset(m->err, 0, sizeof(int)) != cudaSuccess) return FEHMM_ERR_CUDA;
  return FEHMM_OK;
}

int fehmm_mlp_grad_buffer(fehmm_mlp* m, float** dev_ptr, int* n) {
  if (!m || !dev_ptr) return FEHMM_ERR_ARG;
  *dev_ptr = m->G;
  if (n) *n = N_PARAMS;
  return FEHMM_OK;
}

// Surrogate file: magic, format version, parameter count, the packed FP32 parameters, then the
// fehmm_surrogate_params fields as little-endian doubles in declaration order (every double of
// the struct is written, so a load reproduces the evaluation exactly).
namespace {
constexpr char kMagic[8] = {'F', 'E', 'H', 'M', 'M', 'S', 'U', 'R'};
constexpr int32_t kFormat = 2;  // 2: with the polynomial part
constexpr size_t kSpDoubles = sizeof(fehmm_surrogate_params) / sizeof(double);
static_assert(sizeof(fehmm_surrogate_params) == kSpDoubles * sizeof(double), "surrogate params are all doubles");
}  // namespace

int fehmm_surrogate_save(fehmm_mlp* m, const fehmm_surrogate_params* sp, const char* path) {
  if (!m || !sp || !path) return FEHMM_ERR_ARG;
  std::vector<float> params(N_PARAMS);
  const int rc = fehmm_mlp_get_params(m, params.data(), nullptr);
  if (rc != FEHMM_OK) return rc;
  FILE* f = fopen(path, "wb");
  if (!f) return FEHMM_ERR_ARG;
  const int32_t np = N_PARAMS, nsp = (int32_t)kSpDoubles;
  bool ok = fwrite(kMagic, 1, 8, f) == 8 && fwrite(&kFormat, sizeof(kFormat), 1, f) == 1 &&
            fwrite(&np, sizeof(np), 1, f) == 1 && fwrite(&nsp, sizeof(nsp), 1, f) == 1 &&
            fwrite(params.data(), sizeof(float), N_PARAMS, f) == (size_t)N_PARAMS &&
            fwrite(sp, sizeof(double), kSpDoubles, f) == kSpDoubles;
  ok = (fclose(f) == 0) && ok;
  return ok ? FEHMM_OK : FEHMM_ERR_ARG;
}

int fehmm_surrogate_load(fehmm_mlp* m, fehmm_surrogate_params* sp, const char* path) {
  if (!m || !sp || !path) return FEHMM_ERR_ARG;
  FILE* f = fopen(path, "rb");
  if (!f) return FEHMM_ERR_ARG;
  char magic[8];
  int32_t fmt = 0, np = 0, nsp = 0;
  std::vector<float> params(N_PARAMS);
  fehmm_surrogate_params tmp;
  bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, kMagic, 8) == 0 && fread(&fmt, sizeof(fmt), 1, f) == 1 &&
            fmt == kFormat && fread(&np, sizeof(np), 1, f) == 1 && np == N_PARAMS &&
            fread(&nsp, sizeof(nsp), 1, f) == 1 && nsp == (int32_t)kSpDoubles &&
            fread(params.data(), sizeof(float), N_PARAMS, f) == (size_t)N_PARAMS &&
            fread(&tmp, sizeof(double), kSpDoubles, f) == kSpDoubles;
  fclose(f);
  if (!ok) return FEHMM_ERR_ARG;
  const int rc = fehmm_mlp_set_params(m, params.data());
  if (rc != FEHMM_OK) return rc;
  *sp = tmp;
  return FEHMM_OK;
}

}  // extern "C"
