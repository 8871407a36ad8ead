// A stand-in for the CUDA runtime on the CPU, for tests of the library's host code: device memory is host memory,
// kernels are not run, and one call can be made to fail.  fake_fail(k): the k-th call from now of those that can fail
// for want of memory or resources returns an error (0: none does); it returns the number of such calls since the last
// fake_fail.  fake_blocks: allocations not yet freed.  fake_watch(a): remember the int that is argument a of the launches
// that follow; it returns the last one.
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <set>

static int g_fail = 0, g_calls = 0, g_arg = -1, g_seen = 0;
static std::set<void*> g_blocks;
static bool fails() { return ++g_calls == g_fail; }

extern "C" {
int fake_fail(int k) {
  const int n = g_calls;
  g_fail = k;
  g_calls = 0;
  return n;
}
int fake_watch(int arg) {
  const int seen = g_seen;
  g_arg = arg;
  return seen;
}
int fake_blocks() { return (int)g_blocks.size(); }

cudaError_t cudaMalloc(void** p, size_t n) {
  *p = nullptr;
  if (fails()) return cudaErrorMemoryAllocation;
  *p = calloc(1, n ? n : 1);
  g_blocks.insert(*p);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  if (!g_blocks.erase(p)) abort();  // not allocated, or freed twice
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  if (fails()) return cudaErrorInvalidValue;
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  if (fails()) return cudaErrorInvalidValue;
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  if (fails()) return cudaErrorMemoryAllocation;
  *e = (cudaEvent_t)e;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  if (fails()) return cudaErrorMemoryAllocation;
  *s = (cudaStream_t)s;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return fails() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 4;  // SMs
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorUnknown; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
// what nvcc's launch syntax and registration refer to
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void** args, size_t, cudaStream_t) {
  if (g_arg >= 0) g_seen = *(int*)args[g_arg];
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
