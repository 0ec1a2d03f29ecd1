// The network's host code (unet.o) linked against a CUDA runtime of two make-believe devices that runs no
// kernel: it keeps each device's shared-memory opt-ins, and refuses a launch that needs more than the
// 48 KB every kernel has when the current device was not opted in for it.  A network on each device in turn
// goes through a training pass.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <utility>
#include <vector>

#include "dda.h"

namespace {
int device = 0, launches = 0, large = 0, refused = 0;
std::map<std::pair<int, const void*>, int> optin;
struct Config { dim3 grid, block; size_t smem; cudaStream_t st; } config;
CUresult encode(...) { return CUDA_SUCCESS; }
}  // namespace

namespace dda { void add_launches(unsigned long long) {} }

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, struct CUstream_st* st) {
  config = {g, b, s, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = config.grid;
  *b = config.block;
  *s = config.smem;
  *(cudaStream_t*)st = config.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  ++launches;
  if (smem <= 48 * 1024) return cudaSuccess;
  ++large;
  const auto it = optin.find({device, (const void*)k});
  if (it == optin.end() || (size_t)it->second < smem) ++refused;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) optin[{device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(n ? n : 1, 1); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)&config; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *f = (void*)encode;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}

int main() {
  const int32_t ch[4] = {16, 32, 48, 64}, dims[3] = {32, 24, 16};
  const int B = 2, cin = 9, cout = 6;
  const size_t vox = (size_t)dims[0] * dims[1] * dims[2] * B;
  std::vector<float> x(vox * cin), y(vox * cout);
  for (int dev = 0; dev < 2; ++dev) {
    dda_unet* n = nullptr;
    const int before = refused, large0 = large;
    if (dda_unet_create(&n, dev, nullptr, cin, cout, ch, 1) != DDA_OK) return 2;
    device = 1 - dev;  // every entry point has to select its own device
    if (dda_unet_forward_train(n, x.data(), y.data(), B, dims) != DDA_OK) return 2;
    if (dda_unet_backward(n, y.data(), B, dims) != DDA_OK) return 2;
    if (large == large0) return 2;  // the test has to reach such launches
    std::printf("device %d: %d launches above 48 KB, %d refused\n", dev, large - large0, refused - before);
    dda_unet_destroy(n);
  }
  return refused ? 1 : 0;
}
