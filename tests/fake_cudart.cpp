// Stand-ins for the CUDA runtime (an executable's definitions come before the library's).  Device
// memory is host memory, kernels do not run, and a launch is refused, as the runtime does, when
// its dynamic shared memory exceeds 48 KB and what the kernel was allowed on the current device.
#include "fake_cudart.hpp"

#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>

namespace {
const int SMS[2] = {152, 100};
thread_local int t_dev = 0;
thread_local cudaError_t t_last = cudaSuccess;
thread_local std::vector<unsigned> t_grids;   // grid sizes of this thread's launches
std::mutex g_mu;
std::map<std::pair<int, const void*>, size_t> g_allowed;
int g_bad = 0;
bool g_maps = true;
}  // namespace

void set_device(int dev) { t_dev = dev; }
int multiprocessors(int dev) { return SMS[dev]; }
std::vector<unsigned>& grids() { return t_grids; }
bool& tensor_maps() { return g_maps; }
void finding(const std::string& what) {
  std::lock_guard<std::mutex> lock(g_mu);
  ++g_bad;
  printf("device %d: %s\n", t_dev, what.c_str());
}
int findings() { return g_bad; }

namespace {
cudaError_t launch(const void* f, dim3 grid, size_t smem) {
  {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_allowed.find({t_dev, f});
    if (smem <= (it == g_allowed.end() ? 48u * 1024u : it->second)) {
      t_grids.push_back(grid.x);
      return cudaSuccess;
    }
  }
  finding("launch with " + std::to_string(smem) + " bytes of dynamic shared memory refused");
  return t_last = cudaErrorInvalidValue;
}
CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, g, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_allowed[{t_dev, f}] = (size_t)v;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = t_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int dev) {
  *v = a == cudaDevAttrMultiProcessorCount ? SMS[dev] : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 233472;
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { const cudaError_t e = t_last; t_last = cudaSuccess; return e; }
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = g_maps ? (void*)encode : nullptr;
  *r = g_maps ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
}
