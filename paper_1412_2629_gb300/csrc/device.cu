// What belongs to a device and not to the process: its limits, and the kernels that have been
// allowed more dynamic shared memory than the 48 KB every kernel may use.  A process may hold
// contexts on several devices and call them from several threads, so both are kept per device
// and under a mutex (tens of nanoseconds beside a launch).
#include <map>
#include <mutex>

#include "dd_kernels.hpp"

namespace dd {

static std::mutex g_mutex;

DeviceInfo device_info() {
  static std::map<int, DeviceInfo> known;
  int dev = 0;
  DeviceInfo d;
  if (cudaGetDevice(&dev) != cudaSuccess) return d;
  std::lock_guard<std::mutex> lock(g_mutex);
  auto it = known.find(dev);
  if (it != known.end()) return it->second;
  int sms = 0, block = 0, sm = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess || sms < 1)
    return d;
  d.sms = sms;
  d.smem_block = block;
  d.smem_sm = sm;
  known[dev] = d;
  return d;
}

void allow_smem(const void* kernel, size_t bytes) {
  static std::map<std::pair<int, const void*>, size_t> allowed;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  std::lock_guard<std::mutex> lock(g_mutex);
  size_t& have = allowed[{dev, kernel}];
  if (have >= bytes) return;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess) have = bytes;
}

}  // namespace dd
