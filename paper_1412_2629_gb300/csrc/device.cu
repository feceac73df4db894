// What belongs to a device and not to the process: its limits, and the kernels that have been
// allowed more dynamic shared memory than the 48 KB every kernel may use.  A process may hold
// contexts on several devices and call them from several threads.  Both are looked up in every
// launch, so the path after the first takes no lock (with a mutex and maps: 567 us for 32 half-sweeps
// on 8^4, 563 without).
#include "dd_kernels.hpp"

namespace dd {

const DeviceInfo& device_info() {
  static const DeviceInfo unknown;
  static std::atomic<const DeviceInfo*> known[MAX_DEVICES];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return unknown;
  if (const DeviceInfo* d = known[dev].load(std::memory_order_acquire)) return *d;
  int sms = 0, block = 0, sm = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess || sms < 1)
    return unknown;
  DeviceInfo* mine = new DeviceInfo;
  mine->id = dev;
  mine->sms = sms;
  mine->smem_block = block;
  mine->smem_sm = sm;
  const DeviceInfo* first = nullptr;
  if (known[dev].compare_exchange_strong(first, mine, std::memory_order_acq_rel)) return *mine;
  delete mine;   // another thread was first
  return *first;
}

void allow_smem(SmemAllowed& done, const DeviceInfo& dev, const void* kernel, size_t bytes) {
  const unsigned long long bit = dev.id < 0 ? 0 : 1ull << dev.id;
  if (done.devices.load(std::memory_order_acquire) & bit) return;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess)
    done.devices.fetch_or(bit, std::memory_order_acq_rel);
}

}  // namespace dd
