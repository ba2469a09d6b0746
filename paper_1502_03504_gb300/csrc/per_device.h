// What belongs to a device and is found once for each: the number of its SMs,
// a kernel's shared-memory limit and its resident blocks.  A program may use
// several devices, and several threads may come first (all find the same).
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace lope {

class PerDevice {
 public:
  // *value: what find(value) gave on the current device, greater than 0.
  template <class F> cudaError_t get(int* value, F&& find) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::atomic<int>* slot = dev >= 0 && dev < kDevices ? &found_[dev] : nullptr;
    if (slot && (*value = slot->load(std::memory_order_acquire)) > 0) return cudaSuccess;
    if ((e = find(value)) == cudaSuccess && slot) slot->store(*value, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 64;  // devices past these are asked each time
  std::atomic<int> found_[kDevices] = {};
};

// SMs of the current device (1 without a device).
inline int device_sms() {
  static PerDevice sms;
  int n = 0;
  const cudaError_t e = sms.get(&n, [](int* v) {
    int dev = 0;
    cudaGetDevice(&dev);
    return cudaDeviceGetAttribute(v, cudaDevAttrMultiProcessorCount, dev);
  });
  return e == cudaSuccess && n > 0 ? n : 1;
}

// Opt a kernel in to `smem` bytes of dynamic shared memory and count its resident
// blocks per SM (at least 1), once per device; `memo` belongs to the kernel.
template <class Kernel>
cudaError_t blocks_per_sm(PerDevice& memo, Kernel kern, int threads, size_t smem, int* blocks) {
  return memo.get(blocks, [&](int* v) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    int n = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem);
    *v = n > 0 ? n : 1;
    return e;
  });
}

}  // namespace lope
