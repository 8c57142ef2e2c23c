// Values that belong to a device and are the same for the life of the process there: its SM count, the
// size of a persistent grid, a kernel's shared-memory limit.  A process may hold contexts on several
// devices and use them from several threads, so these are kept per device.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace chebmg {

constexpr int kMaxDevices = 64;   // devices beyond are asked at every use

// A value computed at its first use on each device; make() gives 0 where it could not (asked again at
// the next use).  Two threads may both compute it: make() has the same result and effect each time.
class PerDevice {
  std::atomic<int> v_[kMaxDevices] = {};

 public:
  template <typename F>
  int operator()(F&& make) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return make();
    int x = v_[dev].load(std::memory_order_acquire);
    if (x == 0) {
      x = make();
      v_[dev].store(x, std::memory_order_release);
    }
    return x;
  }
};

inline int device_attribute(cudaDeviceAttr attr) {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, attr, dev) != cudaSuccess) return 0;
  return v;
}
inline int sm_count() {   // at least 1
  static PerDevice sms;
  const int n = sms([] { return device_attribute(cudaDevAttrMultiProcessorCount); });
  return n > 0 ? n : 1;
}

// Lets kernel k take `bytes` of dynamic shared memory on the current device; `done` is the kernel's own.
// Blocks that stay below the 48 KB every kernel may take (8 KB left to static arrays) need nothing: small
// calls are bound by the host, and asking for the device costs it.
inline void allow_smem(PerDevice& done, const void* k, size_t bytes) {
  if (bytes <= 40 * 1024) return;
  done([=] {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess ? 1 : 0;
  });
}
// Blocks of kernel k that are resident on the current device at once (at least one per SM).
inline int resident_blocks(PerDevice& value, const void* k, int threads, size_t smem) {
  return value([=] {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
    return sm_count() * (per_sm > 0 ? per_sm : 1);
  });
}

}  // namespace chebmg
