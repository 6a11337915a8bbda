// What a launch looks up once per device: a kernel's shared-memory limit and the
// number of SMs.  Both belong to a device, not to the process, and host threads
// that step the cut groups of a batch side by side ask for them at the same time.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace hotrg {

constexpr int kAttrDevices = 64;   // devices beyond these are asked at every launch

// One static object per kernel: raises its dynamic shared-memory limit on the
// current device the first time it is launched there.
class SmemLimit {
 public:
  cudaError_t raise(const void *kernel, int bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < kAttrDevices ? 1ull << dev : 0;
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<unsigned long long> done_{0};
};

// SMs of the current device (a B200's 148 if it cannot be asked)
inline int sm_count() {
  static std::atomic<int> known[kAttrDevices];
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (dev < kAttrDevices && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 148;
  if (dev < kAttrDevices) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

}  // namespace hotrg
