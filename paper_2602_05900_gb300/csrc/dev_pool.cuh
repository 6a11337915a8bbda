// Device memory of the library's objects and of its stand-alone calls.
//
// A context allocates some twenty buffers and frees them when it is destroyed;
// cudaMalloc and cudaFree map and unmap memory and synchronise the device
// (0.3 ms for a D = 8 context, 2 ms for a BF16XS D = 32 one, 12 ms for a batch of
// 24; 0.4 ms of a 0.48 ms hotrg_dgemm_emu call).  Buffers come instead from one
// CUDA memory pool per device, created on first use, which keeps up to
// kPoolKeep bytes of freed memory mapped and gives the rest back to the
// device (0.1 ms for a context of any size that fits).  The driver takes idle pool
// memory back by itself before an allocation fails: with 273.2 GiB free and 2.6 GiB
// idle, cudaMalloc of 273.7 GiB succeeds.  The pool's own locking
// and stream ordering make it safe with several threads and streams.  Buffers of
// kPoolBlock bytes or more -- contexts the pool would not keep -- are allocated and
// freed directly: through the pool they took longer (D = 64: 13.6 ms against 8.6).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <vector>

namespace hotrg {

constexpr unsigned long long kPoolKeep = 4ull << 30;   // idle bytes a device's pool may hold
constexpr std::size_t kPoolBlock = std::size_t(1) << 30;   // buffers from here on bypass it

// Allocations of one owner on the device that is current when it is made.  The
// memory may be used on any stream once ready() has returned; free_all() is called
// when no work that uses it is in flight.
class DeviceBuffers {
 public:
  DeviceBuffers() = default;
  DeviceBuffers(const DeviceBuffers &) = delete;
  DeviceBuffers &operator=(const DeviceBuffers &) = delete;
  ~DeviceBuffers() { free_all(); }
  cudaError_t alloc(void **p, std::size_t bytes);   // 256-byte aligned
  cudaError_t ready();
  void free_all();

 private:
  int dev_ = -1;
  std::vector<void *> pooled_, direct_;
};

// One buffer of a stand-alone call, ordered on the call's own stream.
class StreamBuffer {
 public:
  explicit StreamBuffer(cudaStream_t s) : s_(s) {}
  StreamBuffer(const StreamBuffer &) = delete;
  StreamBuffer &operator=(const StreamBuffer &) = delete;
  ~StreamBuffer();
  cudaError_t alloc(std::size_t bytes);
  char *data() const { return static_cast<char *>(p_); }

 private:
  cudaStream_t s_;
  void *p_ = nullptr;
  bool pooled_ = false;
};

}  // namespace hotrg
