// Kernel launches with programmatic dependent launch.
//
// The eigensolver, the exact-slice products and iTEBD are chains of hundreds of
// kernels of a few microseconds; started one after the other, each waits for the
// last block of the one before to drain and then for its own launch.  Launched
// with `launch_pdl`, a kernel may start while its predecessor still runs, and
// waits inside (pdl_enter, before any access to global memory) until that one
// has completed and its writes are visible.
//
// Every kernel launched this way calls pdl_enter (or pdl_trigger and pdl_wait) in
// every block that touches global memory and in at least one block: its
// completion then implies its predecessor's, and so on down the stream.
// Measured, without and with it: TF32 D = 32 job 58.9 and 51.3 ms, D = 13 chain 8.8
// and 6.6 ms, one iTEBD chain at D_b = 30 17.5 and 15.1 ms.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace hotrg {

// lets the next kernel of the stream start (it waits for this one in pdl_wait)
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// waits until the kernel before this one has completed (no-op in a plain launch)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// In this order: triggered before the wait, the kernels of a chain would pile up
// behind a long one and hold the SMs' shared memory while they wait.
__device__ __forceinline__ void pdl_enter() {
  pdl_wait();
  pdl_trigger();
}

// Whether this host thread's launches may start early.  The threads that step the
// cut groups of a batch side by side turn it off: blocks that wait for their own
// group's kernel would hold SMs that another group's could use (24-instance
// sweep: 160-166 ms with, 154 ms without).
inline bool &pdl_allowed() {
  thread_local bool on = true;
  return on;
}

inline cudaLaunchAttribute pdl_attribute() {
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = pdl_allowed() ? 1 : 0;
  return a;
}

template <class T>
struct same_type {
  using type = T;
};

template <class... P>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, std::size_t smem, cudaStream_t s,
                   typename same_type<P>::type... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr = pdl_attribute();
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace hotrg
