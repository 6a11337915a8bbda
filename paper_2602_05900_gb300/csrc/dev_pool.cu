// Memory pools of the library (see dev_pool.cuh).
#include <mutex>

#include "dev_pool.cuh"

namespace hotrg {
namespace {

constexpr int kMaxDevices = 64;

struct Pool {
  bool tried = false;
  cudaMemPool_t pool = nullptr;    // null: the device has no pools, cudaMalloc is used
  cudaStream_t stream = nullptr;   // orders the allocations and frees of DeviceBuffers
};

Pool g_pools[kMaxDevices];
std::mutex g_mu;

// The device's pool, made on first use and kept until the process exits.
Pool *pool_of(int dev) {
  if (dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lk(g_mu);
  Pool &p = g_pools[dev];
  if (!p.tried) {
    p.tried = true;
    int has = 0;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    unsigned long long keep = kPoolKeep;
    if (cudaDeviceGetAttribute(&has, cudaDevAttrMemoryPoolsSupported, dev) != cudaSuccess || !has ||
        cudaStreamCreateWithFlags(&p.stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaMemPoolCreate(&p.pool, &props) != cudaSuccess ||
        cudaMemPoolSetAttribute(p.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      (void)cudaGetLastError();
      if (p.pool) cudaMemPoolDestroy(p.pool);
      if (p.stream) cudaStreamDestroy(p.stream);
      p.pool = nullptr;
      p.stream = nullptr;
    }
  }
  return p.pool ? &p : nullptr;
}

}  // namespace

cudaError_t DeviceBuffers::alloc(void **p, std::size_t bytes) {
  *p = nullptr;
  if (dev_ < 0) {
    const cudaError_t e = cudaGetDevice(&dev_);
    if (e != cudaSuccess) return e;
  }
  Pool *pl = bytes < kPoolBlock ? pool_of(dev_) : nullptr;
  const cudaError_t e = pl ? cudaMallocFromPoolAsync(p, bytes, pl->pool, pl->stream) : cudaMalloc(p, bytes);
  if (e == cudaSuccess) (pl ? pooled_ : direct_).push_back(*p);
  return e;
}

cudaError_t DeviceBuffers::ready() {
  return pooled_.empty() ? cudaSuccess : cudaStreamSynchronize(pool_of(dev_)->stream);
}

void DeviceBuffers::free_all() {
  for (void *p : direct_) cudaFree(p);
  direct_.clear();
  if (pooled_.empty()) return;
  Pool *pl = pool_of(dev_);
  for (void *p : pooled_) cudaFreeAsync(p, pl->stream);
  pooled_.clear();
  // memory beyond the pool's bound goes back to the device at a synchronisation
  cudaStreamSynchronize(pl->stream);
}

cudaError_t StreamBuffer::alloc(std::size_t bytes) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  Pool *pl = bytes < kPoolBlock ? pool_of(dev) : nullptr;
  pooled_ = pl != nullptr;
  return pl ? cudaMallocFromPoolAsync(&p_, bytes, pl->pool, s_) : cudaMalloc(&p_, bytes);
}

StreamBuffer::~StreamBuffer() {
  if (!p_) return;
  if (pooled_) cudaFreeAsync(p_, s_);
  else cudaFree(p_);
}

}  // namespace hotrg
