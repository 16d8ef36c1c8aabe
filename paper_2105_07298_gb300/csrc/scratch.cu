// The library's scratch pool (scratch.h).
#include "scratch.h"

#include <mutex>

namespace apsp {

static std::mutex g_mu;
static cudaMemPool_t g_pool[64];  // per device, created on first use

static cudaError_t create_pool(int dev, cudaMemPool_t *pool) {
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaError_t e = cudaMemPoolCreate(pool, &props);
  if (e != cudaSuccess) return e;
  unsigned long long keep = kKeepBytes;
  return cudaMemPoolSetAttribute(*pool, cudaMemPoolAttrReleaseThreshold, &keep);
}

cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  int dev = 0;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone ||
      cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
    return cudaMallocAsync(p, bytes, s);
  std::lock_guard<std::mutex> lock(g_mu);
  // A second attempt with a new pool: a device reset has taken the old one.
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (!g_pool[dev] && create_pool(dev, &g_pool[dev]) != cudaSuccess) break;
    const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, g_pool[dev], s);
    if (e == cudaSuccess || e == cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    g_pool[dev] = nullptr;
  }
  cudaGetLastError();
  g_pool[dev] = nullptr;
  return cudaMallocAsync(p, bytes, s);
}

}  // namespace apsp
