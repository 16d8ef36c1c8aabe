// The library's scratch pool (scratch.h).
#include "scratch.h"

#include <mutex>

namespace apsp {

static std::mutex g_mu;
static cudaMemPool_t g_pool[64];  // per device, created on first use, kept to the end of the process

static cudaMemPool_t create_pool(int dev) {
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) return nullptr;
  unsigned long long keep = kKeepBytes;
  if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess) return pool;
  cudaMemPoolDestroy(pool);
  return nullptr;
}

cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  int dev = 0;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone ||
      cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
    return cudaMallocAsync(p, bytes, s);
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_pool[dev]) g_pool[dev] = create_pool(dev);
  if (g_pool[dev]) {
    if (cudaMallocFromPoolAsync(p, bytes, g_pool[dev], s) == cudaSuccess) return cudaSuccess;
    cudaMemPoolTrimTo(g_pool[dev], 0);
  }
  cudaGetLastError();
  return cudaMallocAsync(p, bytes, s);
}

}  // namespace apsp
