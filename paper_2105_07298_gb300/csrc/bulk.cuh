// Bulk asynchronous copies (TMA engine, 1-D form) and mbarrier helpers for
// sm_103a, as inline PTX.  Internal header.
//
// A copy of `bytes` (multiple of 16, both addresses 16-byte aligned) from
// global to shared memory completes on an mbarrier as transaction bytes.
// Every wait is bounded: after kWaitLimit polls (kPollLimit of the kind that
// suspends the thread, about 3 us each) it reports failure, and the
// caller records APSP_ETIMEOUT in the translation unit's error word
// (report_wait_timeout) and leaves instead of spinning forever.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/apsp_fw.h"

namespace apsp {

constexpr uint32_t kWaitLimit = 1u << 22, kPollLimit = 1u << 18;  // both under a second

// Error word the kernels of a translation unit set when a bounded wait runs
// out (read back by apsp_device_status).
static __device__ int g_device_error = 0;

// Records that a bounded wait ran out (any thread may call it).
__device__ __forceinline__ void report_wait_timeout() { atomicExch(&g_device_error, APSP_ETIMEOUT); }

// Host side: returns and clears this translation unit's error word (APSP_OK if
// no wait ran out since the last call; APSP_ECUDA if the copy itself failed).
static inline int take_tu_device_error() {
  int v = 0;
  const int zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_device_error, sizeof(int)) != cudaSuccess) return APSP_ECUDA;
  if (v != 0 && cudaMemcpyToSymbol(g_device_error, &zero, sizeof(int)) != cudaSuccess) return APSP_ECUDA;
  return v;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// Invalidates a barrier whose phases have all completed, so that its memory
// can be initialised again (or used for anything else).
__device__ __forceinline__ void mbar_inval(uint64_t *bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Makes barrier initialisation visible to the async proxy (the copy engine).
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Orders this thread's earlier generic-proxy writes of global memory before
// later async-proxy (bulk copy) reads of it.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Orders earlier generic-proxy accesses of shared memory before later
// async-proxy (bulk copy) accesses.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Thread-block clusters: this CTA's rank, the address of a peer's shared
// memory, the cluster-wide barrier, and a 16-byte asynchronous store to a
// peer that completes on that peer's mbarrier as 16 transaction bytes.
__device__ __forceinline__ uint32_t cluster_cta_rank() {
  uint32_t v;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
  return v;
}
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank) {
  uint32_t v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(v) : "r"(addr), "r"(rank));
  return v;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ void st_async16(uint32_t addr, unsigned long long a, unsigned long long b, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(addr),
               "l"(a), "l"(b), "r"(bar)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// As mbar_wait, polling without suspending the thread: for short waits on a
// critical path (the wake-up of a suspended wait costs more than the wait).
__device__ __forceinline__ bool mbar_spin(uint64_t *bar, uint32_t parity, uint32_t limit = kWaitLimit) {
  for (uint32_t it = 0; it < limit; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// Waits for phase `parity` of `bar` to complete; false if `limit` polls ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint32_t limit = kPollLimit) {
  for (uint32_t it = 0; it < limit; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// What one thread of a CTA does whose wait ran out, before the CTA leaves:
// records it, and waits once more (bounded) for the copies still on their way, so
// that none lands in shared memory that has passed to another CTA.
__device__ __forceinline__ void give_up(uint64_t *bar, uint32_t parity) {
  report_wait_timeout();
  mbar_wait(bar, parity);
}

// The same for a CTA of a cluster to which others send (call it after the cluster's
// last barrier, when all is sent): bar[q], q < count, is completed by CTA q / own,
// phase 0 alone.  Out of line, since it is not expected to run: inside phase 1 of
// FP64 it cost 2 % of an n = 1000 solve.
static __device__ __noinline__ void drain_ring(uint64_t *bar, int count, int own, int cta) {
#pragma unroll 1
  for (int q = 0; q < count; ++q)
    if (q / own != cta) mbar_spin(&bar[q], 0, kWaitLimit / 32);
}

}  // namespace apsp
