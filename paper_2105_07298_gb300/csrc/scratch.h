// Stream-ordered scratch of a call, from a memory pool of the library's own
// (internal header).  The device's default pool gives everything back at each
// synchronisation, so a caller that waits for every solve had its scratch
// mapped again by the next one (about 0.1 ms for the packed gradient call).
// This pool keeps at most kKeepBytes mapped per device between calls and gives
// back what is above that; freeing is cudaFreeAsync.  Allocation order, streams
// and host threads are the driver's to handle, as with cudaMallocAsync.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

namespace apsp {

constexpr size_t kKeepBytes = size_t(256) << 20;

// cudaMallocAsync while `s` is being captured (the allocation then belongs to
// the graph), and where the pool cannot be had or cannot hold the block: what it
// keeps is then given back first, and the default pool may have room that other
// code of the process keeps there.
cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t s);

}  // namespace apsp
