// The round schedule shared by the single-graph paths (FP32 and FP64), and the
// block sets of phase 4.  Internal header.
//
// Look-ahead: everything the next round waits for runs on a second stream of
// higher priority: phase 4 of round r on row and column r+1, then phases 1-3 of
// round r+1.  The rest of round r's phase 4 runs on the caller's stream beside
// it, filling the SMs the chain leaves free; the two touch disjoint blocks and
// write/read different operand sets (round parity).
//
// No launch is programmatic (griddepcontrol), although that hides about 2.5 us a
// kernel of the chain: a dependent waits on the SMs for everything before it in its
// hardware queue, other streams' kernels among it where they share the queue, and
// these may find no SM with room beside the waiting CTAs.  Two solves at once hung so.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace apsp {

constexpr int kSms = 152;

// Block sets of one phase-4 launch.
constexpr int kSetAll = 0;   // all (R-1)^2 blocks off row/column r
constexpr int kSetNext = 1;  // the 2R-3 blocks in row r+1 or column r+1
constexpr int kSetRest = 2;  // the (R-2)^2 blocks off rows/columns r and r+1

__host__ __device__ constexpr int set_blocks(int set, int R) {
  return set == kSetNext ? 2 * R - 3 : set == kSetRest ? (R - 2) * (R - 2) : (R - 1) * (R - 1);
}

// The output block (I, J) of a launch's tile-th block in round r (R blocks a side).
__device__ __forceinline__ void block_of(int set, int tile, int r, int R, int &I, int &J) {
  if (set == kSetNext) {  // row r+1, then column r+1
    const bool row = tile < R - 1;
    const int o = row ? tile : tile - (R - 1);
    I = row ? r + 1 : o + (o >= r);
    I += !row && I >= r + 1;
    J = row ? o + (o >= r) : r + 1;
    return;
  }
  const int side = set == kSetAll ? R - 1 : R - 2;
  I = tile / side;
  J = tile % side;
  I += (I >= r);
  J += (J >= r);
  if (set == kSetRest) {
    I += (I >= r + 1);
    J += (J >= r + 1);
  }
}

// All rounds of an R-block solve.  diag(r, stream) and panels(r, stream)
// enqueue phases 1 and 2+3, phase4(r, set, blocks, stream) phase 4 on a block
// set, init(stream) what must precede every panel but not the first diagonal
// block.  While the caller's stream is being captured every phase stays on it
// (no stream is created or destroyed mid-capture).
template <typename Init, typename Diag, typename Panels, typename Phase4>
inline int run_rounds(int R, cudaStream_t s, bool capturing, Init init, Diag diag, Panels panels, Phase4 phase4) {
  if (R <= 2 || capturing) {
    if (R > 1) init(s);
    for (int r = 0; r < R; ++r) {
      diag(r, s);
      if (R == 1) break;
      panels(r, s);
      phase4(r, kSetAll, (R - 1) * (R - 1), s);
    }
    return APSP_OK;
  }
  cudaStream_t s2 = nullptr;
  cudaEvent_t ev_rest = nullptr, ev_panels = nullptr;
  int lo = 0, hi = 0;
  cudaDeviceGetStreamPriorityRange(&lo, &hi);
  if (cudaStreamCreateWithPriority(&s2, cudaStreamNonBlocking, hi) != cudaSuccess ||
      cudaEventCreateWithFlags(&ev_rest, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&ev_panels, cudaEventDisableTiming) != cudaSuccess) {
    if (s2) cudaStreamDestroy(s2);
    if (ev_rest) cudaEventDestroy(ev_rest);
    cudaGetLastError();
    return APSP_ECUDA;
  }
  cudaEventRecord(ev_panels, s);
  init(s);
  cudaEventRecord(ev_rest, s);
  cudaStreamWaitEvent(s2, ev_panels, 0);
  diag(0, s2);
  cudaStreamWaitEvent(s2, ev_rest, 0);
  panels(0, s2);
  cudaEventRecord(ev_panels, s2);
  for (int r = 0; r + 1 < R; ++r) {
    phase4(r, kSetNext, 2 * R - 3, s2);
    diag(r + 1, s2);
    cudaStreamWaitEvent(s, ev_panels, 0);  // round r's panels
    panels(r + 1, s2);
    cudaEventRecord(ev_panels, s2);
    phase4(r, kSetRest, (R - 2) * (R - 2), s);
    cudaEventRecord(ev_rest, s);
    cudaStreamWaitEvent(s2, ev_rest, 0);
  }
  cudaStreamWaitEvent(s, ev_panels, 0);
  phase4(R - 1, kSetAll, (R - 1) * (R - 1), s);
  cudaStreamDestroy(s2);
  cudaEventDestroy(ev_rest);
  cudaEventDestroy(ev_panels);
  return APSP_OK;
}

}  // namespace apsp
