// Backward pass of Floyd-Warshall (an extension; the paper has no gradient).
//
// D[i][j] is the sum of the weights along path(i,j), the path encoded by the
// forward pass's P: path(i,j) = (i -> j) when P[i][j] = -1, otherwise
// path(i,k) ++ path(k,j) with k = P[i][j].  Hence for a loss L(D)
//     dL/dW[u][v] = sum of dL/dD[i][j] over the pairs (i,j) whose path uses
//                   the edge (u,v),
// which is piecewise constant in W (exact away from ties).
//
// Kernels: a thread walks path(i,j) by recomputing it from P (in-order traversal
// of the split tree, with an explicit stack of pending right endpoints) and adds
// dL/dD[i][j] to every edge it meets with an FP32 atomic add.  Nothing but P and D
// is kept from the forward pass.  A warp takes a row i of a graph, its lanes the
// columns j; in graphs of at most kFlat vertices its lanes take adjacent pairs.
//
// Bound: the latency of the dependent reads of P along a path, so what counts
// is how many walks are in flight and how near their reads are: lanes of a warp
// share the row i, where every path's first splits are read.  Few rows are cut
// into several column ranges each; a packed batch gives each graph many warps
// (adjacent ones), since one CTA per graph leaves the largest graphs to run alone
// at the end.  Measured, kernels and their launches, us (a thread per pair, found by
// two 64-bit divisions, and one CTA per packed graph; a warp per row whatever the
// size, and eight CTAs per packed graph; now):
//   stacks   256 x 256          364, 224, 223     20000 x 8   44, 94, 38
//            64 x 100            30,  31,  27      1024 x 24  30, 32, 27
//   packed   300, n 20-200      380, 113, 113     20000, n 2-8    51, 203, 39
//            2000, n 100-200   1490, 714, 695     4096, n 16-32   55,  83, 55
//            4096, n 16-256    4300, 1690, 1670   4096, n 16-24   42,  78, 48
// Up to 64 or 128 vertices a thread per pair: 64 x 100 32 / 27 us; above, 256 x 256
// 223 / 261.  Packed, 16 or 32 warps a graph: 2000, n 100-200, 1040 / 780 us.
#include <stdint.h>

#include <algorithm>

#include "common.cuh"

namespace apsp {

constexpr int kWalkDepth = 256;  // pending right endpoints per thread (local memory)

// Graphs of at most kFlat vertices are taken a thread per pair, the pairs of all
// graphs in one sequence: a warp per row would leave lanes without a column.
constexpr int kFlat = 128;

template <typename Index>
struct Pair {
  int64_t o, i, j;  // the graph's offset, row and column
  __device__ __forceinline__ Pair(Index e, Index n, int64_t stride) {
    const Index per = n * n, b = e / per, rem = e - b * per, row = rem / n;
    o = (int64_t)b * stride, i = row, j = rem - row * n;
  }
};

template <typename Index>
__global__ void __launch_bounds__(256)
    zero_pairs(float *__restrict__ G, Index n, int64_t ld, Index total, int64_t stride) {
  const Index step = (Index)gridDim.x * blockDim.x;
  for (Index e = (Index)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += step) {
    const Pair<Index> p(e, n, stride);
    G[p.o + p.i * ld + p.j] = 0.0f;
  }
}

__global__ void __launch_bounds__(256)
    zero_matrices(float *__restrict__ G, int64_t n, int64_t ld, int64_t batch, int64_t stride) {
  const int lane = threadIdx.x & 31;
  const int64_t rows = n * batch, step = (int64_t)gridDim.x * (blockDim.x / 32);
  for (int64_t row = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); row < rows; row += step) {
    const int64_t b = row / n, i = row - b * n;
    float *out = G + b * stride + i * ld;
    for (int64_t j = lane; j < n; j += 32) out[j] = 0.0f;
  }
}

// Adds g to every edge of path(i,j) of one graph (P, gW with leading
// dimension ld, n vertices).  A path of a valid P has at most n - 1 edges, so
// the walk takes at most 2n - 3 steps; the cap also ends the walk on a
// malformed P (an index outside 0..n-1 or a split cycle), which is reported
// as APSP_ETOODEEP like a recursion deeper than the stack.
__device__ __forceinline__ void scatter_path(const int32_t *__restrict__ Pg, float *__restrict__ Gg, int64_t n,
                                             int64_t ld, int64_t i, int64_t j, float g, int32_t (&stack)[kWalkDepth],
                                             int32_t *__restrict__ status) {
  int64_t a = i, c = j;
  int sp = 0;
  for (int64_t steps = 0;; ++steps) {
    const int32_t k = Pg[a * ld + c];
    if (k < 0) {  // leaf: the edge a -> c
      atomicAdd(&Gg[a * ld + c], g);
      if (sp == 0) break;
      a = c;
      c = stack[--sp];
    } else {
      if (sp == kWalkDepth || k >= n || steps > 2 * n) {
        if (status) atomicExch(status, APSP_ETOODEEP);
        break;
      }
      stack[sp++] = (int32_t)c;
      c = k;
    }
  }
}

// The walk of pair (i, j) of one graph.
__device__ __forceinline__ void scatter_pair(const float *__restrict__ gD, const int32_t *__restrict__ P,
                                             const float *__restrict__ D, float *__restrict__ gW, int64_t n, int64_t ld,
                                             int64_t i, int64_t j, int32_t (&stack)[kWalkDepth],
                                             int32_t *__restrict__ status) {
  if (i == j || !(D[i * ld + j] < inf<float>())) return;  // no path: contributes nothing
  const float g = gD[i * ld + j];
  if (g != 0.0f) scatter_path(P, gW, n, ld, i, j, g, stack, status);
}

__global__ void __launch_bounds__(256)
    fw_backward_scatter_f32(const float *__restrict__ gD, const int32_t *__restrict__ P,
                            const float *__restrict__ D, float *__restrict__ gW, int64_t n,
                            int64_t ld, int64_t batch, int64_t stride, int ranges, int32_t *__restrict__ status) {
  int32_t stack[kWalkDepth];
  const int lane = threadIdx.x & 31;
  const int64_t units = n * batch * ranges, step = (int64_t)gridDim.x * (blockDim.x / 32);
  for (int64_t u = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); u < units; u += step) {
    const int64_t row = u / ranges, b = row / n, i = row - b * n, o = b * stride;
    for (int64_t j = (u - row * ranges) * 32 + lane; j < n; j += 32 * (int64_t)ranges)
      scatter_pair(gD + o, P + o, D + o, gW + o, n, ld, i, j, stack, status);
  }
}

template <typename Index>
__global__ void __launch_bounds__(256)
    fw_backward_pairs_f32(const float *__restrict__ gD, const int32_t *__restrict__ P, const float *__restrict__ D,
                          float *__restrict__ gW, Index n, int64_t ld, Index total, int64_t stride,
                          int32_t *__restrict__ status) {
  int32_t stack[kWalkDepth];
  const Index step = (Index)gridDim.x * blockDim.x;
  for (Index e = (Index)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += step) {
    const Pair<Index> p(e, n, stride);
    scatter_pair(gD + p.o, P + p.o, D + p.o, gW + p.o, n, ld, p.i, p.j, stack, status);
  }
}

// Packed batch of uneven graphs (the layout of the batched forward): graph g has
// ns[g] vertices at element offset offs[g] (ld = ns[g]) and is shared by `slices`
// (a power of two) warps, adjacent ones, so that they find its rows in the caches.
// used(n): how many of them have work.  A small graph leaves most without: a lane
// looks after each of the warp's next 32 shares, and f(n, off, slice, lane) is called
// only where there is work.  Which slice of a graph a warp gets moves on from graph
// to graph (the grid is an odd multiple of a graph's share), so that those with work
// are spread over all warps.
template <typename Used, typename F>
__device__ __forceinline__ void packed_slices(const int32_t *__restrict__ ns, const int64_t *__restrict__ offs, int num,
                                              int slices, int32_t *__restrict__ status, Used used, F f) {
  const int lane = threadIdx.x & 31, shift = __ffs(slices) - 1;
  const int64_t units = (int64_t)num << shift, warps = (int64_t)gridDim.x * 8;
  for (int64_t u0 = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); u0 < units; u0 += 32 * warps) {
    const int64_t u = u0 + lane * warps, g = u >> shift;
    const int slice = (int)(u + g) & (slices - 1);
    int n = 0;
    int64_t off = -1;
    if (u < units) {
      n = ns[g];
      off = offs[g];
      if (n < 0 && slice == 0 && status) atomicExch(status, APSP_EINVAL);
    }
    for (unsigned left = __ballot_sync(kFullMask, n > 0 && off >= 0 && slice < used(n)); left; left &= left - 1) {
      const int src = __ffs(left) - 1;
      f((int64_t)__shfl_sync(kFullMask, n, src), __shfl_sync(kFullMask, off, src), __shfl_sync(kFullMask, slice, src), lane);
    }
  }
}

__global__ void __launch_bounds__(256)
    zero_packed(float *__restrict__ gW, const int32_t *__restrict__ ns, const int64_t *__restrict__ offs, int num,
                int slices, int32_t *__restrict__ status) {
  packed_slices(
      ns, offs, num, slices, status, [](int64_t n) { return (n * n + 31) / 32; },
      [&](int64_t n, int64_t off, int slice, int lane) {
        for (int64_t e = 32 * slice + lane; e < n * n; e += 32 * slices) gW[off + e] = 0.0f;
      });
}

__global__ void __launch_bounds__(256)
    fw_backward_packed_f32(const float *__restrict__ gD, const int32_t *__restrict__ P,
                           const float *__restrict__ D, float *__restrict__ gW,
                           const int32_t *__restrict__ ns, const int64_t *__restrict__ offs, int num,
                           int slices, int32_t *__restrict__ status) {
  int32_t stack[kWalkDepth];
  packed_slices(
      ns, offs, num, slices, nullptr, [](int64_t n) { return n <= kFlat ? (n * n + 31) / 32 : n; },
      [&](int64_t n, int64_t off, int slice, int lane) {
        auto walk = [&](int64_t i, int64_t j) {
          scatter_pair(gD + off, P + off, D + off, gW + off, n, n, i, j, stack, status);
        };
        if (n <= kFlat) {
          const unsigned m = (unsigned)n;
          for (unsigned e = 32 * slice + lane; e < m * m; e += 32 * slices) walk(e / m, e % m);
        } else {
          for (int64_t i = slice; i < n; i += slices)
            for (int64_t j = lane; j < n; j += 32) walk(i, j);
        }
      });
}

}  // namespace apsp

APSP_EXPORT int apsp_fw_backward_f32(const float *d_grad_dist, const int32_t *d_path,
                                     const float *d_dist, float *d_grad_w, int64_t n, int64_t ld,
                                     int64_t batch, int64_t stride, int32_t *d_status,
                                     void *stream) {
  if (n < 0 || batch < 0) return APSP_EINVAL;
  if (n == 0 || batch == 0) {
    if (d_status) return cudaMemsetAsync(d_status, 0, 4, reinterpret_cast<cudaStream_t>(stream)) ==
                                 cudaSuccess ? APSP_OK : APSP_ECUDA;
    return APSP_OK;
  }
  if (!d_grad_dist || !d_path || !d_dist || !d_grad_w || ld < n) return APSP_EINVAL;
  if (batch > 1 && stride < n * ld) return APSP_EINVAL;
  if (n > (1 << 18)) return APSP_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaGetLastError();
  if (d_status && cudaMemsetAsync(d_status, 0, 4, s) != cudaSuccess) return APSP_ECUDA;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t cap = (int64_t)sms * 64, total = n * n * batch;
  if (n <= apsp::kFlat) {
    const int grid = (int)std::min((total + 255) / 256, cap);
    const auto run = [&](auto nn, auto sum) {
      apsp::zero_pairs<<<grid, 256, 0, s>>>(d_grad_w, nn, ld, sum, stride);
      apsp::fw_backward_pairs_f32<<<grid, 256, 0, s>>>(d_grad_dist, d_path, d_dist, d_grad_w, nn, ld, sum, stride,
                                                       d_status);
    };
    if (total < (int64_t(1) << 31)) run((uint32_t)n, (uint32_t)total);  // (32-bit divisions; a step beyond still fits)
    else run(n, total);
    return apsp::status_from(cudaGetLastError());
  }
  // A row per warp, cut into ranges of columns until there are two warps for
  // every resident one (64 per SM); eight warps a CTA.
  const int64_t rows = n * batch;
  const int64_t ranges = std::min((n + 31) / 32, std::max<int64_t>(1, 2 * cap / rows)), want = (rows * ranges + 7) / 8;
  const int grid = (int)(want < cap ? want : cap);
  apsp::zero_matrices<<<grid, 256, 0, s>>>(d_grad_w, n, ld, batch, stride);
  apsp::fw_backward_scatter_f32<<<grid, 256, 0, s>>>(d_grad_dist, d_path, d_dist, d_grad_w, n, ld,
                                                      batch, stride, (int)ranges, d_status);
  return apsp::status_from(cudaGetLastError());
}

APSP_EXPORT int apsp_fw_backward_packed_f32(const float *d_grad_dist, const int32_t *d_path,
                                            const float *d_dist, float *d_grad_w, const int32_t *d_n,
                                            const int64_t *d_off, int32_t num_graphs, int32_t *d_status,
                                            void *stream) {
  if (num_graphs < 0) return APSP_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaGetLastError();
  if (d_status && cudaMemsetAsync(d_status, 0, 4, s) != cudaSuccess) return APSP_ECUDA;
  if (num_graphs == 0) return APSP_OK;
  if (!d_grad_dist || !d_path || !d_dist || !d_grad_w || !d_n || !d_off) return APSP_EINVAL;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // 64 warps a graph, more where few graphs would leave SMs idle; the gradient is
  // zeroed by eight.  Many graphs: half as many CTAs take more of them each.
  const bool many = num_graphs >= sms * 16;
  int slices = 64;
  while (slices < 1024 && (int64_t)num_graphs * slices < (int64_t)sms * 64) slices *= 2;
  const int zero_slices = num_graphs < sms * 8 ? slices : 8;
  const auto grid = [&](int per, int ctas) {
    return (int)std::min<int64_t>((int64_t)num_graphs * (per / 8), (int64_t)(per / 8) * ((sms * ctas / (per / 8)) | 1));
  };
  apsp::zero_packed<<<grid(zero_slices, 16), 256, 0, s>>>(d_grad_w, d_n, d_off, num_graphs, zero_slices, d_status);
  apsp::fw_backward_packed_f32<<<grid(slices, many ? 32 : 64), 256, 0, s>>>(d_grad_dist, d_path, d_dist, d_grad_w, d_n,
                                                                            d_off, num_graphs, slices, d_status);
  return apsp::status_from(cudaGetLastError());
}
