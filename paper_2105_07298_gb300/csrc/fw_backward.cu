// Backward pass of Floyd-Warshall (an extension; the paper has no gradient).
//
// D[i][j] is the sum of the weights along path(i,j), the path encoded by the
// forward pass's P: path(i,j) = (i -> j) when P[i][j] = -1, otherwise
// path(i,k) ++ path(k,j) with k = P[i][j].  Hence for a loss L(D)
//     dL/dW[u][v] = sum of dL/dD[i][j] over the pairs (i,j) whose path uses
//                   the edge (u,v),
// which is piecewise constant in W (exact away from ties).
//
// Kernels: a warp takes a row i of a graph, its lanes the columns j; the thread
// walks path(i,j) by recomputing it from P (in-order traversal of the split
// tree, with an explicit stack of pending right endpoints) and adds dL/dD[i][j]
// to every edge it meets with an FP32 atomic add.  Nothing but P and D is kept
// from the forward pass.
//
// Bound: the latency of the dependent reads of P along a path, so what counts
// is how many walks are in flight and how near their reads are: lanes of a warp
// share the row i, where every path's first splits are read.  Few rows are cut
// into several column ranges each; a packed batch gives each graph several CTAs
// (its rows dealt out by warps), since one CTA per graph leaves the largest
// graphs to run alone at the end.  Measured: 256 graphs of 256 vertices 212 us
// (358 us with a thread per pair, located by two 64-bit divisions), 300 packed
// graphs of 20..200 vertices 104 us (375 us with one CTA per graph), one graph
// of 1000 23 us (26 us).
#include <stdint.h>

#include <algorithm>

#include "common.cuh"

namespace apsp {

constexpr int kWalkDepth = 256;  // pending right endpoints per thread (local memory)

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

// The walks of row i of one graph from column j0 on, every dj-th range of 32
// columns (lanes: columns).
__device__ __forceinline__ void scatter_row(const float *__restrict__ gD, const int32_t *__restrict__ P,
                                            const float *__restrict__ D, float *__restrict__ gW, int64_t n, int64_t ld,
                                            int64_t i, int64_t j0, int64_t dj, int32_t (&stack)[kWalkDepth],
                                            int32_t *__restrict__ status) {
  for (int64_t j = j0; j < n; j += dj) {
    if (i == j) continue;
    if (!(D[i * ld + j] < inf<float>())) continue;  // no path: contributes nothing
    const float g = gD[i * ld + j];
    if (g == 0.0f) continue;
    scatter_path(P, gW, n, ld, i, j, g, stack, status);
  }
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
    scatter_row(gD + o, P + o, D + o, gW + o, n, ld, i, (u - row * ranges) * 32 + lane, 32 * (int64_t)ranges, stack,
                status);
  }
}

// Packed batch of uneven graphs (the layout of the batched forward): graph g
// has ns[g] vertices at element offset offs[g] (ld = ns[g]), shared by `parts`
// CTAs.
__global__ void __launch_bounds__(256)
    zero_packed(float *__restrict__ gW, const int32_t *__restrict__ ns, const int64_t *__restrict__ offs, int num,
                int parts, int32_t *__restrict__ status) {
  for (int64_t t = blockIdx.x; t < (int64_t)num * parts; t += gridDim.x) {
    const int g = (int)(t / parts), part = (int)(t % parts);
    const int64_t n = ns[g], off = offs[g];
    if (n <= 0 || off < 0) {
      if (threadIdx.x == 0 && part == 0 && status && n < 0) atomicExch(status, APSP_EINVAL);
      continue;
    }
    for (int64_t e = part * 256 + threadIdx.x; e < n * n; e += parts * 256) gW[off + e] = 0.0f;
  }
}

__global__ void __launch_bounds__(256)
    fw_backward_packed_f32(const float *__restrict__ gD, const int32_t *__restrict__ P,
                           const float *__restrict__ D, float *__restrict__ gW,
                           const int32_t *__restrict__ ns, const int64_t *__restrict__ offs, int num,
                           int parts, int32_t *__restrict__ status) {
  int32_t stack[kWalkDepth];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t t = blockIdx.x; t < (int64_t)num * parts; t += gridDim.x) {
    const int g = (int)(t / parts), part = (int)(t % parts);
    const int64_t n = ns[g], off = offs[g];
    if (n <= 0 || off < 0) continue;
    for (int64_t i = part * 8 + w; i < n; i += parts * 8)
      scatter_row(gD + off, P + off, D + off, gW + off, n, n, i, lane, 32, stack, status);
  }
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
  // A row per warp, cut into ranges of columns until there are two warps for
  // every resident one (64 per SM); eight warps a CTA.
  const int64_t rows = n * batch, cap = (int64_t)sms * 64;
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
  // Eight CTAs per graph, more where few graphs would leave SMs idle.
  const int64_t cap = (int64_t)sms * 64;
  const int parts = (int)std::min<int64_t>(128, std::max<int64_t>(8, (int64_t)sms * 8 / num_graphs));
  const int64_t want = (int64_t)num_graphs * parts;
  const int grid = (int)(want < cap ? want : cap);
  apsp::zero_packed<<<grid, 256, 0, s>>>(d_grad_w, d_n, d_off, num_graphs, parts, d_status);
  apsp::fw_backward_packed_f32<<<grid, 256, 0, s>>>(d_grad_dist, d_path, d_dist, d_grad_w, d_n, d_off,
                                                     num_graphs, parts, d_status);
  return apsp::status_from(cudaGetLastError());
}
