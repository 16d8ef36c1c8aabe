// Batched Floyd-Warshall: thousands of independent graphs of uneven size in
// one persistent launch (an extension; the paper solves one matrix at a time).
//
// Work distribution: the plan orders the graphs largest first (longest
// processing time first) and the CTAs of a grid sized to fill every SM pop
// graph indices from one atomic counter.  A CTA solves its graph alone, so no
// CTA ever waits on another.
//
// Per graph (n_g <= 1024, row-major, ld = n_g) the CTA runs the blocked FW of
// §2.2 on the matrix in global memory, with one of three kernel variants
// chosen per size class by the autotuner:
//   variants 0 and 1, 64 x 64 blocks, 4 x 4 register tile per thread:
//     phase 1     register-resident closure of the diagonal block;
//     phases 2+3  row block (r,J) <- min(C, D*(r,r) (x) C) and column block
//                 (I,r) <- min(C, C (x) D*(r,r)): once the diagonal block is
//                 closed, the sequential k loop over a panel block equals one
//                 min-plus product with the closed block (same value in exact
//                 arithmetic), so these phases use the phase-4 block product;
//     phase 4     (I,J) <- min(C, D(I,r) (x) D(r,J)), both operand blocks whole
//                 in shared memory (k-pair layout);
//     path matrix: variant 0 recovers each improved output's first argmin k
//     from the operands after the product (lazy), variant 1 keeps the index
//     of the last improving k-pair in the inner loop (eager);
//     variant 1, and every variant run without a path matrix, closes the
//     diagonal block four steps per barrier and pipelines the products of a
//     phase group: the operands the next product does not share with this one
//     are copied while this one computes.
//   variant 2, 128 x 128 blocks, 8 x 4 register tile per thread: the
//     single-graph kernels' code run by one CTA: the register-resident closure
//     for phase 1, the k-sequential line kernel for phases 2+3 (the paper's
//     order), which also writes the round's operand panels into this CTA's
//     scratch, and the bulk-copy ring product for phase 4 (two 128 x 64
//     halves per block), tracking the path eagerly in the product's inner
//     loop (a graph of n <= 1024 has at most 8 rounds, all dense in
//     improvements).
// On integer-valued weights all sums are exact and D equals every other
// correct FW whatever the variant; on real weights variant 2 gives the
// sequential blocked FW's values at TB = 128 (those of apsp_fw_f32), variants
// 0 and 1 round phases 2/3 through the closed block instead.
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <exception>
#include <numeric>
#include <vector>

#include "bulk.cuh"
#include "common.cuh"
#include "scratch.h"
#include "minplus_f32.cuh"
#include "phases_f32.cuh"

namespace apsp {

constexpr int kBatchedMaxN = 1024;

constexpr int kNumClasses = 4;
static const int32_t kClassLo[kNumClasses] = {1, 65, 129, 257};
static const int32_t kClassHi[kNumClasses] = {64, 128, 256, kBatchedMaxN};
__host__ __device__ constexpr int class_of_n(int32_t n) {
  return n <= 64 ? 0 : n <= 128 ? 1 : n <= 256 ? 2 : 3;
}
constexpr int kNumVariants = 3;
static int g_variant[kNumClasses] = {1, 1, 1, 1};
// Block edge, register tile and path tracking of each variant (for the
// autotuner's table).
static const int kVariantBlock[kNumVariants] = {64, 64, 128};
static const int kVariantTileRows[kNumVariants] = {4, 4, 8};
static const int kVariantTileCols[kNumVariants] = {4, 4, 4};
static const int kVariantEager[kNumVariants] = {0, 1, 1};
constexpr int kT128 = mp32::T;
// Per-CTA operand panels of the 128-block variants: Apan and Bpan of every
// block of one round (R <= 8 blocks for n <= 1024), 4-byte words.
__host__ __device__ constexpr size_t panel_words_per_array(int rmax) { return (size_t)rmax * kT128 * kT128; }
__host__ __device__ constexpr size_t panel_bytes_per_cta(int rmax) { return 2 * panel_words_per_array(rmax) * 4; }

static int class_of(int32_t n) { return class_of_n(n); }

namespace b64 {
constexpr int T = 64;           // block edge
constexpr int TM = 4;           // 4 x 4 outputs per thread, 256 threads
constexpr int KP = T / 2;       // k-pairs per block
constexpr int ST = T + 2;       // row stride of the pair arrays (16-byte rows, fewer conflicts)
constexpr int CS = T + 8;       // row stride of Cs: a warp's 8-byte stores (four rows two
                                // apart) take the minimum two shared-memory wavefronts

struct ProdSmem {
  unsigned long long As[KP][ST];  // As[kp][i] = (A[i][2kp], A[i][2kp+1])
  unsigned long long Bs[KP][ST];  // Bs[kp][j] = (B[2kp][j], B[2kp+1][j])
  float Cs[T][CS];                // new candidates
};
}  // namespace b64

// Copies of operand blocks in shared memory: the k-paired layout of the A and
// the B operand, two buffers each.
struct Bufs64 {
  unsigned long long A[2][b64::KP][b64::ST];  // A[kp][i] = (A[i][2kp], A[i][2kp+1])
  unsigned long long B[2][b64::KP][b64::ST];  // B[kp][j] = (B[2kp][j], B[2kp+1][j])
};
// The closure's histories.
struct Quad64 {
  unsigned long long hr[b64::KP][b64::T];    // (row 2kp, row 2kp+1), each at its own step
  unsigned long long hcol[b64::T][b64::KP];  // (column 2kp, column 2kp+1) likewise
  float x[2][b64::T][4];                     // columns of the current quad before its steps
};

union BatchedSmem {
  b64::ProdSmem prod;
  Bufs64 bufs;
  Quad64 quad;
  mp32::DiagSmemT<64> diag;
  mp32::DiagSmemT<128> diag128;
  float lines_M[k2::T * k2::MS];
  k3::Smem prod128;
};

__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

// C(baseI, baseJ) <- min(C, A(baseI, baseK) (x) B(baseK, baseJ)), TB = 64,
// all 256 threads, the lazy path matrix of variant 0 (each improved output's
// first argmin k recovered from the operands after the product).  C may be
// the same block as A or B: the operands are copied to shared memory first
// and C is written only after every read.
__device__ __forceinline__ void product64_lazy(float *__restrict__ D, int ld, int32_t *__restrict__ P,
                                               int baseI, int baseJ, int baseK, int mI, int mJ, int mK,
                                               b64::ProdSmem &sm) {
  using namespace b64;
  using mp32::col_at;
  using mp32::row_at;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ty = mp32::thread_ty(), tx = mp32::thread_tx();
  const float INF = inf<float>();
  __syncthreads();  // the previous user of sm is done with it
  {  // both operand blocks, every element one 4-byte asynchronous copy
    float *as = reinterpret_cast<float *>(&sm.As[0][0]);
    float *bs = reinterpret_cast<float *>(&sm.Bs[0][0]);
#pragma unroll
    for (int q = 0; q < T * T / 256; ++q) {
      const int idx = tid + q * 256, i = idx / T, k = idx % T;
      float *dst = as + ((k >> 1) * ST + i) * 2 + (k & 1);
      if (i < mI && k < mK) mp32::cp_async4(dst, D + (int64_t)(baseI + i) * ld + baseK + k);
      else *dst = INF;
    }
#pragma unroll
    for (int q = 0; q < T * T / 256; ++q) {
      const int idx = tid + q * 256, k = idx / T, j = idx % T;
      float *dst = bs + ((k >> 1) * ST + j) * 2 + (k & 1);
      if (j < mJ && k < mK) mp32::cp_async4(dst, D + (int64_t)(baseK + k) * ld + baseJ + j);
      else *dst = INF;
    }
    mp32::cp_async_commit();
    mp32::cp_async_wait<0>();
  }
  __syncthreads();
  float acc[TM][TM];
#pragma unroll
  for (int a = 0; a < TM; ++a)
#pragma unroll
    for (int c = 0; c < TM; ++c) acc[a][c] = INF;
  const int kpn = (mK + 1) / 2;
  auto load_pair = [&](int kp, unsigned long long (&a)[TM], unsigned long long (&b)[TM]) {
#pragma unroll
    for (int rr = 0; rr < TM; rr += 2) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(&sm.As[kp][row_at(rr, ty)]);
      a[rr] = t.x;
      a[rr + 1] = t.y;
    }
#pragma unroll
    for (int cc = 0; cc < TM; cc += 2) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(&sm.Bs[kp][col_at(cc, tx)]);
      b[cc] = t.x;
      b[cc + 1] = t.y;
    }
  };
#pragma unroll 1
  for (int kp = 0; kp < kpn; ++kp) {
    unsigned long long a[TM], b[TM];
    load_pair(kp, a, b);
#pragma unroll
    for (int rr = 0; rr < TM; ++rr)
#pragma unroll
      for (int cc = 0; cc < TM; ++cc) mp32::relax2(acc[rr][cc], a[rr], b[cc]);
  }
  // Epilogue: candidates to shared memory; each warp then owns 8 whole rows,
  // lane l the columns 2l and 2l+1.
#pragma unroll
  for (int rr = 0; rr < TM; ++rr)
#pragma unroll
    for (int cc = 0; cc < TM; cc += 2) {
      *reinterpret_cast<float2 *>(&sm.Cs[row_at(rr, ty)][col_at(cc, tx)]) =
          make_float2(acc[rr][cc], acc[rr][cc + 1]);
    }
  __syncthreads();
  const int i0 = w * 8, j0 = 2 * lane;
  float o[8][2];
#pragma unroll
  for (int t = 0; t < 8; ++t)
#pragma unroll
    for (int q = 0; q < 2; ++q)
      o[t][q] = (i0 + t < mI && j0 + q < mJ) ? D[(int64_t)(baseI + i0 + t) * ld + baseJ + j0 + q] : INF;
  unsigned flags = 0u;  // bit 2t + q: row i0 + t, column j0 + q improved
#pragma unroll
  for (int t = 0; t < 8; ++t)
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (sm.Cs[i0 + t][j0 + q] < o[t][q]) flags |= 1u << (2 * t + q);
  if (P) {
    // lazy P: one improved output per warp pass; lane l tests k = 2l, 2l+1
    // with one paired add of As[l][i] and Bs[l][j] (shared memory).
    unsigned wflags = __reduce_or_sync(kFullMask, flags);
#pragma unroll 1
    while (wflags) {
      const int t = (__ffs(wflags) - 1) >> 1;
      wflags &= ~(3u << (2 * t));
      const int i = i0 + t;
      unsigned imp = (flags >> (2 * t)) & 3u;
      unsigned bal = __ballot_sync(kFullMask, imp != 0);
      const unsigned long long av = sm.As[lane][i];
      while (bal) {
        const int src = __ffs(bal) - 1;
        const unsigned sim = __shfl_sync(kFullMask, imp, src);
        const int q0 = __ffs(sim) - 1;
        if (lane == src) imp &= imp - 1;
        if (!(sim & (sim - 1))) bal &= bal - 1;
        const int sj = 2 * src + q0;
        const float tgt = sm.Cs[i][sj];
        const unsigned long long bv = sm.Bs[lane][sj];
        float c0, c1;
        asm("{\n\t.reg .b64 t;\n\tadd.rn.f32x2 t, %2, %3;\n\tmov.b64 {%0, %1}, t;\n\t}"
            : "=f"(c0), "=f"(c1)
            : "l"(av), "l"(bv));
        const unsigned h = (c0 == tgt ? 1u : 0u) | (c1 == tgt ? 2u : 0u);
        const unsigned hb = __ballot_sync(kFullMask, h != 0);
        const int L = __ffs(hb) - 1;
        const unsigned hL = __shfl_sync(kFullMask, h, L & 31);
        if (lane == 0 && hb) P[(int64_t)(baseI + i) * ld + baseJ + sj] = baseK + 2 * L + (__ffs(hL) - 1);
      }
    }
  }
  __syncthreads();  // every read of the operands precedes the writes
#pragma unroll
  for (int t = 0; t < 8; ++t)
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if ((flags >> (2 * t + q)) & 1u) {
        const int64_t g = (int64_t)(baseI + i0 + t) * ld + baseJ + j0 + q;
        D[g] = sm.Cs[i0 + t][j0 + q];
      }
}

// Variant 0 with a path matrix: unpipelined products, lazy path recovery.
__device__ __forceinline__ void solve_graph_lazy_f32(float *__restrict__ D, int32_t *__restrict__ P,
                                                int n, BatchedSmem &sm) {
  constexpr int T = b64::T;
  const int ld = n;
  const int R = (n + T - 1) / T;
  for (int r = 0; r < R; ++r) {
    const int base = r * T, m = min(T, n - base);
    __syncthreads();
    mp32::diag_closure<4>(D, ld, P, base, m, sm.diag);
    __syncthreads();
    for (int J = 0; J < R; ++J) {
      if (J == r) continue;
      product64_lazy(D, ld, P, base, J * T, base, m, min(T, n - J * T), m, sm.prod);
    }
    for (int I = 0; I < R; ++I) {
      if (I == r) continue;
      product64_lazy(D, ld, P, I * T, base, base, min(T, n - I * T), m, m, sm.prod);
    }
    __syncthreads();
    for (int I = 0; I < R; ++I) {
      if (I == r) continue;
      for (int J = 0; J < R; ++J) {
        if (J == r) continue;
        product64_lazy(D, ld, P, I * T, J * T, base, min(T, n - I * T), min(T, n - J * T), m, sm.prod);
      }
    }
  }
  __syncthreads();
}

// --------------------------------------------------------------------------
// Variant 1, and every variant without a path matrix: 64-block closure by
// quads of steps, then pipelined 64-block products.
// --------------------------------------------------------------------------

// Phase 1 on the diagonal block at `base` (m valid vertices, 256 threads): each
// thread keeps 4 x 4 adjacent elements, and the four steps of a quad share one
// barrier.  The threads of the quad's rows (one half-warp) take the quad's own
// 4 x 4 entries by shuffle, bring their rows to each row's step and publish
// them; the threads of its columns publish those as they are; after the
// barrier every thread brings its rows' four column values to their steps
// against the published 4 x 4 entries and relaxes its elements (two packed
// adds and two three-input mins each).  Step k never changes row or column k.
// TRACK: elements are compared once per quad, and the k of the last improvement
// found among its four steps afterwards (the first whose candidate from the
// histories equals the final value).
template <bool TRACK>
__device__ __forceinline__ void closure64(float *__restrict__ D, int ld, int32_t *__restrict__ P, int base, int m,
                                          Quad64 &sm) {
  using mp32::pack2;
  const int tid = threadIdx.x, w = tid >> 5, ty = tid >> 4, tx = tid & 15;
  const int i0 = 4 * ty, j0 = 4 * tx;
  const float INF = inf<float>();
  float d[4][4];
  int aux[4][4];  // TRACK: last quad that lowered the element, -1 none; else its input's bits
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      d[a][c] = (i0 + a < m && j0 + c < m) ? D[(base + i0 + a) * ld + base + j0 + c] : INF;
      aux[a][c] = TRACK ? -1 : __float_as_int(d[a][c]);
    }
  const int nq = (m + 3) / 4;
  const bool idle = 8 * w >= m;  // warp-uniform: no valid row
#pragma unroll 1
  for (int q = 0; q < nq; ++q) {
    float e01, e02, e03, e12, e13, e23;
    auto pivots = [&](float (&p)[4]) {  // a row's values at the quad's columns brought to their steps
      p[1] = fminf(p[1], __fadd_rn(p[0], e01));
      p[2] = mp32::min3f(p[2], __fadd_rn(p[0], e02), __fadd_rn(p[1], e12));
      p[3] = fminf(mp32::min3f(p[3], __fadd_rn(p[0], e03), __fadd_rn(p[1], e13)), __fadd_rn(p[2], e23));
    };
    if (tx == q) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
        *reinterpret_cast<float4 *>(&sm.x[q & 1][i0 + a][0]) = make_float4(d[a][0], d[a][1], d[a][2], d[a][3]);
    }
    if (w == q >> 1) {
      float x[4][4];
      const int src = (q & 1) * 16 + q;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) x[a][c] = __shfl_sync(kFullMask, d[a][c], src);
      if (ty == q) {
        e01 = x[0][1], e02 = x[0][2], e03 = x[0][3];
        e12 = fminf(x[1][2], __fadd_rn(x[1][0], e02));
        e13 = fminf(x[1][3], __fadd_rn(x[1][0], e03));
        const float y21 = fminf(x[2][1], __fadd_rn(x[2][0], e01));
        e23 = mp32::min3f(x[2][3], __fadd_rn(x[2][0], e03), __fadd_rn(y21, e13));
#pragma unroll
        for (int a = 1; a < 4; ++a) pivots(x[a]);
        unsigned long long ha[4], hb[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float r0 = d[0][c], r1 = fminf(d[1][c], __fadd_rn(x[1][0], r0));
          const float r2 = mp32::min3f(d[2][c], __fadd_rn(x[2][0], r0), __fadd_rn(x[2][1], r1));
          const float r3 = fminf(mp32::min3f(d[3][c], __fadd_rn(x[3][0], r0), __fadd_rn(x[3][1], r1)),
                                 __fadd_rn(x[3][2], r2));
          ha[c] = pack2(r0, r1);
          hb[c] = pack2(r2, r3);
        }
#pragma unroll
        for (int c = 0; c < 4; c += 2) {
          *reinterpret_cast<ulonglong2 *>(&sm.hr[2 * q][j0 + c]) = make_ulonglong2(ha[c], ha[c + 1]);
          *reinterpret_cast<ulonglong2 *>(&sm.hr[2 * q + 1][j0 + c]) = make_ulonglong2(hb[c], hb[c + 1]);
        }
      }
    }
    __syncthreads();
    if (idle) continue;
    const ulonglong2 q0 = *reinterpret_cast<const ulonglong2 *>(&sm.hr[2 * q][4 * q]);
    const ulonglong2 q1 = *reinterpret_cast<const ulonglong2 *>(&sm.hr[2 * q][4 * q + 2]);
    e01 = __uint_as_float((unsigned)q0.y);
    e02 = __uint_as_float((unsigned)q1.x);
    e03 = __uint_as_float((unsigned)q1.y);
    e12 = __uint_as_float((unsigned)(q1.x >> 32));
    e13 = __uint_as_float((unsigned)(q1.y >> 32));
    e23 = __uint_as_float((unsigned)sm.hr[2 * q + 1][4 * q + 3]);
    unsigned long long ha[4], hb[4];
#pragma unroll
    for (int c = 0; c < 4; c += 2) {
      const ulonglong2 ta = *reinterpret_cast<const ulonglong2 *>(&sm.hr[2 * q][j0 + c]);
      const ulonglong2 tb = *reinterpret_cast<const ulonglong2 *>(&sm.hr[2 * q + 1][j0 + c]);
      ha[c] = ta.x, ha[c + 1] = ta.y, hb[c] = tb.x, hb[c + 1] = tb.y;
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float4 t = *reinterpret_cast<const float4 *>(&sm.x[q & 1][i0 + a][0]);
      float p[4] = {t.x, t.y, t.z, t.w};
      pivots(p);
      const unsigned long long pa = pack2(p[0], p[1]), pb = pack2(p[2], p[3]);
      if (TRACK && tx == 0) *reinterpret_cast<ulonglong2 *>(&sm.hcol[i0 + a][2 * q]) = make_ulonglong2(pa, pb);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float v = mp32::min3f_pair(mp32::min3f_pair(d[a][c], pa, ha[c]), pb, hb[c]);
        if (TRACK) aux[a][c] = v < d[a][c] ? q : aux[a][c];
        d[a][c] = v;
      }
    }
  }
  if (idle) return;
  __syncwarp();  // hcol is written and read by the same half-warps
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = i0 + a, j = j0 + c, e = (base + i) * ld + base + j;
      const float g = d[a][c];
      if constexpr (TRACK) {
        const int q = aux[a][c];
        if (q < 0) continue;  // (improved elements are valid)
        const float2 t0 = mp32::sum2(sm.hcol[i][2 * q], sm.hr[2 * q][j]);
        const float2 t1 = mp32::sum2(sm.hcol[i][2 * q + 1], sm.hr[2 * q + 1][j]);
        D[e] = g;
        P[e] = base + 4 * q + (t0.x == g ? 0 : t0.y == g ? 1 : t1.x == g ? 2 : 3);
      } else {
        if (g < __int_as_float(aux[a][c])) D[e] = g;
      }
    }
}

// The A operand D(baseI.., baseK..) into a buffer (+inf outside the valid
// extents), asynchronously: 8-byte copies of a k-pair where every pair starts
// on an 8-byte boundary (even ld and an aligned D), else 4-byte ones.
__device__ __forceinline__ void stage_a(unsigned long long (&dst)[b64::KP][b64::ST], const float *__restrict__ D,
                                        int ld, int baseI, int baseK, int mI, int mK) {
  using namespace b64;
  const int tid = threadIdx.x;
  const float INF = inf<float>();
  if ((ld & 1) == 0 && (reinterpret_cast<uintptr_t>(D) & 7) == 0) {
#pragma unroll
    for (int q = 0; q < T * KP / 256; ++q) {
      const int idx = tid + q * 256, i = idx / KP, kp = idx % KP;
      unsigned long long *to = &dst[kp][i];
      const float *from = D + (baseI + i) * ld + baseK + 2 * kp;
      if (i < mI && 2 * kp + 1 < mK) {
        cp_async8(to, from);
      } else {
        float *f = reinterpret_cast<float *>(to);
        f[1] = INF;
        if (i < mI && 2 * kp < mK) mp32::cp_async4(f, from);
        else f[0] = INF;
      }
    }
  } else {
#pragma unroll
    for (int q = 0; q < T * T / 256; ++q) {
      const int idx = tid + q * 256, i = idx / T, k = idx % T;
      float *to = reinterpret_cast<float *>(&dst[k >> 1][i]) + (k & 1);
      if (i < mI && k < mK) mp32::cp_async4(to, D + (baseI + i) * ld + baseK + k);
      else *to = INF;
    }
  }
}
// The B operand D(baseK.., baseJ..).
__device__ __forceinline__ void stage_b(unsigned long long (&dst)[b64::KP][b64::ST], const float *__restrict__ D,
                                        int ld, int baseK, int baseJ, int mK, int mJ) {
  using namespace b64;
  const int tid = threadIdx.x;
  const float INF = inf<float>();
#pragma unroll
  for (int q = 0; q < T * T / 256; ++q) {
    const int idx = tid + q * 256, k = idx / T, j = idx % T;
    float *to = reinterpret_cast<float *>(&dst[k >> 1][j]) + (k & 1);
    if (j < mJ && k < mK) mp32::cp_async4(to, D + (baseK + k) * ld + baseJ + j);
    else *to = INF;
  }
}

// C(baseI, baseJ) <- min(C, A (x) B) from filled buffers, all 256 threads.  A
// warp owns eight rows (one without a valid row does nothing), a thread 4 x 4
// outputs.  The accumulators start at C, so an output improves exactly
// when its accumulator falls.  TRACK: compared once per four k (one compare and
// one select per output); the first of the last improving four whose candidate
// equals the new value is the path entry (the sequential loop's, strict "<").
// Fewer comparisons lose here: with 8 or 16 candidates to look through for
// every improved output (20-90 % of them in a round) the 4096-graph batch took
// 23.3 and 26.2 ms against 21.0.
// Bound: instruction issue and the ALU pipe (a min, a compare and a select per
// two pairs).  Measured on that batch (n ~ U[16, 512]): 21.0 ms with P, 13.8
// without (22.7 and 15.9 with every product copying both operands 4 bytes at a
// time and computing all 64 rows of a ragged block); lanes two rows of pairs by
// sixteen columns: four by eight took 21.6 ms.
template <bool TRACK>
__device__ __forceinline__ void product64(float *__restrict__ D, int ld, int32_t *__restrict__ P, int baseI, int baseJ,
                                          int baseK, int mI, int mJ, int mK,
                                          const unsigned long long (&A)[b64::KP][b64::ST],
                                          const unsigned long long (&B)[b64::KP][b64::ST]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (8 * w >= mI) return;  // warp-uniform
  const int r0 = 8 * w + 2 * (lane >> 4), c0 = 2 * (lane & 15);
  const float INF = inf<float>();
  float acc[4][4];
  int aux[4][4];  // TRACK: last k-pair step (two pairs) that lowered the output, -1 none; else C's bits
  const int e0 = (baseI + r0) * ld + baseJ + c0;  // output (a, c): row (a & 1) + 4 (a >> 1), column (c & 1) + 32 (c >> 1) further
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int di = (a & 1) + 4 * (a >> 1), dj = (c & 1) + 32 * (c >> 1);
      acc[a][c] = (r0 + di < mI && c0 + dj < mJ) ? D[e0 + di * ld + dj] : INF;
      aux[a][c] = TRACK ? -1 : __float_as_int(acc[a][c]);
    }
  auto load = [&](int kp, unsigned long long (&a)[4], unsigned long long (&b)[4]) {
#pragma unroll
    for (int u = 0; u < 4; u += 2) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(&A[kp][r0 + 2 * u]);
      const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&B[kp][c0 + 16 * u]);
      a[u] = t.x, a[u + 1] = t.y, b[u] = v.x, b[u + 1] = v.y;
    }
  };
  const int kpn = ((mK + 3) / 4) * 2;  // whole steps of two k-pairs: the operands are +inf past mK
#pragma unroll 1
  for (int kp = 0; kp < kpn; kp += 2) {
    unsigned long long a0[4], b0[4], a1[4], b1[4];
    load(kp, a0, b0);
    load(kp + 1, a1, b1);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float m = mp32::min3f_pair(mp32::min3f_pair(acc[a][c], a0[a], b0[c]), a1[a], b1[c]);
        if (TRACK) aux[a][c] = m < acc[a][c] ? kp : aux[a][c];
        acc[a][c] = m;
      }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int di = (a & 1) + 4 * (a >> 1), dj = (c & 1) + 32 * (c >> 1), e = e0 + di * ld + dj;
      const float g = acc[a][c];
      if constexpr (TRACK) {
        const int kp = aux[a][c];
        if (kp < 0) continue;  // (improved outputs are valid)
        const unsigned long long *pa = &A[kp][r0 + di], *pb = &B[kp][c0 + dj];
        const float2 t0 = mp32::sum2(pa[0], pb[0]), t1 = mp32::sum2(pa[b64::ST], pb[b64::ST]);
        D[e] = g;
        P[e] = baseK + 2 * kp + (t0.x == g ? 0 : t0.y == g ? 1 : t1.x == g ? 2 : 3);
      } else {
        if (g < __int_as_float(aux[a][c])) D[e] = g;
      }
    }
}

// The products of round r (m valid vertices) in group 0 (phases 2+3: the row
// blocks (r, J), then the column blocks (I, r), each with the closed diagonal
// block) or group 1 (phase 4, column by column).  No product of a group reads
// a block another one writes, so the operands of the next product are copied
// while the current one computes; an operand two products share is copied once.
template <bool TRACK>
__device__ __forceinline__ void run_group64(float *__restrict__ D, int ld, int32_t *__restrict__ P, int n, int r,
                                            int group, Bufs64 &sm) {
  constexpr int T = b64::T;
  const int R = (n + T - 1) / T, base = r * T, m = min(T, n - base);
  const int np = group == 0 ? 2 * (R - 1) : (R - 1) * (R - 1);
  auto coords = [&](int p, int &I, int &J) {
    if (group == 0) {
      const int o = p % (R - 1), O = o + (o >= r);
      I = p < R - 1 ? r : O;
      J = p < R - 1 ? O : r;
    } else {
      I = p % (R - 1);
      J = p / (R - 1);
      I += I >= r;
      J += J >= r;
    }
  };
  int I, J, ba = 0, bb = 0;  // the product and the buffers that hold its operands
  coords(0, I, J);
  stage_a(sm.A[0], D, ld, I * T, base, min(T, n - I * T), m);
  stage_b(sm.B[0], D, ld, base, J * T, m, min(T, n - J * T));
  mp32::cp_async_commit();
#pragma unroll 1
  for (int p = 0; p < np; ++p) {
    int nI = I, nJ = J, na = ba, nb = bb;
    if (p + 1 < np) {
      coords(p + 1, nI, nJ);
      __syncthreads();  // product p-1 is done with the buffers refilled here
      if (nI != I) {
        na = ba ^ 1;
        stage_a(sm.A[na], D, ld, nI * T, base, min(T, n - nI * T), m);
      }
      if (nJ != J) {
        nb = bb ^ 1;
        stage_b(sm.B[nb], D, ld, base, nJ * T, m, min(T, n - nJ * T));
      }
      mp32::cp_async_commit();
      mp32::cp_async_wait<1>();
    } else {
      mp32::cp_async_wait<0>();
    }
    __syncthreads();  // every thread's copies for product p are visible
    product64<TRACK>(D, ld, P, I * T, J * T, base, min(T, n - I * T), min(T, n - J * T), m, sm.A[ba], sm.B[bb]);
    I = nI;
    J = nJ;
    ba = na;
    bb = nb;
  }
}

template <bool TRACK>
__device__ __forceinline__ void solve_graph_pipe_f32(float *__restrict__ D, int32_t *__restrict__ P, int n,
                                                     BatchedSmem &sm) {
  constexpr int T = b64::T;
  const int ld = n;
  const int R = (n + T - 1) / T;
  for (int r = 0; r < R; ++r) {
    const int base = r * T, m = min(T, n - base);
    __syncthreads();  // the previous round's products are done with the buffers
    closure64<TRACK>(D, ld, P, base, m, sm.quad);
    __syncthreads();
    if (R == 1) break;
    run_group64<TRACK>(D, ld, P, n, r, 0, sm.bufs);
    __syncthreads();  // the panels are final (and visible) before phase 4 copies them
    run_group64<TRACK>(D, ld, P, n, r, 1, sm.bufs);
  }
  __syncthreads();
}

// The 128-block variant: the single-graph phases run by this CTA alone.
// The panels (this CTA's scratch) are rewritten every round: every thread fences
// its generic writes before the bulk copies read them.
// Returns false if a bounded copy wait ran out (error word set).
__device__ __forceinline__ bool solve_graph128_f32(float *__restrict__ D, int32_t *__restrict__ P, int n,
                                                   const Panels &pan, bool aligned, unsigned char *smem_raw) {
  constexpr int T = kT128;
  BatchedSmem &sm = *reinterpret_cast<BatchedSmem *>(smem_raw);
  const int64_t ld = n;
  const int R = (n + T - 1) / T;
  const int vec_ok = aligned && (n % 4 == 0);
  for (int r = 0; r < R; ++r) {
    const int base = r * T, m = min(T, n - base);
    __syncthreads();
    mp32::diag_closure<8>(D, ld, P, base, m, sm.diag128);
    __syncthreads();
    if (R == 1) break;
    for (int side = 0; side < 2; ++side) {  // row blocks (r, J), then column blocks (I, r)
      const bool is_row = side == 0;
      lines_load_diag(D, ld, n, r, is_row);
      __syncthreads();
      for (int o = 0; o < R; ++o) {
        if (o == r) continue;
        for (int part = 0; part < k2::PARTS; ++part) lines_part_f32(D, ld, P, n, r, o, is_row, part, pan);
      }
      __syncthreads();
    }
    fence_proxy_async_global();
    __syncthreads();
    for (int I = 0; I < R; ++I) {
      if (I == r) continue;
      for (int J = 0; J < R; ++J) {
        if (J == r) continue;
        for (int hJ = 0; hJ < 2; ++hJ) {
          __syncthreads();  // the previous product's epilogue is done with the shared memory
          if (!minplus_half_f32(D, ld, P, n, I, J, hJ, r, vec_ok, pan)) return false;
        }
      }
    }
  }
  __syncthreads();
  return true;
}

// Work item t: graph order[t] & 0x3fffffff, variant order[t] >> 30.
// scratch: per-CTA panel space of the 128-block variant (panel_bytes_per_cta(rmax)
// bytes per CTA).  Two instances: the 64-block variants alone (three CTAs per
// SM), and all variants (two CTAs per SM: the 128-block code needs more
// registers); a plan launches the second only if some graph uses variant 2.
template <bool WITH128>
__device__ __forceinline__ void persistent_body(float *__restrict__ Dp, int32_t *__restrict__ Pp,
                                                const int32_t *__restrict__ order, const int32_t *__restrict__ ns,
                                                const int64_t *__restrict__ offs, int num, int *__restrict__ counter,
                                                unsigned char *__restrict__ scratch, int rmax) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  BatchedSmem &sm = *reinterpret_cast<BatchedSmem *>(smem_raw);
  __shared__ int s_next;
  Panels pan{};
  if (WITH128 && scratch) {
    unsigned char *base = scratch + (size_t)blockIdx.x * panel_bytes_per_cta(rmax);
    const size_t words = panel_words_per_array(rmax);
    pan.Apan = reinterpret_cast<unsigned long long *>(base);
    pan.Bpan = reinterpret_cast<unsigned long long *>(base + words * 4);
  }
  for (;;) {
    if (threadIdx.x == 0) s_next = atomicAdd(counter, 1);
    __syncthreads();
    const int t = s_next;
    __syncthreads();  // all threads have read s_next before it is overwritten
    if (t >= num) break;
    const int item = order[t];
    const int g = item & 0x3fffffff, variant = (int)((unsigned)item >> 30);
    const int64_t off = offs[g];
    const int n = ns[g];
    float *D = Dp + off;
    int32_t *P = Pp ? Pp + off : nullptr;
    if (P) {
      for (int e = threadIdx.x; e < n * n; e += blockDim.x) P[e] = -1;
    }
    bool ok = true;
    if constexpr (WITH128) {
      if (variant == 2 && scratch) {
        const bool aligned = (reinterpret_cast<uintptr_t>(D) & 15) == 0;
        ok = solve_graph128_f32(D, P, n, pan, aligned, smem_raw);
        if (!ok) return;  // a copy wait ran out: the error word is set, this CTA stops
        continue;
      }
    }
    if (!P)
      solve_graph_pipe_f32<false>(D, P, n, sm);
    else if (variant == 1 || variant == 2)
      solve_graph_pipe_f32<true>(D, P, n, sm);
    else
      solve_graph_lazy_f32(D, P, n, sm);
  }
}

__global__ void __launch_bounds__(mp32::THREADS, 3)
    fw_batched_persistent_f32(float *__restrict__ Dp, int32_t *__restrict__ Pp,
                              const int32_t *__restrict__ order, const int32_t *__restrict__ ns,
                              const int64_t *__restrict__ offs, int num, int *__restrict__ counter,
                              unsigned char *__restrict__ scratch, int rmax) {
  persistent_body<false>(Dp, Pp, order, ns, offs, num, counter, scratch, rmax);
}

__global__ void __launch_bounds__(mp32::THREADS, 2)
    fw_batched_persistent128_f32(float *__restrict__ Dp, int32_t *__restrict__ Pp,
                                 const int32_t *__restrict__ order, const int32_t *__restrict__ ns,
                                 const int64_t *__restrict__ offs, int num, int *__restrict__ counter,
                                 unsigned char *__restrict__ scratch, int rmax) {
  persistent_body<true>(Dp, Pp, order, ns, offs, num, counter, scratch, rmax);
}

int take_device_error_batched() { return take_tu_device_error(); }

}  // namespace apsp

struct apsp_batched_plan {
  int32_t num;
  int32_t *d_order;
  int32_t *d_n;
  int64_t *d_off;
  int *d_counter;
  int grid;
  unsigned char *d_scratch;  // panels of the 128-block variants (grid CTAs), or NULL
  int rmax;                  // blocks per side of the largest graph that uses them
};

namespace {

int validate(const int32_t *h_n, const int64_t *h_off, int32_t num) {
  if (num < 0 || (num > 0 && (!h_n || !h_off))) return APSP_EINVAL;
  if (num > (1 << 30)) return APSP_EUNSUPPORTED;
  for (int32_t g = 0; g < num; ++g) {
    if (h_n[g] < 1 || h_n[g] > apsp::kBatchedMaxN) return h_n[g] < 1 ? APSP_EINVAL : APSP_EUNSUPPORTED;
    if (h_off[g] < 0 || (h_off[g] & 3)) return APSP_EINVAL;
  }
  return APSP_OK;
}

// Largest graphs first (longest processing time first); each entry carries
// the variant of its size class in bits 30-31.  *rmax: blocks per side (of
// 128) of the largest graph given a 128-block variant, 0 if none is.
std::vector<int32_t> lpt_order(const int32_t *h_n, int32_t num, int *rmax) {
  std::vector<int32_t> order(num);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return h_n[a] > h_n[b]; });
  *rmax = 0;
  for (auto &g : order) {
    const int v = apsp::g_variant[apsp::class_of(h_n[g])];
    if (v >= 2) *rmax = std::max(*rmax, (h_n[g] + apsp::kT128 - 1) / apsp::kT128);
    g |= v << 30;
  }
  return order;
}

int g_smem_batched[64], g_smem_batched128[64];

using PersistentKernel = void (*)(float *, int32_t *, const int32_t *, const int32_t *, const int64_t *, int, int *,
                                  unsigned char *, int);

PersistentKernel kernel_for(bool with128) {
  return with128 ? apsp::fw_batched_persistent128_f32 : apsp::fw_batched_persistent_f32;
}

// Grid of the persistent launch: every SM filled with resident CTAs.
int grid_for(int32_t num, bool with128) {
  int dev = 0, sms = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  const PersistentKernel k = kernel_for(with128);
  if (apsp::ensure_smem(k, (int)sizeof(apsp::BatchedSmem), with128 ? g_smem_batched128 : g_smem_batched))
    return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, apsp::mp32::THREADS, sizeof(apsp::BatchedSmem)) !=
      cudaSuccess)
    return -1;
  const int g = sms * std::max(occ, 1);
  return std::max(1, std::min<int>(g, num));
}

}  // namespace

APSP_EXPORT int apsp_batched_plan_create(const int32_t *h_n, const int64_t *h_off, int32_t num,
                                         apsp_batched_plan **out_plan) {
  if (!out_plan) return APSP_EINVAL;
  *out_plan = nullptr;
  int st = validate(h_n, h_off, num);
  if (st) return st;
  apsp_batched_plan *p = (apsp_batched_plan *)calloc(1, sizeof(apsp_batched_plan));
  if (!p) return APSP_ENOMEM;
  p->num = num;
  const size_t cnt = (size_t)std::max(num, 1);
  if (cudaMalloc(&p->d_order, cnt * 4) != cudaSuccess || cudaMalloc(&p->d_n, cnt * 4) != cudaSuccess ||
      cudaMalloc(&p->d_off, cnt * 8) != cudaSuccess || cudaMalloc(&p->d_counter, 4) != cudaSuccess) {
    apsp_batched_plan_destroy(p);
    return APSP_ENOMEM;
  }
  if (num > 0) {
    std::vector<int32_t> order = lpt_order(h_n, num, &p->rmax);
    if (cudaMemcpy(p->d_order, order.data(), (size_t)num * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(p->d_n, h_n, (size_t)num * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(p->d_off, h_off, (size_t)num * 8, cudaMemcpyHostToDevice) != cudaSuccess) {
      apsp_batched_plan_destroy(p);
      return APSP_ECUDA;
    }
  }
  p->grid = grid_for(num, p->rmax > 0);
  if (p->grid < 0) {
    apsp_batched_plan_destroy(p);
    return APSP_ECUDA;
  }
  if (p->rmax > 0 &&
      cudaMalloc(&p->d_scratch, (size_t)p->grid * apsp::panel_bytes_per_cta(p->rmax)) != cudaSuccess) {
    cudaGetLastError();
    apsp_batched_plan_destroy(p);
    return APSP_ENOMEM;
  }
  *out_plan = p;
  return APSP_OK;
}

APSP_EXPORT int apsp_batched_plan_destroy(apsp_batched_plan *p) {
  if (!p) return APSP_OK;
  cudaFree(p->d_order);
  cudaFree(p->d_n);
  cudaFree(p->d_off);
  cudaFree(p->d_counter);
  cudaFree(p->d_scratch);
  free(p);
  return APSP_OK;
}

APSP_EXPORT int apsp_fw_batched_run_f32(const apsp_batched_plan *p, float *d_dist, int32_t *d_path,
                                        void *stream) {
  if (!p) return APSP_EINVAL;
  if (p->num == 0) return APSP_OK;
  if (!d_dist) return APSP_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaGetLastError();
  if (cudaMemsetAsync(p->d_counter, 0, sizeof(int), s) != cudaSuccess) return APSP_ECUDA;
  kernel_for(p->rmax > 0)<<<p->grid, apsp::mp32::THREADS, sizeof(apsp::BatchedSmem), s>>>(
      d_dist, d_path, p->d_order, p->d_n, p->d_off, p->num, p->d_counter, p->d_scratch, p->rmax);
  return apsp::status_from(cudaGetLastError());
}

APSP_EXPORT int apsp_fw_batched_f32(float *d_dist, int32_t *d_path, const int32_t *h_n,
                                    const int64_t *h_off, int32_t num, void *stream) try {
  int st = validate(h_n, h_off, num);
  if (st) return st;
  if (num == 0) return APSP_OK;
  if (!d_dist) return APSP_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // A graph would replay the upload of the work list from host memory of this
  // call, which is gone by then.
  bool capturing = false;
  if ((st = apsp::stream_capturing(s, &capturing))) return st;
  if (capturing) return APSP_ECUDA;
  int rmax = 0;
  std::vector<int32_t> order = lpt_order(h_n, num, &rmax);
  int grid = grid_for(num, rmax > 0);
  if (grid <= 0) return APSP_ECUDA;
  // One scratch block: counter | order | n | offsets | panels of the 128-block
  // variants.  The work list, its counter already zero, goes up in one copy.
  const size_t list_bytes = 16 + (((size_t)num * 8 + 15) & ~(size_t)15) + (size_t)num * 8;
  const size_t list_span = (list_bytes + 255) & ~(size_t)255;
  std::vector<char> list(list_bytes, 0);
  int32_t *l_order = reinterpret_cast<int32_t *>(list.data() + 16);
  std::copy(order.begin(), order.end(), l_order);
  std::copy(h_n, h_n + num, l_order + num);
  memcpy(list.data() + list_bytes - (size_t)num * 8, h_off, (size_t)num * 8);
  const size_t bytes = list_span + (rmax > 0 ? (size_t)grid * apsp::panel_bytes_per_cta(rmax) : 0);
  char *scratch = nullptr;
  cudaGetLastError();
  if (apsp::scratch_alloc((void **)&scratch, bytes, s) != cudaSuccess) {
    cudaGetLastError();
    return APSP_ENOMEM;
  }
  unsigned char *panels = rmax > 0 ? reinterpret_cast<unsigned char *>(scratch + list_span) : nullptr;
  int *d_counter = reinterpret_cast<int *>(scratch);
  int32_t *d_order = reinterpret_cast<int32_t *>(scratch + 16);
  int32_t *d_n = d_order + num;
  int64_t *d_off = reinterpret_cast<int64_t *>(scratch + list_bytes - (size_t)num * 8);
  cudaError_t e = cudaMemcpyAsync(scratch, list.data(), list_bytes, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    kernel_for(rmax > 0)<<<grid, apsp::mp32::THREADS, sizeof(apsp::BatchedSmem), s>>>(
        d_dist, d_path, d_order, d_n, d_off, num, d_counter, panels, rmax);
    e = cudaGetLastError();
  }
  // Copies from pageable host memory have consumed their sources when they
  // return, so `list` may go out of scope; the scratch is freed in stream order.
  cudaFreeAsync(scratch, s);
  return apsp::status_from(e);
} catch (const std::exception &) {  // host memory for the work list (nothing enqueued yet)
  return APSP_ENOMEM;
}

APSP_EXPORT int apsp_batched_num_classes(void) { return apsp::kNumClasses; }

APSP_EXPORT int apsp_batched_class_bounds(int cls, int32_t *lo, int32_t *hi) {
  if (cls < 0 || cls >= apsp::kNumClasses || !lo || !hi) return APSP_EINVAL;
  *lo = apsp::kClassLo[cls];
  *hi = apsp::kClassHi[cls];
  return APSP_OK;
}

APSP_EXPORT int apsp_batched_num_variants(int cls) {
  return (cls < 0 || cls >= apsp::kNumClasses) ? 0 : apsp::kNumVariants;
}

APSP_EXPORT int apsp_batched_set_variant(int cls, int variant) {
  if (cls < 0 || cls >= apsp::kNumClasses || variant < 0 || variant >= apsp::kNumVariants)
    return APSP_EINVAL;
  apsp::g_variant[cls] = variant;
  return APSP_OK;
}

APSP_EXPORT int apsp_batched_get_variant(int cls) {
  return (cls < 0 || cls >= apsp::kNumClasses) ? -1 : apsp::g_variant[cls];
}

APSP_EXPORT int apsp_batched_variant_info(int variant, int32_t *block, int32_t *tile_rows, int32_t *tile_cols,
                                          int32_t *eager) {
  if (variant < 0 || variant >= apsp::kNumVariants || !block || !tile_rows || !tile_cols || !eager)
    return APSP_EINVAL;
  *block = apsp::kVariantBlock[variant];
  *tile_rows = apsp::kVariantTileRows[variant];
  *tile_cols = apsp::kVariantTileCols[variant];
  *eager = apsp::kVariantEager[variant];
  return APSP_OK;
}

// ---------------------------------------------------------------------------
// No-allocation batched entry point (no counterpart in the paper).
//
// Some callers cannot allocate device memory at call time: a serving loop
// that forbids cudaMalloc on its hot path, code whose device memory comes
// from an allocator CUDA does not own, or a library embedded where any hidden
// allocation is an error.  This entry point takes the work list (counter,
// largest-first order, sizes, offsets) from one file-scope device array of
// fixed size instead of allocating it, and builds the order on the GPU, so it
// allocates nothing, on the device or on the host.
//
// The array (1 MiB + 16 bytes, up to kNoAllocMaxGraphs graphs) is held by
// every GPU that loads the library until the process exits.  Host code cannot
// pass the array's name to a kernel (in host code it is only a stand-in, not
// a device address): every call looks its address up with
// cudaGetSymbolAddress while the caller's device is current.  The first call
// on a device also loads the library's module there, so it should come
// before any stream capture on that device.  All calls
// share the array and it keeps the previous call's contents; each call
// resets the counter it needs.  Calls that overlap on the GPU (other streams,
// other host threads) race on the array and must be serialised by the caller.
// ---------------------------------------------------------------------------
namespace apsp {

constexpr int kNoAllocMaxGraphs = 65536;
constexpr size_t kNoAllocBytes = 16 + (size_t)kNoAllocMaxGraphs * (4 + 4 + 8);
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// One CTA: counting sort of the graphs by decreasing size (ties in any
// order), each entry tagged with its class's variant; also resets the work
// counter.
__global__ void __launch_bounds__(1024)
    fw_batched_order(const int32_t *__restrict__ ns, int num, int32_t *__restrict__ order,
                     int *__restrict__ counter, int v0, int v1, int v2, int v3) {
  __shared__ int start[kBatchedMaxN + 2];
  for (int v = threadIdx.x; v < kBatchedMaxN + 2; v += blockDim.x) start[v] = 0;
  __syncthreads();
  for (int g = threadIdx.x; g < num; g += blockDim.x) atomicAdd(&start[ns[g]], 1);
  __syncthreads();
  if (threadIdx.x == 0) {  // exclusive scan from the largest size down
    int run = 0;
    for (int v = kBatchedMaxN; v >= 1; --v) {
      const int c = start[v];
      start[v] = run;
      run += c;
    }
    *counter = 0;
  }
  __syncthreads();
  const int var[kNumClasses] = {v0, v1, v2, v3};
  for (int g = threadIdx.x; g < num; g += blockDim.x) {
    const int n = ns[g];
    order[atomicAdd(&start[n], 1)] = g | (var[class_of_n(n)] << 30);
  }
}

}  // namespace apsp

APSP_EXPORT int apsp_fw_batched_f32_noalloc(float *d_dist, int32_t *d_path, const int32_t *h_n,
                                            const int64_t *h_off, int32_t num, void *stream) {
  int st = validate(h_n, h_off, num);
  if (st) return st;
  if (num > apsp::kNoAllocMaxGraphs) return APSP_EUNSUPPORTED;
  if (num == 0) return APSP_OK;
  if (!d_dist) return APSP_EINVAL;
  // The array's device address on the current device, looked up on every call
  // (cheap, allocates nothing) so that it stays right after a device reset
  // reloads the module.  The first call on a device loads the module there.
  void *ptr = nullptr;
  if (cudaGetSymbolAddress(&ptr, apsp::g_noalloc_scratch) != cudaSuccess || !ptr) {
    cudaGetLastError();
    return APSP_ECUDA;
  }
  unsigned char *base = static_cast<unsigned char *>(ptr);
  int *d_counter = reinterpret_cast<int *>(base);
  int32_t *d_order = reinterpret_cast<int32_t *>(base + 16);
  int32_t *d_n = d_order + apsp::kNoAllocMaxGraphs;
  int64_t *d_off = reinterpret_cast<int64_t *>(d_n + apsp::kNoAllocMaxGraphs);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int grid = grid_for(num, false);
  if (grid <= 0) return APSP_ECUDA;
  cudaGetLastError();
  cudaError_t e = cudaMemcpyAsync(d_n, h_n, (size_t)num * 4, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_off, h_off, (size_t)num * 8, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return APSP_ECUDA;
  // The 128-block variant needs per-CTA panel space this entry point does not
  // have: its classes run the 64-block variant with the same path tracking.
  int v[apsp::kNumClasses];
  for (int c = 0; c < apsp::kNumClasses; ++c) v[c] = apsp::g_variant[c] == 2 ? 1 : apsp::g_variant[c];
  apsp::fw_batched_order<<<1, 1024, 0, s>>>(d_n, num, d_order, d_counter, v[0], v[1], v[2], v[3]);
  apsp::fw_batched_persistent_f32<<<grid, apsp::mp32::THREADS, sizeof(apsp::BatchedSmem), s>>>(
      d_dist, d_path, d_order, d_n, d_off, num, d_counter, nullptr, 0);
  return apsp::status_from(cudaGetLastError());
}
