// Single-graph blocked Floyd-Warshall for sm_103a.
//
// Schedule (§2.2 "Blocked FW Algorithm", kernels as in §3.2): the n x n
// matrix is cut into TB x TB blocks; each of the R = ceil(n / TB) rounds runs
//   K1  fw_phase1_diag      phase 1: the diagonal block (r,r), k sequential;
//   K2  fw_phase2_lines     phases 2+3: the row blocks (r,J) and the column
//                           blocks (I,r), k sequential inside each block;
//   K3  fw_phase3_small     phase 4: every other block (I,J) gets
//                           C = min(C, A (x) B) with A = block (I,r) and
//                           B = block (r,J), a min-plus product over the
//                           round's TB values of k.
// Relaxation rule: Algorithm 1 with a strict "<" (see apsp_fw.h).
//
// Rounds overlap: what round r+1 waits for (phase 4 of round r on row and
// column r+1, then K1 and K2 of round r+1) runs on a second stream of higher
// priority beside the rest of round r's phase 4.
//
// Differences from the Pascal design of §3.2 (one output per thread, TB <= 32):
//  * K3 pairs consecutive k: one packed add.rn.f32x2 forms the two candidates
//    of an output and one three-input min.f32 folds both into the accumulator
//    (FADD2 and FMNMX3 run on different pipes).  A CTA takes a 32- or 64-row
//    piece of a block, operands by bulk copy.
//  * Path state: the pieces note once per 16 k which outputs fell, and the k of
//    an improved output is found afterwards among its last 16: exactly that of
//    the sequential loop (ascending k, strict "<" keeps the first k reaching the
//    final minimum).
//  * From round 8 on (n > 2688) a bf16 product on the tensor cores finds the
//    outputs that may improve, and only those are relaxed.
//  * K1 is one cluster of eight CTAs, K2 keeps each row/column line in
//    registers; both keep only minima per step and settle P afterwards.
//  * Nothing reads P: K1/K2/K3 write P only where D strictly improved.
#include <stddef.h>
#include <stdint.h>

#include <algorithm>

#include "common.cuh"
#include "scratch.h"
#include "bulk.cuh"
#include "minplus_f32.cuh"
#include "phases_f32.cuh"
#include "profile.h"
#include "rounds.cuh"
#include "screen.cuh"

namespace apsp {

// --------------------------------------------------------------------------
// K0: P := -1 over an n x n region with leading dimension ld, but for its
// first skip x skip block.
// --------------------------------------------------------------------------
__global__ void fw_path_init(int32_t *__restrict__ P, int64_t n, int64_t ld, int64_t skip) {
  const int64_t total = n * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / n, j = e - i * n;
    if (i >= skip || j >= skip) P[i * ld + j] = -1;
  }
}

// Alignment of the caller's matrices: every row of D (of P) starts on a
// 16-byte boundary.
constexpr int kVecD = 1, kVecP = 2;

constexpr int kScreenParts = 4;  // parts of a block K2 reports on in a screened round

// The closed diagonal block of a round in K2's operand layouts (K1 writes them).
struct DiagOps {
  unsigned long long *A, *B;
};

// __byte_perm selector that replaces byte c of its first operand with byte 0 of its second.
__device__ __forceinline__ constexpr unsigned byte_sel(int c) {
  return 0x3210 ^ ((0x3210 & (0xF << (4 * c))) ^ (4 << (4 * c)));
}

// --------------------------------------------------------------------------
// K1 (FP32): phase 1, Algorithm 1 on the diagonal block (r,r), by one cluster
// of eight CTAs of four warps.  A warp owns the four rows 4 kq .. 4 kq + 3,
// lane l their columns 4l..4l+3 in registers; the four steps k = 4 kq + s are
// taken together.  The warp owning rows kq brings each to its value at its own
// step and publishes them k-paired in its CTA's history; the CTAs form a ring
// and pass each published quad on (16-byte st.async, counted by the receiver's
// barrier of that quad), so no SM sends more than its share.  Every warp then
// relaxes its rows through the four steps: the pivots of a row come by
// shuffle, are brought to their steps against the quad's own 4 x 4 entries,
// and two packed adds and two three-input mins per element do the rest.
//   hist[kp][j] = (row 2 kp at step 2 kp, row 2 kp + 1 at step 2 kp + 1)
//   hcol[i][kp] = (column 2 kp of row i at its step, column 2 kp + 1 likewise)
// Step k never changes row or column k (D[k][k] = 0), so these are the values
// the sequential loop uses.  Only minima are kept in the loop; with a path
// matrix the element is compared once per 16 steps (strictly lower: the last
// improvement lies there), and afterwards the first k of those 16 whose
// candidate from the histories equals the final value is the path entry - the
// k of the sequential loop's last strict improvement.
//
// What bounds it: the serial chain of 32 quads (shuffles, a few dependent
// adds and mins, publish, barrier), not arithmetic.  One CTA that keeps the
// block in the registers of 256 threads is bound by its one SM's pipes
// (2.1e6 relaxations: 12 us at the measured pair rate) and a barrier per step.
// Measured per launch between events, n = 1024: 21 us, 25 us with a path
// matrix (such a one-CTA kernel: 39 and 64 us); 0.3 us a quad and about 8 us
// of launch, load and store.  Publishing to all seven peers at once, by
// st.async or by bulk copies, measured 29 and 34 us: the sends hold up the
// owner SM's own shared-memory accesses.  Two rows a warp: 23 us.
//
// Also writes the final block as K2's operands: diagA[kp][i] = (D[i][2kp],
// D[i][2kp+1]), diagB[kp][j] = (D[2kp][j], D[2kp+1][j]), +inf past n.
// --------------------------------------------------------------------------
namespace k1 {
constexpr int T = mp32::T, CTAS = 8, WARPS = 4, ROWS = T / CTAS, PAIRS = T / 2, QUADS = T / 4;
struct Smem {
  unsigned long long hist[PAIRS][T];
  unsigned long long hcol[ROWS][PAIRS];
  uint64_t bar[QUADS];
};
}  // namespace k1

template <bool PATH>
__global__ void __cluster_dims__(k1::CTAS, 1, 1) __launch_bounds__(32 * k1::WARPS, 1)
    fw_phase1_diag_f32(float *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int vec,
                       int first, DiagOps ops, unsigned *range) {
  using namespace k1;
  using mp32::pack2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const int base = r * T, m = min(T, n - base), nquad = (m + 3) / 4;
  const int cta = (int)cluster_cta_rank(), tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int own = cta * WARPS + w;  // this warp's row quad
  const int i0 = 4 * own, j0 = 4 * lane;
  const float INF = inf<float>();
  // A quad another CTA owns completes its barrier here by its 2 KiB; the
  // quads owned here use the CTA barrier instead.
  if (tid < QUADS) {
    mbar_init(&sm.bar[tid], 1);
    fence_mbar_init();
    if (tid / WARPS != cta) mbar_expect_tx(&sm.bar[tid], 4 * T * 4);
  }
  float d[4][4];
#pragma unroll
  for (int rr = 0; rr < 4; ++rr) {
    const float *row = D + (int64_t)(base + i0 + rr) * ld + base;
#pragma unroll
    for (int c = 0; c < 4; ++c) d[rr][c] = INF;
    if (i0 + rr < m) {
      if ((vec & kVecD) && j0 + 3 < m) {
        const float4 t = *reinterpret_cast<const float4 *>(row + j0);
        d[rr][0] = t.x, d[rr][1] = t.y, d[rr][2] = t.z, d[rr][3] = t.w;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (j0 + c < m) d[rr][c] = row[j0 + c];
      }
    }
  }
  cluster_sync();  // every barrier of the cluster is set up before anyone publishes
  float prev[4][4];   // the elements at the start of the current 16 steps (without P: the input)
  unsigned chunk[4];  // PATH: byte c: last group of 16 steps that lowered element c, 0xFF none
#pragma unroll
  for (int rr = 0; rr < 4; ++rr) {
    chunk[rr] = 0xFFFFFFFFu;
#pragma unroll
    for (int c = 0; c < 4; ++c) prev[rr][c] = d[rr][c];
  }
  bool ok = true;
  const unsigned next = (unsigned)(cta + 1) % CTAS;
  const uint32_t next_base = cluster_map(smem_addr(smem_raw), next) - smem_addr(smem_raw);
#pragma unroll 1
  for (int kq = 0; kq < nquad; ++kq) {
    const int g = kq / WARPS;  // the owning CTA
    // The rows' values at the quad's columns, before its steps.
    float x[4][4];
#pragma unroll
    for (int rr = 0; rr < 4; ++rr)
#pragma unroll
      for (int c = 0; c < 4; ++c) x[rr][c] = __shfl_sync(kFullMask, d[rr][c], kq);
    // e: row 4 kq + s at its step, at the quad's column t > s.
    float e01, e02, e03, e12, e13, e23;
    unsigned long long ha[4], hb[4];  // this lane's columns: rows (0, 1) and (2, 3) of the quad
    auto pivots = [&](float (&p)[4]) {  // a row's pivots brought to their steps
      p[1] = fminf(p[1], __fadd_rn(p[0], e01));
      p[2] = mp32::min3f(p[2], __fadd_rn(p[0], e02), __fadd_rn(p[1], e12));
      p[3] = fminf(mp32::min3f(p[3], __fadd_rn(p[0], e03), __fadd_rn(p[1], e13)), __fadd_rn(p[2], e23));
    };
    const bool mine = kq == own;
    if (mine) {  // warp-uniform
      e01 = x[0][1], e02 = x[0][2], e03 = x[0][3];
      e12 = fminf(x[1][2], __fadd_rn(x[1][0], e02));
      e13 = fminf(x[1][3], __fadd_rn(x[1][0], e03));
      const float y21 = fminf(x[2][1], __fadd_rn(x[2][0], e01));
      e23 = mp32::min3f(x[2][3], __fadd_rn(x[2][0], e03), __fadd_rn(y21, e13));
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) pivots(x[rr]);
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
        *reinterpret_cast<ulonglong2 *>(&sm.hist[2 * kq][j0 + c]) = make_ulonglong2(ha[c], ha[c + 1]);
        *reinterpret_cast<ulonglong2 *>(&sm.hist[2 * kq + 1][j0 + c]) = make_ulonglong2(hb[c], hb[c + 1]);
      }
    }
    if (cta == g) __syncthreads();
    else if (ok) ok = mbar_spin(&sm.bar[kq], 0);
    if (!mine) {
#pragma unroll
      for (int c = 0; c < 4; c += 2) {
        const ulonglong2 ta = *reinterpret_cast<const ulonglong2 *>(&sm.hist[2 * kq][j0 + c]);
        const ulonglong2 tb = *reinterpret_cast<const ulonglong2 *>(&sm.hist[2 * kq + 1][j0 + c]);
        ha[c] = ta.x, ha[c + 1] = ta.y, hb[c] = tb.x, hb[c + 1] = tb.y;
      }
      const ulonglong2 q0 = *reinterpret_cast<const ulonglong2 *>(&sm.hist[2 * kq][4 * kq]);
      const ulonglong2 q1 = *reinterpret_cast<const ulonglong2 *>(&sm.hist[2 * kq][4 * kq + 2]);
      e01 = __uint_as_float((unsigned)q0.y);
      e02 = __uint_as_float((unsigned)q1.x);
      e03 = __uint_as_float((unsigned)q1.y);
      e12 = __uint_as_float((unsigned)(q1.x >> 32));
      e13 = __uint_as_float((unsigned)(q1.y >> 32));
      e23 = __uint_as_float((unsigned)sm.hist[2 * kq + 1][4 * kq + 3]);
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) pivots(x[rr]);
    }
    if (w == kq % WARPS && next != (unsigned)g) {  // pass the quad on to the next CTA of the ring
      const uint32_t to = next_base + smem_addr(&sm.hist[2 * kq][j0]), bar = next_base + smem_addr(&sm.bar[kq]);
      st_async16(to, ha[0], ha[1], bar);
      st_async16(to + 16, ha[2], ha[3], bar);
      st_async16(to + T * 8, hb[0], hb[1], bar);
      st_async16(to + T * 8 + 16, hb[2], hb[3], bar);
    }
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const unsigned long long xa = pack2(x[rr][0], x[rr][1]), xb = pack2(x[rr][2], x[rr][3]);
      if (PATH && lane == 0)
        *reinterpret_cast<ulonglong2 *>(&sm.hcol[4 * w + rr][2 * kq]) = make_ulonglong2(xa, xb);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        mp32::relax2(d[rr][c], xa, ha[c]);
        mp32::relax2(d[rr][c], xb, hb[c]);
      }
    }
    if (PATH && ((kq & 3) == 3 || kq + 1 == nquad)) {
#pragma unroll
      for (int rr = 0; rr < 4; ++rr)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (d[rr][c] < prev[rr][c]) chunk[rr] = __byte_perm(chunk[rr], (unsigned)(kq >> 2), byte_sel(c));
          prev[rr][c] = d[rr][c];
        }
    }
  }
  __syncwarp();
  if (!ok) report_wait_timeout();  // D and P stay as they are
  if (ok) {
    if (range) {
      unsigned hi = 0u, lo = 0u;
#pragma unroll
      for (int rr = 0; rr < 4; ++rr)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (d[rr][c] < INF) {
            hi = max(hi, fkey(d[rr][c]));
            lo = max(lo, fkey(-d[rr][c]));
          }
      screen_range(range, hi, lo);
    }
    if (ops.A) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 4; c += 2)
          *reinterpret_cast<ulonglong2 *>(&ops.B[(int64_t)(2 * own + h) * T + j0 + c]) =
              make_ulonglong2(pack2(d[2 * h][c], d[2 * h + 1][c]), pack2(d[2 * h][c + 1], d[2 * h + 1][c + 1]));
#pragma unroll
      for (int c = 0; c < 4; c += 2)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<ulonglong2 *>(&ops.A[(int64_t)(2 * lane + c / 2) * T + i0 + 2 * h]) =
              make_ulonglong2(pack2(d[2 * h][c], d[2 * h][c + 1]), pack2(d[2 * h + 1][c], d[2 * h + 1][c + 1]));
    }
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int i = i0 + rr;
      if (i >= m) continue;
      const int64_t row = (int64_t)(base + i) * ld + base;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (j0 + c >= m) continue;
        const unsigned g = (chunk[rr] >> (8 * c)) & 0xFFu;
        if (PATH ? g != 0xFFu : d[rr][c] < prev[rr][c]) D[row + j0 + c] = d[rr][c];
        if (!PATH) continue;
        int k = -1;
        if (g != 0xFFu) {
#pragma unroll
          for (int q = 7; q >= 0; --q) {
            const float2 t = mp32::sum2(sm.hcol[4 * w + rr][8 * g + q], sm.hist[8 * g + q][j0 + c]);
            k = t.y == d[rr][c] ? 16 * (int)g + 2 * q + 1 : k;
            k = t.x == d[rr][c] ? 16 * (int)g + 2 * q : k;
          }
        }
        // the first round's block is not initialised: every entry is written
        if (first || k >= 0) P[row + j0 + c] = k >= 0 ? base + k : -1;
      }
    }
  }
  cluster_sync();  // no CTA leaves while another may still send to its history
  if (!ok) drain_ring(sm.bar, nquad, WARPS, cta);  // nor while one may still arrive
}

// --------------------------------------------------------------------------
// K2 (FP32): phases 2 and 3.  Blocks b < R-1 of the grid cover row block
// (r, J), the others column block (I, r); PARTS CTAs share a block.  Within a
// row block every column evolves on its own, within a column block every row:
//   row block, column j:  own[i][j] = min(own[i][j], diag[i][k] + own[k][j])
//   column block, row i:  own[i][j] = min(own[i][j], own[i][k] + diag[k][j])
// for k ascending over the round's vertices (the diagonal block is final
// after K1).  A warp keeps LINES such lines in registers, lane l holding
// positions 2l, 2l+1, 2l+64, 2l+65 of each.  Steps 2 kp and 2 kp + 1 are taken
// together: the two pivot values come by shuffle, the second is brought to its
// step with one add and min, and each position takes both candidates with one
// packed add against the k-paired diagonal block in shared memory (one bulk
// copy of K1's operands) and one three-input min.  No barrier in the loop.
// Paths as in K1: one comparison per 16 steps in the loop, the k inside the
// last improving 16 settled afterwards from the pivot history in shared
// memory.  The finished blocks are also written, padded with +inf to T x T,
// in the layouts phase 4 reads this round:
//   row block (r,J):    Bpan[J][j/64][kp][j%64] = (own[2kp][j], own[2kp+1][j]),
//                       Bt[J][j][k] = own[k][j]
//   column block (I,r): Apan[I][kp][i] = (own[i][2kp], own[i][2kp+1]),
//                       Acp[I][i][k] = own[i][k]
// Bound: issue and the shuffle-add-min chain of a step pair (latency) where a
// launch has few CTAs, the FP32 pipes where it fills the chip.  Measured per
// launch, n = 1024: 10.5 us, 13.7 us with a path matrix (a compare and two
// selects per relaxation, one step at a time, the block read element by
// element: 29.5 us); with four lines a warp instead of two 13.5 and 20 us
// there, since 56 CTAs leave SMs idle.
// --------------------------------------------------------------------------
namespace k2s {
constexpr int T = mp32::T, THREADS = 256, PAIRS = T / 2;
__host__ __device__ constexpr int parts(int lines) { return T / (THREADS / 32 * lines); }  // CTAs per block
template <int LINES>
struct Smem {
  unsigned long long M[PAIRS][T];  // row block: diagA, column block: diagB
  unsigned long long hist[PAIRS][THREADS / 32 * LINES];
  uint64_t bar;
};
}  // namespace k2s

template <bool PATH, int LINES>
__global__ void __launch_bounds__(k2s::THREADS, 2)
    fw_phase2_lines_f32(float *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, int vec_in,
                        DiagOps ops, Panels pan, Screen scr) {
  using namespace k2s;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  static_assert(LINES == 2 || LINES == 4, "the lines of a position are one 8- or 16-byte access");
  constexpr int PARTS = parts(LINES), CTA_LINES = T / PARTS;
  Smem<LINES> &sm = *reinterpret_cast<Smem<LINES> *>(smem_raw);
  const int b = blockIdx.x / PARTS, part = blockIdx.x % PARTS;
  const bool is_row = b < R - 1;
  int other = is_row ? b : b - (R - 1);
  other += (other >= r);
  const int base_r = r * T, m_r = min(T, n - base_r);
  const int base_o = other * T, m_o = min(T, n - base_o);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const float INF = inf<float>();
  if (tid == 0) {
    mbar_init(&sm.bar, 1);
    fence_mbar_init();
    mbar_expect_tx(&sm.bar, sizeof(sm.M));
    fence_proxy_async_global();
    bulk_g2s(&sm.M[0][0], is_row ? ops.A : ops.B, sizeof(sm.M), &sm.bar);
  }
  const int wl = w * LINES, line0 = part * CTA_LINES + wl;
  // Element (line, pos) of the own block sits at D[g0 + line * sl + pos * sp];
  // slot q of a lane is position 2 lane + (q & 1) + 64 (q >> 1).
  const int64_t g0 = is_row ? (int64_t)base_r * ld + base_o : (int64_t)base_o * ld + base_r;
  const int64_t sl = is_row ? 1 : ld, sp = is_row ? ld : 1;
  float v[LINES][4];
#pragma unroll
  for (int c = 0; c < LINES; ++c)
#pragma unroll
    for (int q = 0; q < 4; ++q) v[c][q] = INF;
  // row blocks: the LINES lines of a position are one access
  const bool whole = line0 + LINES <= m_o, vec = (vec_in & kVecD) && whole;
  const bool vec_out = vec && (!PATH || (vec_in & kVecP));
  if (is_row && vec) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int pos = 2 * lane + (q & 1) + 64 * (q >> 1);
      if (pos < m_r) {
        const float *src = &D[g0 + line0 + pos * sp];
        if constexpr (LINES == 4) {
          const float4 t = *reinterpret_cast<const float4 *>(src);
          v[0][q] = t.x, v[1][q] = t.y, v[2][q] = t.z, v[3][q] = t.w;
        } else {
          const float2 t = *reinterpret_cast<const float2 *>(src);
          v[0][q] = t.x, v[1][q] = t.y;
        }
      }
    }
  } else {
#pragma unroll
    for (int c = 0; c < LINES; ++c)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int line = line0 + c, pos = 2 * lane + (q & 1) + 64 * (q >> 1);
        if (line < m_o && pos < m_r) v[c][q] = D[g0 + line * sl + pos * sp];
      }
  }
  float prev[LINES][4];   // the lines at the start of the current 16 steps
  unsigned chunk[LINES];  // byte q: last group of 16 steps that lowered slot q, 0xFF none
#pragma unroll
  for (int c = 0; c < LINES; ++c) {
    chunk[c] = 0xFFFFFFFFu;
#pragma unroll
    for (int q = 0; q < 4; ++q) prev[c][q] = v[c][q];
  }
  __syncthreads();
  const bool ok = mbar_wait(&sm.bar, 0);
  if (__syncthreads_or(!ok)) {  // the diagonal block never arrived: leave D, P and the panels as they are
    if (tid == 0) give_up(&sm.bar, 0);
    return;
  }
  // Positions 2 kp, 2 kp + 1: slots 2 h, 2 h + 1 of lane kp mod 32, h = kp / 32.
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int src = 8 * g + u, kp = 32 * h + src;
        const ulonglong2 ma = *reinterpret_cast<const ulonglong2 *>(&sm.M[kp][2 * lane]);
        const ulonglong2 mb = *reinterpret_cast<const ulonglong2 *>(&sm.M[kp][64 + 2 * lane]);
        // step 2 kp's diagonal entry for position 2 kp + 1
        const float e = __uint_as_float((unsigned)sm.M[kp][2 * kp + 1]);
        unsigned long long xx[LINES];
#pragma unroll
        for (int c = 0; c < LINES; ++c) {
          const float x0 = __shfl_sync(kFullMask, v[c][2 * h], src);
          const float x1 = fminf(__shfl_sync(kFullMask, v[c][2 * h + 1], src), __fadd_rn(x0, e));
          xx[c] = mp32::pack2(x0, x1);
          mp32::relax2(v[c][0], xx[c], ma.x);
          mp32::relax2(v[c][1], xx[c], ma.y);
          mp32::relax2(v[c][2], xx[c], mb.x);
          mp32::relax2(v[c][3], xx[c], mb.y);
        }
        if (PATH && lane == 0) {
#pragma unroll
          for (int c = 0; c < LINES; c += 2)
            *reinterpret_cast<ulonglong2 *>(&sm.hist[kp][wl + c]) = make_ulonglong2(xx[c], xx[c + 1]);
        }
      }
#pragma unroll
      for (int c = 0; c < LINES; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (PATH) {
            if (v[c][q] < prev[c][q]) chunk[c] = __byte_perm(chunk[c], (unsigned)(4 * h + g), byte_sel(q));
            prev[c][q] = v[c][q];
          }
    }
  }
  __syncwarp();  // lane 0's history writes
  if (!PATH) {  // which positions improved (prev still holds the input)
#pragma unroll
    for (int c = 0; c < LINES; ++c)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (v[c][q] < prev[c][q]) chunk[c] = __byte_perm(chunk[c], 0u, byte_sel(q));
  }
  // The phase-4 panels (padded): position pair hq of a line is k-pair lane + 32 hq.
  const int64_t blk = other;
#pragma unroll
  for (int hq = 0; hq < 2; ++hq) {
    const int kp = lane + 32 * hq;
    unsigned long long *dst = is_row ? &pan.Bpan[((blk * 2 + (line0 >> 6)) * (T / 2) + kp) * (T / 2) + (line0 & 63)]
                                     : &pan.Apan[(blk * (T / 2) + kp) * T + line0];
    float *rows = is_row ? pan.Bt : pan.Acp;
#pragma unroll
    for (int c = 0; c < LINES; c += 2)
      *reinterpret_cast<ulonglong2 *>(dst + c) = make_ulonglong2(mp32::pack2(v[c][2 * hq], v[c][2 * hq + 1]),
                                                                 mp32::pack2(v[c + 1][2 * hq], v[c + 1][2 * hq + 1]));
    if (!scr.EA) continue;  // the rows are the screen's
#pragma unroll
    for (int c = 0; c < LINES; ++c)
      *reinterpret_cast<float2 *>(&rows[(blk * T + line0 + c) * T + 2 * kp]) = make_float2(v[c][2 * hq], v[c][2 * hq + 1]);
  }
  if (scr.EA) {
    const float inv = screen_scale(scr.range);
    uint32_t *E = (is_row ? scr.EB : scr.EA) + blk * (T * T / 2);
    bool whole = true;
#pragma unroll
    for (int c = 0; c < LINES; ++c) {
      const int line = line0 + c;
      const float least = screen_least(v[c][0], v[c][1], v[c][2], v[c][3]);
      float e[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        e[q] = screen_weight(v[c][q], least, inv);
        whole = whole && screen_whole(v[c][q]);
      }
#pragma unroll
      for (int hq = 0; hq < 2; ++hq)  // k = 2 lane + 64 hq, + 1: chunk lane / 4 + 8 hq
        E[line * (T / 2) + (((lane >> 2) + 8 * hq) ^ (line & 7)) * 4 + (lane & 3)] = bf16x2(e[2 * hq], e[2 * hq + 1]);
      if (lane == 0) (is_row ? scr.base_b : scr.base_a)[blk * T + line] = least;
    }
    whole = __syncthreads_and(whole);
    if (tid == 0) (is_row ? scr.whole_b : scr.whole_a)[blk * kScreenParts + part * kScreenParts / PARTS] = whole;
  }
  // D and P where the line improved (such positions lie inside the matrix).
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int pos = 2 * lane + (q & 1) + 64 * (q >> 1);
    unsigned gq[LINES];
    bool all = true;  // every line improved at this position
#pragma unroll
    for (int c = 0; c < LINES; ++c) {
      gq[c] = (chunk[c] >> (8 * q)) & 0xFFu;
      all = all && gq[c] != 0xFFu;
    }
    int k[LINES];
    if (PATH) {
#pragma unroll
      for (int c = 0; c < LINES; ++c) {
        k[c] = 0;
        if (gq[c] == 0xFFu) continue;
#pragma unroll
        for (int u = 7; u >= 0; --u) {
          const int kp = 8 * (int)gq[c] + u;
          const float2 t = mp32::sum2(sm.hist[kp][wl + c], sm.M[kp][pos]);
          k[c] = t.y == v[c][q] ? 2 * kp + 1 : k[c];
          k[c] = t.x == v[c][q] ? 2 * kp : k[c];
        }
      }
    }
    const int64_t gp = g0 + line0 * sl + pos * sp;
    if (is_row && vec_out && all) {
      if constexpr (LINES == 4) {
        *reinterpret_cast<float4 *>(&D[gp]) = make_float4(v[0][q], v[1][q], v[2][q], v[3][q]);
        if (PATH)
          *reinterpret_cast<int4 *>(&P[gp]) = make_int4(base_r + k[0], base_r + k[1], base_r + k[2], base_r + k[3]);
      } else {
        *reinterpret_cast<float2 *>(&D[gp]) = make_float2(v[0][q], v[1][q]);
        if (PATH) *reinterpret_cast<int2 *>(&P[gp]) = make_int2(base_r + k[0], base_r + k[1]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < LINES; ++c)
        if (gq[c] != 0xFFu) {
          D[gp + c * sl] = v[c][q];
          if (PATH) P[gp + c * sl] = base_r + k[c];
        }
    }
  }
}

// --------------------------------------------------------------------------
// K3 (FP32): phase 4 in pieces: one CTA computes a TR x 64 piece of an output
// block (TR = 32 where a launch has few blocks, so that it still uses every SM
// and a CTA's serial time is short; 64 otherwise).  The operands of all 128 k
// come in one go; the old values load while they are under way and start the
// accumulators, so an output improves exactly when its accumulator falls.
// Thread tile 4 x 2 or 4 x 4.  With a path matrix the outputs are compared once
// per 16 k (one compare, one byte permute and one move per 16 relaxations) and
// the k of an improved one is found afterwards among those 16, from the operands
// still in shared memory.
// Bound: the FP32 pipes once a launch fills the chip (52 relax/clk/SM at
// n = 8192 with 32 rows, 56 with 64; a 128 x 64 tile with a two-stage ring 57),
// latency below.  Measured per launch of 13 blocks (n = 1024, row and column
// r+1): 12 us, 17 us with a path matrix; such a 128 x 64 tile 19 and 36 us.
// --------------------------------------------------------------------------
namespace k3s {
constexpr int T = mp32::T, THREADS = 256, TC = 64, PAIRS = T / 2;
__host__ __device__ constexpr int per_block(int tr) { return (T / tr) * (T / TC); }
template <int TR>
struct Smem {
  unsigned long long A[PAIRS][TR];  // A[kp][i] = (A[i][2kp], A[i][2kp+1])
  unsigned long long B[PAIRS][TC];  // B[kp][j] = (B[2kp][j], B[2kp+1][j])
  uint64_t bar;
};
}  // namespace k3s

// Piece `sub` of output block (I, J): all 256 threads, the launch's dynamic
// shared memory from offset 0, its barrier in phase 0.  False if the wait for the
// operands ran out: the CTA must then not set the barrier up again.
template <bool PATH, int TR>
__device__ __forceinline__ bool piece_f32(float *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r,
                                          int I, int J, int sub, int vec_ok, const Panels &pan) {
  using namespace k3s;
  static_assert(TR == 32 || TR == 64, "eight warps of 16 x 16 or 16 x 32 outputs");
  constexpr int CW = TR / 16;  // columns per thread
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem<TR> &sm = *reinterpret_cast<Smem<TR> *>(smem_raw);
  const int si = sub >> 1, hJ = sub & 1;
  const int baseI = I * T + si * TR, baseJ = J * T + hJ * TC, baseK = r * T;
  const int mI = min(TR, n - baseI), mJ = min(TC, n - baseJ), mK = min(T, n - baseK);
  if (mI <= 0 || mJ <= 0) return true;  // past the matrix (uniform exit)
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nkp = (mK + 1) / 2;
  if (tid == 0) {
    mbar_init(&sm.bar, 1);
    fence_mbar_init();
    mbar_expect_tx(&sm.bar, (uint32_t)(nkp * (TR + TC) * 8));
    fence_proxy_async_global();
    bulk_g2s(&sm.B[0][0], pan.Bpan + ((int64_t)J * 2 + hJ) * PAIRS * TC, (uint32_t)(nkp * TC * 8), &sm.bar);
  }
  __syncthreads();
  if (w == 0) {
    const unsigned long long *srcA = pan.Apan + (int64_t)I * PAIRS * T + si * TR;
    fence_proxy_async_global();
    for (int kp = lane; kp < nkp; kp += 32) bulk_g2s(&sm.A[kp][0], srcA + (int64_t)kp * T, TR * 8, &sm.bar);
  }
  // A warp owns 16 x 8 CW outputs; lane (ty, tx) = (l / 8, l % 8) rows
  // 2 ty + (a & 1) + 8 (a >> 1) and columns 2 tx + (c & 1) + 16 (c >> 1) of them.
  constexpr int WC = TC / (8 * CW);  // warps side by side
  const int r0 = (w / WC) * 16 + 2 * (lane >> 3), c0 = (w % WC) * 8 * CW + 2 * (lane & 7);
  float acc[4][CW], prev[4][CW];
  unsigned chunk[CW];  // byte a of chunk[c]: last group of 16 k that lowered output (a, c), 0xFF none
#pragma unroll
  for (int c = 0; c < CW; ++c) chunk[c] = 0xFFFFFFFFu;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int i = r0 + (a & 1) + 8 * (a >> 1);
#pragma unroll
    for (int c = 0; c < CW; c += 2) {
      const int j = c0 + 8 * c;
      const float *src = D + (int64_t)(baseI + i) * ld + baseJ + j;
      float2 t = make_float2(inf<float>(), inf<float>());
      if (i < mI) {
        if (vec_ok && j + 1 < mJ) {
          t = *reinterpret_cast<const float2 *>(src);
        } else {
          if (j < mJ) t.x = src[0];
          if (j + 1 < mJ) t.y = src[1];
        }
      }
      prev[a][c] = acc[a][c] = t.x;
      prev[a][c + 1] = acc[a][c + 1] = t.y;
    }
  }
  __syncwarp();
  const bool ok = mbar_wait(&sm.bar, 0);
  if (__syncthreads_or(!ok)) {  // the operands never arrived: the block stays as it is
    if (tid == 0) give_up(&sm.bar, 0);
    return false;
  }
  if (tid == 0) mbar_inval(&sm.bar);  // its one phase is over: the next piece may set it up again
  auto step = [&](int kp) {
    const ulonglong2 a01 = *reinterpret_cast<const ulonglong2 *>(&sm.A[kp][r0]);
    const ulonglong2 a23 = *reinterpret_cast<const ulonglong2 *>(&sm.A[kp][r0 + 8]);
#pragma unroll
    for (int c = 0; c < CW; c += 2) {
      const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(&sm.B[kp][c0 + 8 * c]);
      mp32::relax2(acc[0][c], a01.x, b.x);
      mp32::relax2(acc[0][c + 1], a01.x, b.y);
      mp32::relax2(acc[1][c], a01.y, b.x);
      mp32::relax2(acc[1][c + 1], a01.y, b.y);
      mp32::relax2(acc[2][c], a23.x, b.x);
      mp32::relax2(acc[2][c + 1], a23.x, b.y);
      mp32::relax2(acc[3][c], a23.y, b.x);
      mp32::relax2(acc[3][c + 1], a23.y, b.y);
    }
  };
  auto note = [&](int g) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        if (acc[a][c] < prev[a][c]) chunk[c] = __byte_perm(chunk[c], (unsigned)g, byte_sel(a));
        prev[a][c] = acc[a][c];
      }
  };
  int g = 0;
#pragma unroll 1
  for (; g < nkp / 8; ++g) {
#pragma unroll
    for (int u = 0; u < 8; ++u) step(8 * g + u);
    if (PATH) note(g);
  }
  if (8 * g < nkp) {  // the last round's remainder
#pragma unroll 1
    for (int kp = 8 * g; kp < nkp; ++kp) step(kp);
    if (PATH) note(g);
  }
  if (!PATH) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        const int i = r0 + (a & 1) + 8 * (a >> 1), j = c0 + 16 * (c >> 1) + (c & 1);
        // (improved outputs lie inside the matrix)
        if (acc[a][c] < prev[a][c]) D[(int64_t)(baseI + i) * ld + baseJ + j] = acc[a][c];
      }
    return true;
  }
  // Each lane takes its own next improved output, so that the warp runs the
  // rest as often as its fullest lane needs and not once per output.
  unsigned left = 0u;  // bit 4 c + a: output (a, c) improved
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < CW; ++c) left |= (((chunk[c] >> (8 * a)) & 0xFFu) != 0xFFu ? 1u : 0u) << (4 * c + a);
#pragma unroll 1
  for (; left; left &= left - 1) {
    const int t = __ffs(left) - 1, a = t & 3, c = t >> 2;
    float x = acc[0][0];
#pragma unroll
    for (int u = 1; u < 4 * CW; ++u) x = t == u ? acc[u & 3][u >> 2] : x;
    unsigned ch = chunk[0];
#pragma unroll
    for (int u = 1; u < CW; ++u) ch = c == u ? chunk[u] : ch;
    const int i = r0 + (a & 1) + 8 * (a >> 1), j = c0 + 16 * (c >> 1) + (c & 1);
    const int gc = (int)((ch >> (8 * a)) & 0xFFu);
    int k = 0;
#pragma unroll
    for (int u = 7; u >= 0; --u) {
      const int kp = min(8 * gc + u, nkp - 1);
      const float2 s = mp32::sum2(sm.A[kp][i], sm.B[kp][j]);
      k = s.y == x ? 2 * kp + 1 : k;
      k = s.x == x ? 2 * kp : k;
    }
    const int64_t e = (int64_t)(baseI + i) * ld + baseJ + j;
    D[e] = x;
    P[e] = baseK + k;
  }
  return true;
}

template <bool PATH, int TR>
__global__ void __launch_bounds__(k3s::THREADS, TR == 32 ? 4 : 3)
    fw_phase3_small_f32(float *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, int vec_ok,
                        Panels pan, int set) {
  constexpr int PER = k3s::per_block(TR);
  int I, J;
  block_of(set, blockIdx.x / PER, r, R, I, J);
  piece_f32<PATH, TR>(D, ld, P, n, r, I, J, blockIdx.x % PER, vec_ok, pan);
}

// The FP32 screen.  Eight lanes settle an output, a warp four: lane s of an
// output adds entries 4 (s + 8 u) + c (u, c < 4) of the row of A and the row of
// B^T, and the minimum and its first k are taken over the lanes - the values and
// the tie rule of the sequential loop.
template <bool PATH, bool PROBE>
__global__ void __launch_bounds__(k3x::THREADS, 4)
    fw_phase3_screen_f32(float *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, int vec_ok,
                         Panels pan, Screen scr, int set) {
  using namespace k3x;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const float INF = inf<float>();
  Tile tile;
  const int count = screen_tile<kScreenParts, PROBE>(sm, tile, n, r, R, scr, set, vec_ok != 0,
                                              [&](int i, int j, int left, auto whole_tile) {
    const float *p = D + (int64_t)i * ld + j;
    if constexpr (decltype(whole_tile)::value) return *reinterpret_cast<const float2 *>(p);
    return make_float2(left > 0 ? p[0] : 0.0f, left > 1 ? p[1] : 0.0f);
  });
  const int baseI = tile.baseI, baseJ = tile.baseJ, baseK = r * T, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float4 *acp = reinterpret_cast<const float4 *>(pan.Acp + (int64_t)baseI * T);
  const float4 *bt = reinterpret_cast<const float4 *>(pan.Bt + (int64_t)baseJ * T);
  const int s8 = lane & 7;
#pragma unroll 1
  for (int g = 4 * w; g < count; g += THREADS / 32 * 4) {
    const int it = g + (lane >> 3), e = sm.list[min(it, count - 1)], i = e / H, j = e % H;
    float *out = D + (int64_t)(baseI + i) * ld + baseJ + j;
    float4 av[4], bv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      av[u] = acp[i * (T / 4) + s8 + 8 * u];
      bv[u] = bt[j * (T / 4) + s8 + 8 * u];
    }
    const float old = *out;
    float c[16], m = INF;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      c[4 * u] = __fadd_rn(av[u].x, bv[u].x);
      c[4 * u + 1] = __fadd_rn(av[u].y, bv[u].y);
      c[4 * u + 2] = __fadd_rn(av[u].z, bv[u].z);
      c[4 * u + 3] = __fadd_rn(av[u].w, bv[u].w);
      m = mp32::min3f(mp32::min3f(m, c[4 * u], c[4 * u + 1]), c[4 * u + 2], c[4 * u + 3]);
    }
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) m = fminf(m, __shfl_xor_sync(kFullMask, m, d));
    const bool better = it < count && m < old;
    if (!__any_sync(kFullMask, better)) continue;
    int k = T;  // this lane's first k that reaches m
    if (PATH) {
#pragma unroll
      for (int u = 3; u >= 0; --u)
#pragma unroll
        for (int q = 3; q >= 0; --q) k = c[4 * u + q] == m ? 4 * (s8 + 8 * u) + q : k;
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) k = min(k, __shfl_xor_sync(kFullMask, k, d));
    }
    if (better && s8 == 0) {
      *out = m;
      if (PATH) P[out - D] = baseK + k;
    }
  }
}

// The tiles the screen listed, relaxed densely: CTAs take 64-row pieces in turn.
template <bool PATH>
__global__ void __launch_bounds__(k3s::THREADS, 3)
    fw_phase3_listed_f32(float *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, int vec_ok,
                         Panels pan, Screen scr, int set) {
  const k3x::Listed listed(scr, set, R);
#pragma unroll 1
  for (int t = blockIdx.x; t < listed.count; t += gridDim.x) {
    const int tile = listed.tile(t);
    int I, J;
    block_of(set, tile / k3x::PER_BLOCK, r, R, I, J);
    fence_proxy_async_smem();
    __syncthreads();  // everyone is done with the previous piece's shared memory
    if (!piece_f32<PATH, 64>(D, ld, P, n, r, I, J, tile % k3x::PER_BLOCK, vec_ok, pan)) return;
  }
}

// Phase timing state (see profile.h).
std::mutex g_prof_mu;
bool g_prof_on = false;
std::vector<PhaseRec> g_prof_recs;
std::vector<cudaEvent_t> g_prof_pool;

// --------------------------------------------------------------------------
// Host side: argument checks and the round loop (all launches on `stream`).
// --------------------------------------------------------------------------
// Largest n: vertex indices and block coordinates stay in 32-bit integers,
// element offsets are 64-bit.  In practice device memory bounds n first
// (FP32 D + P take 8 n^2 bytes: 128 GiB at n = 131072).
constexpr int kMaxN = 1 << 18;

constexpr int kT32 = mp32::T, kT64 = 128;
// Phase 4 by blocks per side R (measured, whole solves, ms): 32-row pieces while
// the whole of phase 4 is about a wave of CTAs or less (n = 2049: 0.96 against 1.02
// with 64 rows, with P 1.35 / 1.41; n = 1024 with P 0.45 / 0.50); 64-row pieces
// otherwise, until the rounds are screened (n = 4096: 32 rows for row and column
// r+1 within 0.3 %).
constexpr int kR32 = 21;
// Phase 4 is screened from round 8 on (5 and 12 rounds: within 2 % at n = 4096
// and 16384; about one output in r + 1 improves in round r of a random graph)
// above 21 blocks a side, where the chain of the next round no longer sets the
// pace.
constexpr int kScreenMinR = 22, kScreenFrom = 8;
// From a round at n = 8192: a tile takes the dense kernel 34 ns (with P 52) and the
// screen 9, 64 settled outputs 2.4 (2.9).  Limits of 9 and 11 without P: 36.6 and 36.3
// ms against 36.3 (n = 8192, U(0, 1)); of 14 and 16 with P 51.9 and 51.4 against 51.4.
constexpr ScreenCost kCost{14, 10}, kCostP{18, 15};
static_assert(kScreenFrom % kProbeRounds == 0, "the first screened round probes");
static_assert(2 * (kScreenMinR - 1) * k2s::parts(4) >= kSms, "a screened round's K2 runs kScreenParts parts");
static int g_smem_k1[2][64], g_smem_k2[2][2][64], g_smem_k3s[2][2][64], g_smem_k3x[2][2][64], g_smem_k3l[2][64];

int run_fw_f64_interval(double *D, int n, int64_t ld, int32_t *P, cudaStream_t s,
                        void (*path_init)(int32_t *, int64_t, int64_t, int64_t, cudaStream_t));
int take_device_error_f64();
int take_device_error_checks();
int take_device_error_int32();
int take_device_error_batched();

static void path_init(int32_t *P, int64_t n, int64_t ld, int64_t skip, cudaStream_t s) {
  const int64_t total = n * n;
  const int blocks = (int)((total + 255) / 256 < 152 * 32 ? (total + 255) / 256 : 152 * 32);
  PhaseScope ps(0, s);
  fw_path_init<<<blocks, 256, 0, s>>>(P, n, ld, skip);
}

static int check_args(const void *D, int64_t n, int64_t ld) {
  if (n < 0 || n > kMaxN) return APSP_EINVAL;
  if (n == 0) return APSP_OK;
  if (!D || ld < n) return APSP_EINVAL;
  return APSP_OK;
}

static int run_fw_f32(float *D, int64_t n64, int64_t ld, int32_t *P, void *stream) {
  int st = check_args(D, n64, ld);
  if (st || n64 == 0) return st;
  const int n = (int)n64;
  constexpr int T = kT32;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int R = (n + T - 1) / T;
  if ((st = ensure_smem(fw_phase1_diag_f32<false>, (int)sizeof(k1::Smem), g_smem_k1[0]))) return st;
  if ((st = ensure_smem(fw_phase1_diag_f32<true>, (int)sizeof(k1::Smem), g_smem_k1[1]))) return st;
  // K2 with two lines a warp while four would not fill the chip.
  const int lines = 2 * (R - 1) * k2s::parts(4) < kSms ? 2 : 4;
  const auto lines_kernel = lines == 2 ? (P ? fw_phase2_lines_f32<true, 2> : fw_phase2_lines_f32<false, 2>)
                                       : (P ? fw_phase2_lines_f32<true, 4> : fw_phase2_lines_f32<false, 4>);
  const int lines_smem = (int)(lines == 2 ? sizeof(k2s::Smem<2>) : sizeof(k2s::Smem<4>));
  if ((st = ensure_smem(lines_kernel, lines_smem, g_smem_k2[lines / 4][P != nullptr]))) return st;
  // Phase 4 in pieces of 32 or 64 rows.
  const auto kernel32 = P ? fw_phase3_small_f32<true, 32> : fw_phase3_small_f32<false, 32>;
  const auto kernel64 = P ? fw_phase3_small_f32<true, 64> : fw_phase3_small_f32<false, 64>;
  if ((st = ensure_smem(kernel32, (int)sizeof(k3s::Smem<32>), g_smem_k3s[0][P != nullptr]))) return st;
  if ((st = ensure_smem(kernel64, (int)sizeof(k3s::Smem<64>), g_smem_k3s[1][P != nullptr]))) return st;
  const auto screen_kernel = P ? fw_phase3_screen_f32<true, false> : fw_phase3_screen_f32<false, false>;
  const auto probe_kernel = P ? fw_phase3_screen_f32<true, true> : fw_phase3_screen_f32<false, true>;
  if ((st = ensure_smem(screen_kernel, (int)sizeof(k3x::Smem), g_smem_k3x[0][P != nullptr])) ||
      (st = ensure_smem(probe_kernel, (int)sizeof(k3x::Smem), g_smem_k3x[1][P != nullptr])) ||
      (st = ensure_smem(P ? fw_phase3_listed_f32<true> : fw_phase3_listed_f32<false>, (int)sizeof(k3s::Smem<64>),
                        g_smem_k3l[P != nullptr])))
    return st;
  cudaGetLastError();  // clear any stale error so the checks below are ours
  // Phase-4 operand panels, written by K2 each round: two sets (round parity)
  // of R*T*T 4-byte words each for Apan and Bpan, and with screened rounds for
  // the rows Acp and Bt, so that K2 of round r+1 can run while phase 4 of round
  // r still reads round r's panels; then K1's two copies of the closed diagonal
  // block.  Stream-ordered scratch, freed after the last round.
  Panels pan[2]{};
  DiagOps ops{};
  char *scratch = nullptr;
  const bool screened = R >= kScreenMinR;
  ScreenSets scr(R, kScreenParts);
  if (R > 1) {
    const size_t words = (size_t)R * T * T, diag = 2 * (size_t)T * T, set = (screened ? 4 : 2) * words;
    const size_t screen_bytes = screened ? 2 * scr.set_bytes() + scr.list_bytes() : 0;
    if (scratch_alloc((void **)&scratch, (2 * set + diag) * 4 + screen_bytes, s) != cudaSuccess) {
      cudaGetLastError();
      return APSP_ENOMEM;
    }
    for (int q = 0; q < 2; ++q) {
      char *base = scratch + (size_t)q * set * 4;
      pan[q].Apan = reinterpret_cast<unsigned long long *>(base);
      pan[q].Bpan = reinterpret_cast<unsigned long long *>(base + words * 4);
      if (!screened) continue;
      pan[q].Acp = reinterpret_cast<float *>(base + 2 * words * 4);
      pan[q].Bt = reinterpret_cast<float *>(base + 3 * words * 4);
    }
    ops.A = reinterpret_cast<unsigned long long *>(scratch + 2 * set * 4);
    ops.B = ops.A + T * T / 2;
    if (screened) {
      char *base = scratch + (2 * set + diag) * 4;
      for (int q = 0; q < 2; ++q, base += scr.set_bytes()) scr.place_set(q, base);
      if (scr.place_lists(base, s) != cudaSuccess) {
        cudaFreeAsync(scratch, s);
        cudaGetLastError();
        return APSP_ECUDA;
      }
    }
  }
  const bool aligned = ld % 4 == 0;
  const int vec = (aligned && (reinterpret_cast<uintptr_t>(D) & 15) == 0 ? kVecD : 0) |
                  (aligned && (reinterpret_cast<uintptr_t>(P) & 15) == 0 ? kVecP : 0);
  const int vec_ok = vec & kVecD;
  bool capturing = false;
  if ((st = stream_capturing(s, &capturing))) {
    if (scratch) cudaFreeAsync(scratch, s);
    return st;
  }
  // The round's screening data, or none where the round is not screened.
  const int probed = set_blocks(capturing ? kSetAll : kSetRest, R);
  auto screen_of = [&](int r) {
    return screened && r >= kScreenFrom ? scr.round(r, kScreenFrom, probed, P ? kCostP : kCost) : Screen{};
  };
  // K1 of round 0 writes all of P's first block; the rest of P is set to -1
  // beside it.
  auto init = [&](cudaStream_t st) {
    if (P) path_init(P, n64, ld, T, st);
  };
  auto diag = [&](int r, cudaStream_t st) {
    PhaseScope ps(1, st);
    (P ? fw_phase1_diag_f32<true> : fw_phase1_diag_f32<false>)<<<k1::CTAS, 32 * k1::WARPS, sizeof(k1::Smem), st>>>(
        D, ld, P, n, r, vec, (int)(P && r == 0), ops, screen_of(r).range);
  };
  auto panels = [&](int r, cudaStream_t st) {
    PhaseScope ps(2, st);
    lines_kernel<<<2 * (R - 1) * k2s::parts(lines), k2s::THREADS, lines_smem, st>>>(D, ld, P, n, r, R, vec, ops,
                                                                                    pan[r & 1], screen_of(r));
  };
  auto phase4 = [&](int r, int set, int blocks, cudaStream_t st) {
    if (blocks <= 0) return;
    const bool screen = screened && r >= kScreenFrom;
    PhaseScope ps(3, st, screen ? 2 : 1);
    if (screen) {
      const Screen sc = screen_of(r);
      (sc.cost ? probe_kernel : screen_kernel)<<<k3x::PER_BLOCK * blocks, k3x::THREADS, sizeof(k3x::Smem), st>>>(
          D, ld, P, n, r, R, vec_ok, pan[r & 1], sc, set);
      (P ? fw_phase3_listed_f32<true> : fw_phase3_listed_f32<false>)<<<std::min(4 * blocks, kListedCtas * kSms),
                                                                       k3s::THREADS, sizeof(k3s::Smem<64>), st>>>(
          D, ld, P, n, r, R, vec_ok, pan[r & 1], sc, set);
    } else if (R <= kR32)
      kernel32<<<k3s::per_block(32) * blocks, k3s::THREADS, sizeof(k3s::Smem<32>), st>>>(D, ld, P, n, r, R, vec_ok,
                                                                                        pan[r & 1], set);
    else
      kernel64<<<k3s::per_block(64) * blocks, k3s::THREADS, sizeof(k3s::Smem<64>), st>>>(D, ld, P, n, r, R, vec_ok,
                                                                                        pan[r & 1], set);
  };
  st = run_rounds(R, s, capturing, init, diag, panels, phase4);
  cudaError_t e = cudaGetLastError();
  if (scratch) {
    cudaError_t f = cudaFreeAsync(scratch, s);
    if (e == cudaSuccess) e = f;
  }
  return st ? st : status_from(e);
}

static int run_fw_f64(double *D, int64_t n64, int64_t ld, int32_t *P, void *stream) {
  int st = check_args(D, n64, ld);
  if (st || n64 == 0) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaGetLastError();
  return run_fw_f64_interval(D, (int)n64, ld, P, s, path_init);
}

}  // namespace apsp

APSP_EXPORT int apsp_fw_f32(float *d_dist, int64_t n, int64_t ld, int32_t *d_path, void *stream) {
  return apsp::run_fw_f32(d_dist, n, ld, d_path, stream);
}

APSP_EXPORT int apsp_fw_f64(double *d_dist, int64_t n, int64_t ld, int32_t *d_path, void *stream) {
  return apsp::run_fw_f64(d_dist, n, ld, d_path, stream);
}

APSP_EXPORT int apsp_fw_block_size(int elem_bytes) {
  return elem_bytes == 4 ? apsp::kT32 : elem_bytes == 8 ? apsp::kT64 : 0;
}

APSP_EXPORT const char *apsp_status_string(int status) {
  switch (status) {
    case APSP_OK: return "APSP_OK";
    case APSP_EINVAL: return "APSP_EINVAL: invalid argument";
    case APSP_ECUDA: return "APSP_ECUDA: CUDA call or launch failed";
    case APSP_ENOMEM: return "APSP_ENOMEM: device allocation failed";
    case APSP_EUNSUPPORTED: return "APSP_EUNSUPPORTED: outside supported sizes";
    case APSP_ETOODEEP: return "APSP_ETOODEEP: path recursion deeper than the walk stack";
    case APSP_ENEGCYCLE: return "APSP_ENEGCYCLE: negative cycle (a diagonal distance is below 0)";
    case APSP_ETIMEOUT: return "APSP_ETIMEOUT: a kernel's bounded wait for an asynchronous copy ran out";
    default: return "APSP: unknown status";
  }
}

APSP_EXPORT int apsp_version(void) { return 100; }

APSP_EXPORT int apsp_profile_enable(int on) {
  std::lock_guard<std::mutex> g(apsp::g_prof_mu);
  if (on) {  // a new recording starts: recycle the old records' events
    for (auto &r : apsp::g_prof_recs) {
      apsp::g_prof_pool.push_back(r.a);
      apsp::g_prof_pool.push_back(r.b);
    }
    apsp::g_prof_recs.clear();
  }
  apsp::g_prof_on = on != 0;
  return APSP_OK;
}

APSP_EXPORT int apsp_profile_collect(double *ms, int64_t *launches) {
  if (!ms || !launches) return APSP_EINVAL;
  for (int p = 0; p < 4; ++p) {
    ms[p] = 0.0;
    launches[p] = 0;
  }
  std::lock_guard<std::mutex> g(apsp::g_prof_mu);
  for (auto &r : apsp::g_prof_recs) {
    if (cudaEventSynchronize(r.b) != cudaSuccess) return APSP_ECUDA;
    float t = 0.f;
    if (cudaEventElapsedTime(&t, r.a, r.b) != cudaSuccess) return APSP_ECUDA;
    ms[r.phase] += t;
    launches[r.phase] += r.launches;
  }
  return APSP_OK;
}

APSP_EXPORT int apsp_profile_records(int32_t *phase, float *ms, int64_t cap, int64_t *count) {
  if (!count || cap < 0 || (cap > 0 && (!phase || !ms))) return APSP_EINVAL;
  std::lock_guard<std::mutex> g(apsp::g_prof_mu);
  int64_t i = 0;
  for (auto &r : apsp::g_prof_recs) {
    if (i < cap) {
      if (cudaEventSynchronize(r.b) != cudaSuccess) return APSP_ECUDA;
      float t = 0.f;
      if (cudaEventElapsedTime(&t, r.a, r.b) != cudaSuccess) return APSP_ECUDA;
      phase[i] = r.phase;
      ms[i] = t;
    }
    ++i;
  }
  *count = i;
  return APSP_OK;
}

APSP_EXPORT int apsp_device_status(void *stream) {
  if (cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess) return APSP_ECUDA;
  const int v = apsp::take_tu_device_error();
  const int v64 = apsp::take_device_error_f64();
  const int vc = apsp::take_device_error_checks();
  const int vi = apsp::take_device_error_int32();
  const int vb = apsp::take_device_error_batched();
  return v != 0 ? v : v64 != 0 ? v64 : vc != 0 ? vc : vi != 0 ? vi : vb;
}
