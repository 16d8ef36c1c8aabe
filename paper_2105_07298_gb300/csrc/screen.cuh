// Phase 4 in rounds where few outputs improve, shared by the FP32 and the FP64
// path.  Internal header.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <type_traits>

#include "bulk.cuh"
#include "common.cuh"
#include "minplus_f32.cuh"
#include "rounds.cuh"

namespace apsp {

// What the screened phase 4 needs of a round besides the panels (all NULL in a
// round that is not screened), see k3x.
//   EA[I][i][k], EB[J][j][k]: bf16 weights of the column and the row panel, 8-k
//     chunks of a line moved to chunk (k / 8) ^ (line % 8);
//   base_a[I][i], base_b[J][j]: the least entry of the line (0 if none is finite);
//   whole_a[I][p], whole_b[J][p]: part p of the block (K2 divides it into PARTS
//     parts, lines in order) holds only integers below 2^21 in magnitude (and +inf);
//   range: of the closed diagonal block, ordered keys of its largest finite
//     entry and of minus its smallest;
//   next, rest: the tiles the screen lists for the dense kernel, by block set, and
//     listed_next, listed_rest: how many;
//   cost: in a probing round, what every kSample-th tile of its rest (or of all, where
//     that is one launch) costs beside the screen itself, in units of 64 settled
//     outputs, `dense` for a listed tile; NULL otherwise;
//   probe: the last probing round's cost (in a probing round that of the one before,
//     NULL in the first): above `enough` this round is relaxed densely without a
//     screen, but for those tiles of a probing round.
struct Screen {
  uint32_t *EA, *EB;
  float *base_a, *base_b;
  int *whole_a, *whole_b;
  unsigned *range;
  int *next, *rest, *listed_next, *listed_rest;
  int *cost;
  const int *probe;
  int dense, enough;
  // Whether the last probe did not pay, and whether the screen is left out.
  __device__ __forceinline__ bool failed() const { return probe && *probe > enough; }
  __device__ __forceinline__ bool skip() const { return !cost && failed(); }
};
// Every eighth round probes.  Where many outputs improve in every round (weights
// down to 0), screening them all costs more than it saves: n = 8192, U(0, 1),
// without P 33.4 ms unscreened, 41.6 with every round screened, 36.3 with these
// probes (37.3 with the number of listed tiles as their measure and no samples; every
// 16 / 32 rounds 38.3 / 39.6 then).  Of what is left over 33.4, 0.9 ms are the screens
// of rounds that go without (their CTAs start, read the probe's cost and end) and
// the dense kernel's CTAs beside them; the chain's kernels find SMs later, too.  A
// probe that follows one that failed takes every eighth tile alone (all of them: 0.15
// ms a probe there, and 36.7); the cost is always added up over these (0.013 ms a
// probe at n = 16384).
constexpr int kProbeRounds = 8, kSample = 8;
// CTAs of the dense kernel per SM of the chip: each takes its pieces in turn, and
// ends early enough that the next round's chain finds room (three per SM, n =
// 4096, U(0, 1): 9.2 ms, twelve 7.8, thirty-two 7.8; n = 16384: 124.3 / 124.5 /
// 124.8).
constexpr int kListedCtas = 12;

// What a tile costs the solve's kernels, in units of 64 settled outputs: relaxed by
// the dense kernel, and the same less the screen itself (a probing round must cost
// less than that beside its screens).
struct ScreenCost {
  int dense, enough;
};

// The scratch of a solve with screened rounds: two sets by round parity (as the
// panels), then the ranges and counts of all rounds and the two lists.
struct ScreenSets {
  size_t R, parts;
  Screen set[2]{};
  unsigned *ranges = nullptr;
  int *listed = nullptr, *costs = nullptr, *next = nullptr, *rest = nullptr;
  ScreenSets(int R, int parts) : R((size_t)R), parts((size_t)parts) {}
  static constexpr size_t kT = mp32::T, kTiles = 4;  // tiles of a block
  size_t set_bytes() const { return (R * kT * kT + 2 * R * kT + 2 * R * parts) * 4; }  // EA, EB: half a word an entry
  size_t list_bytes() const { return (5 * R + kTiles * 2 * R + kTiles * R * R) * 4; }
  void place_set(int q, void *at) {
    Screen &sc = set[q];
    sc.EA = static_cast<uint32_t *>(at);
    sc.EB = sc.EA + R * kT * kT / 2;
    sc.base_a = reinterpret_cast<float *>(sc.EB + R * kT * kT / 2);
    sc.base_b = sc.base_a + R * kT;
    sc.whole_a = reinterpret_cast<int *>(sc.base_b + R * kT);
    sc.whole_b = sc.whole_a + R * parts;
  }
  cudaError_t place_lists(void *at, cudaStream_t s) {
    ranges = static_cast<unsigned *>(at);
    listed = reinterpret_cast<int *>(ranges + 2 * R);
    costs = listed + 2 * R;
    next = costs + R;
    rest = next + kTiles * 2 * R;
    return cudaMemsetAsync(ranges, 0, 5 * R * 4, s);
  }
  // `blocks`: of the set whose cost a probing round adds up.
  // `first`: the first screened round (a probing one).
  Screen round(int r, int first, int blocks, ScreenCost c) const {
    Screen sc = set[r & 1];
    const int at = r - r % kProbeRounds;
    sc.dense = c.dense;
    sc.enough = c.enough * ((int)kTiles * blocks / kSample);
    sc.range = ranges + 2 * r;
    sc.next = next;
    sc.rest = rest;
    sc.listed_next = listed + 2 * r;
    sc.listed_rest = sc.listed_next + 1;
    sc.cost = r == at ? costs + at : nullptr;
    sc.probe = r != at ? costs + at : at > first ? costs + at - kProbeRounds : nullptr;
    return sc;
  }
};

// Unsigned keys with the order of the floats (no NaN), and back.
__device__ __forceinline__ unsigned fkey(float x) {
  const unsigned u = __float_as_uint(x);
  return (u >> 31) ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float fkey_value(unsigned k) { return __uint_as_float((k >> 31) ? k & 0x7fffffffu : ~k); }

// 1 / s of a round, s = (largest - smallest finite entry of the diagonal block) / 96.
__device__ __forceinline__ float screen_scale(const unsigned *range) {
  const unsigned hi = range[0], lo = range[1];
  const float span = hi && lo ? fkey_value(hi) + fkey_value(lo) : 0.0f;
  return span > 0.0f ? fminf(fmaxf(96.0f / span, 1e-30f), 1e30f) : 1e-30f;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The weight of a panel entry (FP64: of its lower bound): at least
// 2^-(x - least) / s, 1/128 above what covers ex2's error and the rounding to bf16.
__device__ __forceinline__ float screen_weight(float x, float least, float inv) {
  return x < inf<float>() ? ex2(-fminf(__fmul_rn(__fsub_rn(x, least), inv), 60.0f)) * 1.0078125f : 0.0f;
}
// The least finite entry of a line, of which a lane holds four; 0 if it has none.
__device__ __forceinline__ float screen_least(float a, float b, float c, float d) {
  const float least = fkey_value(__reduce_min_sync(kFullMask, fkey(fminf(mp32::min3f(a, b, c), d))));
  return least < inf<float>() ? least : 0.0f;
}
__device__ __forceinline__ bool screen_whole(float x) {
  return !(x < inf<float>()) || (x == rintf(x) && fabsf(x) < 2097152.0f);
}
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  uint32_t two;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(two) : "f"(hi), "f"(lo));
  return two;
}
// Adds a warp's entries of the closed diagonal block (keys of the largest
// finite entry and of minus the smallest) to its range.
__device__ __forceinline__ void screen_range(unsigned *range, unsigned hi, unsigned lo) {
  hi = __reduce_max_sync(kFullMask, hi);
  lo = __reduce_max_sync(kFullMask, lo);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&range[0], hi);
    atomicMax(&range[1], lo);
  }
}

// --------------------------------------------------------------------------
// K3 screened: phase 4 in rounds where few outputs improve.  A bf16 product on
// the tensor cores finds the outputs that may improve, and only those are
// relaxed in the solve's own type.
//
// With s > 0 and any bases a_i, b_j, a candidate below the old value, D[i][k] +
// D[k][j] < old, gives 2^-(D[i][k] - a_i)/s * 2^-(D[k][j] - b_j)/s >
// 2^-(old - a_i - b_j)/s =: T.  K2 writes weights at least as large as the two
// factors (the bases are the lines' least entries, so weights are at most about
// 1; entries further than 60 s above get the weight of 60 s, +inf gets 0), so
// the sum X of a row's products over the round's k exceeds T whenever any
// candidate improves.  Outputs with X <= 0.96 T', T' lowered by what rounding
// in its argument can amount to, are left as they are; the FP32 accumulation of
// at most 128 non-negative normal products loses less than the factor covers.
// The other outputs may or may not improve: the test sees a candidate within
// about s log2(how many) of the old value.  Where both blocks hold only
// integers, a candidate below the old value is at most ceil(old) - 1, and with
// s <= 1/8 (128 ties at the old value weigh half of one a step below) the test
// is exact.  In FP64 the panel entries are their lower bounds and the old values
// their upper bounds, which a candidate below the old value is below as well.
//
// Flagged outputs are listed for the caller, which settles them four to a warp,
// eight lanes each.  A tile with more than kScreenDense of them is listed for
// the dense kernel of the type.
//
// Bound: the latency of a tile's loads (weights, old values, then the flagged
// outputs' rows), overlapped over four CTAs per SM; a tile of 128 x 64 with two
// CTAs measured 8 % slower, settling one output a warp 25 %, a test with twice the
// instructions per output 1.7 % (n = 16384: 120.9 against 118.9 ms).  Measured per round
// in FP32 at n = 16384 (U[1, 100], p = 0.5): 0.64 ms from round 60 on, of which
// the screen 0.58 (the dense kernel 2.0 ms); the product itself 0.22 ms on
// mma.sync with 128 x 128 tiles, so its rate is not what counts.  FP32 solves
// with P: n = 4096 6.2 -> 4.6 ms, 8192 42.3 -> 22.5, 16384 289 -> 119; real
// weights and sparse graphs gain likewise (n = 8192: U[0.5, 2) 41.8 -> 22.3 ms, 16
// edges a vertex 46.5 -> 38.9).  FP64: n = 4096 9.8 -> 8.6 ms, 6000 27.3 -> 20.2.
// --------------------------------------------------------------------------
namespace k3x {
constexpr int T = mp32::T, THREADS = 256;
constexpr int H = T / 2, PER_BLOCK = ScreenSets::kTiles;  // a CTA's tile: H x H, a quarter of a block
constexpr int kScreenDense = 800;  // of H H outputs (FP32 with P: 625, 800, 1000 within 1 %; without P 500 is 4 %
                                   // slower at n = 16384; FP64: 400 within 1 %, 200 4 % slower at n = 4096)
struct Smem {
  uint32_t EA[H][T / 2], EB[H][T / 2];
  float base_a[H], base_b[H];  // adjacent; base_b is read in pairs
  uint64_t bar;
  int count, next;
  unsigned short list[kScreenDense];  // flagged outputs, i H + j
};
static_assert(offsetof(Smem, base_b) % 8 == 0 && offsetof(Smem, EB) % 128 == 0, "pairs and bulk copies");
__device__ __forceinline__ void ldmatrix4(uint32_t (&f)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct Tile {
  int I, J, baseI, baseJ;  // block, first row and column of the H x H outputs
};

// Leaves this CTA's tile to the dense kernel.
__device__ __forceinline__ void list_tile(const Screen &scr, int set) {
  const bool nx = set == kSetNext;
  (nx ? scr.next : scr.rest)[atomicAdd(nx ? scr.listed_next : scr.listed_rest, 1)] = blockIdx.x;
}

// One CTA screens its tile: returns how many of its outputs are in sm.list, for
// the caller to settle; 0 if there are none or the tile was listed for the dense
// kernel.  old(i, j, left, whole_tile): the values (FP64: upper bounds) of outputs
// (i, j) and (i, j + 1), anything where `left` columns of the matrix end before
// them; whole_tile: a std::true_type says that they lie inside it, aligned (pairs).
// PROBE: of a probing round (an instance of its own: with its tests in the one
// kernel n = 16384 with P, integers, took 119.6 ms against 118.9).
template <int PARTS, bool PROBE, typename Old>
__device__ __forceinline__ int screen_tile(Smem &sm, Tile &t, int n, int r, int R, const Screen &scr, int set, bool pairs,
                                           Old old) {
  block_of(set, blockIdx.x / PER_BLOCK, r, R, t.I, t.J);
  const int I = t.I, J = t.J;
  const int hI = (blockIdx.x >> 1) & 1, hJ = blockIdx.x & 1;
  const int baseI = t.baseI = I * T + hI * H, baseJ = t.baseJ = J * T + hJ * H;
  const int mI = min(H, n - baseI), mJ = min(H, n - baseJ);
  if (mI <= 0 || mJ <= 0) return 0;  // past the matrix (uniform exit)
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const float INF = inf<float>();
  if (tid == 0) {
    mbar_init(&sm.bar, 1);
    fence_mbar_init();
    mbar_expect_tx(&sm.bar, 2 * H * T * 2);
    sm.count = sm.next = 0;
  }
  if (scr.failed() && (!PROBE || blockIdx.x % kSample)) {  // (uniform)
    if (PROBE && tid == 0) list_tile(scr, set);
    return 0;
  }
  if (tid == 0) {
    fence_proxy_async_global();
    bulk_g2s(&sm.EA[0][0], scr.EA + (int64_t)I * (T * T / 2) + hI * (H * T / 2), H * T * 2, &sm.bar);
    bulk_g2s(&sm.EB[0][0], scr.EB + (int64_t)J * (T * T / 2) + hJ * (H * T / 2), H * T * 2, &sm.bar);
  }
  // Warp (w / 4, w % 4): rows wi .. wi + 31, columns wj .. wj + 15.  Output (a, h,
  // b, q) of lane l: row wi + 16 a + 8 h + l / 4, column wj + 8 b + 2 (l % 4) + q.
  // The old values are under way while the weights arrive and are multiplied.
  const int wi = 32 * (w >> 2), wj = 16 * (w & 3);
  const bool full = mI == H && mJ == H;
  float2 o[2][2][2];
  auto load = [&](auto whole_tile) {
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = wi + 16 * a + 8 * h + (lane >> 2);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const int j = wj + 8 * b + 2 * (lane & 3);
          o[a][h][b] = decltype(whole_tile)::value || i < mI ? old(baseI + i, baseJ + j, mJ - j, whole_tile) : make_float2(0.0f, 0.0f);
        }
      }
  };
  if (full && pairs) load(std::true_type{});
  else load(std::false_type{});
  const float inv = screen_scale(scr.range);
  if (tid < 2 * H) {  // the bases in units of s, less their share of the argument's error
    const float v = tid < H ? scr.base_a[I * T + hI * H + tid] : scr.base_b[J * T + hJ * H + tid - H];
    const float b = fmaf(v, inv, -fabsf(v) * (4.76837158203125e-7f * inv) - 0.03f);
    (&sm.base_a[0])[tid] = fabsf(b) < 1e38f ? b : -INF;  // beyond the floats: the line's outputs are all flagged
  }
  bool whole = true;
#pragma unroll
  for (int p = 0; p < PARTS / 2; ++p)
    whole = whole && scr.whole_a[I * PARTS + hI * (PARTS / 2) + p] && scr.whole_b[J * PARTS + hJ * (PARTS / 2) + p];
  __syncthreads();
  const bool ok = mbar_wait(&sm.bar, 0);
  if (__syncthreads_or(!ok)) {  // the weights never arrived: the block stays as it is
    if (tid == 0) give_up(&sm.bar, 0);
    return 0;
  }
  float x[2][2][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) x[a][b][c] = 0.0f;
  const uint32_t sa = smem_addr(&sm.EA[0][0]), sb = smem_addr(&sm.EB[0][0]);
  const int ar = wi + (lane & 15), ac = lane >> 4;                       // A: row, chunk
  const int br = wj + (lane & 7) + 8 * (lane >> 4), bc = (lane >> 3) & 1;  // B: line, chunk
#pragma unroll
  for (int ks = 0; ks < T / 16; ++ks) {
    uint32_t fb[4];
    ldmatrix4(fb, sb + (uint32_t)(br * (T * 2) + (((2 * ks + bc) ^ (br & 7)) << 4)));
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      uint32_t fa[4];
      ldmatrix4(fa, sa + (uint32_t)((ar + 16 * a) * (T * 2) + (((2 * ks + ac) ^ (ar & 7)) << 4)));
      mma_bf16(x[a][0], fa, fb[0], fb[1]);
      mma_bf16(x[a][1], fa, fb[2], fb[3]);
    }
  }
  // log2(0.96 T') = (a_i + b_j - t) / s, less what its roundings and ex2's can
  // amount to: the bases have 2^-21 of a_i / s and b_j / s taken off, and 0.06,
  // and t / s only enters a fused multiply-add, whose own rounding is within
  // 2^-24 of the result: nothing below 2^-200, where T' is 0, needs more.
  unsigned mine[2][2];  // [a][h]: bit 2 b + q
  int found = 0;
  auto test = [&](auto limit) {  // limit(old): the largest value a candidate below old can have
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        mine[a][h] = 0u;
        const float ai = sm.base_a[wi + 16 * a + 8 * h + (lane >> 2)];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const float2 bj = *reinterpret_cast<const float2 *>(&sm.base_b[wj + 8 * b + 2 * (lane & 3)]);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const float arg = fmaf(-limit(q ? o[a][h][b].y : o[a][h][b].x), inv, ai + (q ? bj.y : bj.x));
            // (NaN, where t / s and the bases overflow, is flagged)
            if (!(x[a][b][2 * h + q] <= ex2(arg))) mine[a][h] |= 1u << (2 * b + q);
          }
        }
        if (!full) {
          const int i = wi + 16 * a + 8 * h + (lane >> 2), j = wj + 2 * (lane & 3);
          if (i >= mI) mine[a][h] = 0u;
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (j + 8 * (q >> 1) + (q & 1) >= mJ) mine[a][h] &= ~(1u << q);
        }
        found += __popc(mine[a][h]);
      }
  };
  if (whole)
    // ceil(old) - 1, by rounding up at 1.5 2^23.  From 2^22 on the result is at least
    // min(ceil(old) - 1, 2^23), which no sum of these blocks passes; below -2^22, where
    // the rounding may be finer, no sum of theirs lies.
    test([](float old) { return __fadd_rn(__fadd_ru(old, 12582912.0f), -12582913.0f); });
  else test([](float old) { return old; });
  found = __reduce_add_sync(kFullMask, found);
  if (lane == 0 && found) atomicAdd(&sm.count, found);
  __syncthreads();
  const int count = sm.count;
  if (count == 0) return 0;
  if (PROBE && tid == 0 && set != kSetNext && blockIdx.x % kSample == 0)
    atomicAdd(scr.cost, count > kScreenDense ? scr.dense : (count + 63) / 64);
  if (count > kScreenDense) {
    if (tid == 0) list_tile(scr, set);
    return 0;
  }
  // The flagged outputs as a list, in any order.
  int at = __popc(mine[0][0]) + __popc(mine[0][1]) + __popc(mine[1][0]) + __popc(mine[1][1]);
  if (at) at = atomicAdd(&sm.next, at);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      for (unsigned bits = mine[a][h]; bits; bits &= bits - 1) {
        const int q = __ffs(bits) - 1;
        sm.list[at++] = (unsigned short)((wi + 16 * a + 8 * h + (lane >> 2)) * H + wj + 8 * (q >> 1) + 2 * (lane & 3) + (q & 1));
      }
  __syncthreads();
  return count;
}

// The tiles left to the dense kernel: how many, and the t-th.
struct Listed {
  int count;
  const int *list;  // NULL: all of the set
  __device__ __forceinline__ Listed(const Screen &scr, int set, int R) {
    const bool nx = set == kSetNext;
    list = scr.skip() ? nullptr : nx ? scr.next : scr.rest;
    count = list ? *(nx ? scr.listed_next : scr.listed_rest) : PER_BLOCK * set_blocks(set, R);
  }
  __device__ __forceinline__ int tile(int t) const { return list ? list[t] : t; }
};
}  // namespace k3x

}  // namespace apsp
