// FP64 blocked Floyd-Warshall for sm_103a, exact, on the FP32 pipes.
//
// GB300 executes FP64 adds at about 2 per clock per SM, 1/64 of its FP32 rate,
// so a native FP64 min-plus product runs ~60x slower than FP32.  This path
// keeps every result bit-exact with IEEE FP64 (round to nearest) while doing
// almost all of the work in FP32:
//
//  * each FP64 operand x has a lower bound rd(x), the largest float <= x;
//  * a candidate a + b is at least lo = rd(rd(a) + rd(b)) (add.rm), and so is
//    its FP64 rounding fl(a + b), since rounding is monotone;
//  * a group of candidates is taken by its lower bounds alone (one packed
//    add.rm.f32x2 and one three-input min per two).  If their minimum X is not
//    below ru(old), the smallest float >= the old value, nothing improves.
//    Otherwise the first candidate with lo = X gets one FP64 add, s.  If s = X,
//    or no other candidate has lo <= ru(s), s is the exact minimum and its k
//    the first that reaches it; if some has (rare: sums within one float step
//    of each other), every candidate with lo <= ru(s) is added in FP64.
//
// Schedule per round r (TB = 128), the blocked FW of §2.2, every phase in the
// paper's k order:
//  K1  fw64_diag     phase 1: Algorithm 1 on block (r,r), k sequential.
//  K2  fw64_lines    phases 2 and 3: the row blocks (r,J) and column blocks
//                    (I,r), k sequential per line; writes the phase-4 operands.
//  K3  fw64_pieces   phase 4: (I,J) <- min(C, D(I,r) (x) D(r,J)); in the later
//      fw64_screen   rounds of large matrices only where a screen on the
//      fw64_listed   tensor cores finds that outputs may improve.
// Rounds overlap as in the FP32 path (rounds.cuh).
// Every candidate sum is one IEEE FP64 addition rounded to nearest, taken in
// the order of the sequential blocked FW, so D and P are bit-exact with it on
// any weights (and with every correct FW on integer-valued weights).
#include <float.h>
#include <stdint.h>

#include <algorithm>

#include "bulk.cuh"
#include "common.cuh"
#include "scratch.h"
#include "profile.h"
#include "rounds.cuh"
#include "screen.cuh"

namespace apsp {
namespace f64 {

constexpr int T = 128, PAIRS = T / 2, QUADS = T / 4;

// Operands of phase 4, written by K2 each round (entries outside the matrix
// are +inf):
//   column block (I,r): A[I][kp][i] = (rd D[i][2kp], rd D[i][2kp+1]),
//                       A64[I][i][k] = D[i][k]
//   row block (r,J):    B[J][j/64][kp][j%64] = (rd D[2kp][j], rd D[2kp+1][j]),
//                       B64[J][j][k] = D[k][j]
// and in a screened round the lower bounds as rows too: Alo[I][i][k] = rd
// A64[I][i][k], Blo[J][j][k] = rd B64[J][j][k].
struct Panels64 {
  unsigned long long *A, *B;
  double *A64, *B64;
  float *Alo, *Blo;
};
// The closed diagonal block in K2's layouts, written by K1: lower bounds
// k-paired, Alo[kp][i] = (rd D[i][2kp], rd D[i][2kp+1]), Blo[kp][j] =
// (rd D[2kp][j], rd D[2kp+1][j]), and values A64[k][i] = D[i][k], B64[k][j] =
// D[k][j].
struct DiagOps64 {
  unsigned long long *Alo, *Blo;
  double *A64, *B64;
};

// ---------------------------------------------------------------- bounds
// Largest float <= x and smallest float >= x for any non-NaN double, from the
// bit pattern (integer pipes only).  Tight in the normal float range; below
// it the bound is loosened to 0 / +-FLT_MIN, which keeps it valid.
__device__ __forceinline__ float f64_up(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ff), fe = e - 1023 + 127;
  unsigned f = ((unsigned)fe << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);  // magnitude toward zero
  f += (lo & 0x1fffffffu) && !sign ? 1u : 0u;
  if (fe >= 255) f = e == 0x7ff || !sign ? 0x7f800000u : 0x7f7fffffu;            // infinity, or beyond the floats
  if (fe <= 0) f = sign || ((hi << 1) | lo) == 0u ? 0u : 0x00800000u;           // below the normal floats
  return __uint_as_float(f | sign);
}

__device__ __forceinline__ float f64_down(double x) { return -f64_up(-x); }

// Exact float -> double bits (integer pipes; subnormal floats via cvt).
__device__ __forceinline__ unsigned long long f32_to_f64_bits(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xff;
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  if (e == 0) {
    if ((u & 0x7fffffu) == 0) return sign;
    return (unsigned long long)__double_as_longlong((double)f);
  }
  if (e == 0xff) return sign | 0x7ff0000000000000ull | ((unsigned long long)(u & 0x7fffffu) << 29);
  return sign | ((unsigned long long)(e - 127 + 1023) << 52) | ((unsigned long long)(u & 0x7fffffu) << 29);
}

__device__ __forceinline__ double f32_as_f64(float x) { return __longlong_as_double((long long)f32_to_f64_bits(x)); }

// a < b for doubles (no NaN) on the integer pipes: as signed integers, with
// the order of two negative values reversed, and -0 equal to +0.
__device__ __forceinline__ bool dless(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  const long long kx = x ^ (long long)((unsigned long long)(x >> 63) >> 1);
  const long long ky = y ^ (long long)((unsigned long long)(y >> 63) >> 1);
  return kx < ky && ((x | y) << 1) != 0;
}

__device__ __forceinline__ unsigned long long packf2(float lo, float hi) {
  return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}

// Lower-bound sums of two candidates (add.rm, as the main loop).
__device__ __forceinline__ float2 sum2_rm(unsigned long long a, unsigned long long b) {
  unsigned long long t;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(t) : "l"(a), "l"(b));
  return make_float2(__uint_as_float((unsigned)t), __uint_as_float((unsigned)(t >> 32)));
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

__device__ __forceinline__ void relax2_rm(float &acc, unsigned long long a, unsigned long long b) {
  asm("{\n\t.reg .b64 t;\n\t.reg .f32 x, y;\n\t"
      "add.rm.f32x2 t, %1, %2;\n\t"
      "mov.b64 {x, y}, t;\n\t"
      "min.f32 %0, %0, x, y;\n\t}"
      : "+f"(acc)
      : "l"(a), "l"(b));
}

// __byte_perm selector that replaces byte c of its first operand with byte 0 of its second.
__device__ __forceinline__ constexpr unsigned byte_sel64(int c) {
  return 0x3210 ^ ((0x3210 & (0xF << (4 * c))) ^ (4 << (4 * c)));
}

// ---------------------------------------------------------------- K1, K2
// Both phases take four steps k = 4 kq + s at a time on lines held four
// elements a lane: a line's pivots p[s] (its values at positions 4 kq + s, each
// at its own step) against the quad's rows r[s].
//
// The pivots of up to four lines at once: lane 4 c + t (c, t < 4) holds line
// c's value v at position 4 kq + t.  e[s]: row s of the quad at position
// 4 kq + t, at its own step; elo[s]: its lower bound.  Brings v to its step; vlo
// is its lower bound.  The FP64 additions run only if some lane's candidates
// may improve.  All lanes call.
template <typename E>
__device__ __forceinline__ void quad_pivots(double &v, float &vlo, const float (&elo)[3], int lane, E e) {
  const int t = lane & 3;
  vlo = f64_down(v);
  const float vhi = f64_up(v);
  bool may = false;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const float pivot = __shfl_sync(kFullMask, vlo, (lane & ~3) | s);
    may |= t > s && __fadd_rd(pivot, elo[s]) < vhi;
  }
  if (!__any_sync(kFullMask, may && lane < 16)) return;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const double cand = __dadd_rn(__shfl_sync(kFullMask, v, (lane & ~3) | s), e(s));
    if (t > s && dless(cand, v)) v = cand;
  }
  vlo = f64_down(v);
}
// The same for the quad's own four rows (line c = row c), whose entries are
// each other's e (returned too).
__device__ __forceinline__ void quad_pivots_own(double &v, float &vlo, double (&e)[3], int lane) {
  const int t = lane & 3;
  vlo = f64_down(v);
  const float vhi = f64_up(v);
  bool may = false;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    e[s] = __shfl_sync(kFullMask, v, 4 * s + t);
    // row s itself takes D[k][k] + its own value: no change unless D[k][k] < 0
    const float pivot = __shfl_sync(kFullMask, vlo, (lane & ~3) | s);
    const float row = __shfl_sync(kFullMask, vlo, 4 * s + t);
    may |= t > s && __fadd_rd(pivot, row) < vhi && !(lane >> 2 == s && pivot >= 0.0f);
  }
  if (!__any_sync(kFullMask, may && lane < 16)) return;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    e[s] = __shfl_sync(kFullMask, v, 4 * s + t);
    const double cand = __dadd_rn(__shfl_sync(kFullMask, v, (lane & ~3) | s), e[s]);
    if (t > s && dless(cand, v)) v = cand;
  }
  vlo = f64_down(v);
}

// A warp's four lines, in shared memory.
struct WarpLines {
  double d[4][T];
  float hi[4][T];          // ru(d)
  double ps[4][4];         // the quad's pivots [line][s]
  float plo[4][4];         // their lower bounds
  unsigned short list[4 * T];
  unsigned char pk[4][T];  // k of the last improvement, 0xFF none
};

// The warp's lines through the quad's four steps.  rlo01, rlo23: the rows'
// lower bounds (rows 0, 1 and 2, 3, paired, by position), r64(s, pos): their
// values.  Lane l tests its positions 4l..4l+3 of each line by lower bounds; the
// elements that may improve are then listed and taken by all lanes together,
// one each, so that the FP64 additions (16 clocks a warp per SM however many
// lanes need them) and the work around them are shared.
//
// The element at position k itself takes D[k][k] + its own value at step k,
// and (own: the lines are the quad's rows) so does every element of row k;
// neither can lower it unless D[k][k] < 0.  Those candidates are left out,
// since their lower bounds alone would list every value that is not a float.
template <typename Rv>
__device__ __forceinline__ void relax_lines(WarpLines &L, int kq, bool own, int lane, const unsigned long long *rlo01,
                                            const unsigned long long *rlo23, Rv r64) {
  auto bounds = [](float (&l)[4], unsigned long long pa, unsigned long long pb, unsigned long long ra,
                   unsigned long long rb) {
    const float2 l01 = sum2_rm(pa, ra), l23 = sum2_rm(pb, rb);
    l[0] = l01.x, l[1] = l01.y, l[2] = l23.x, l[3] = l23.y;
  };
  auto leave_out = [](float (&l)[4], int c, unsigned long long ra, unsigned long long rb) {
    const unsigned long long rc = c < 2 ? ra : rb;
    if (__uint_as_float((unsigned)((c & 1) ? rc >> 32 : rc)) >= 0.0f) {
#pragma unroll
      for (int s = 0; s < 4; ++s) l[s] = s == c ? inf<float>() : l[s];
    }
  };
  unsigned may = 0u;  // bit 4 c + q
  {
    unsigned long long ra[4], rb[4];
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
      const ulonglong2 ta = *reinterpret_cast<const ulonglong2 *>(&rlo01[4 * lane + q]);
      const ulonglong2 tb = *reinterpret_cast<const ulonglong2 *>(&rlo23[4 * lane + q]);
      ra[q] = ta.x, ra[q + 1] = ta.y, rb[q] = tb.x, rb[q + 1] = tb.y;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float4 p4 = *reinterpret_cast<const float4 *>(&L.plo[c][0]);
      float &pc = c == 0 ? p4.x : c == 1 ? p4.y : c == 2 ? p4.z : p4.w;
      if (own && pc >= 0.0f) pc = inf<float>();
      const unsigned long long pa = packf2(p4.x, p4.y), pb = packf2(p4.z, p4.w);
      const float4 h = *reinterpret_cast<const float4 *>(&L.hi[c][4 * lane]);
      const float hi[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float l[4];
        bounds(l, pa, pb, ra[q], rb[q]);
        if (lane == kq) leave_out(l, q, ra[q], rb[q]);
        may |= (fminf(min3f(l[0], l[1], l[2]), l[3]) < hi[q] ? 1u : 0u) << (4 * c + q);
      }
    }
  }
  if (!__any_sync(kFullMask, may != 0u)) return;
  int end = __popc(may);  // inclusive prefix sum of the counts
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFullMask, end, o);
    end += lane >= o ? t : 0;
  }
  const int total = __shfl_sync(kFullMask, end, 31);
  for (int at = end - __popc(may); may; may &= may - 1) {
    const int b = __ffs(may) - 1;
    L.list[at++] = (unsigned short)((b >> 2) * T + 4 * lane + (b & 3));
  }
  __syncwarp();
#pragma unroll 1
  for (int t = lane; t < total; t += 32) {
    const int c = L.list[t] / T, pos = L.list[t] % T;
    const ulonglong2 pp = *reinterpret_cast<const ulonglong2 *>(&L.plo[c][0]);
    const unsigned long long ra = rlo01[pos], rb = rlo23[pos];
    float l[4];
    bounds(l, pp.x, pp.y, ra, rb);
    if (pos >> 2 == kq) leave_out(l, pos & 3, ra, rb);
    if (own && L.plo[c][c] >= 0.0f) {
#pragma unroll
      for (int u = 0; u < 4; ++u) l[u] = u == c ? inf<float>() : l[u];
    }
    const float X = fminf(min3f(l[0], l[1], l[2]), l[3]);
    int s = l[0] == X ? 0 : l[1] == X ? 1 : l[2] == X ? 2 : 3;
    double best = __dadd_rn(L.ps[c][s], r64(s, pos));
    float up = f64_up(best);
    const int near = (l[0] <= up) + (l[1] <= up) + (l[2] <= up) + (l[3] <= up);
    if (near > 1 && best != f32_as_f64(X)) {  // others within one float step: add them too
      best = inf<double>();
#pragma unroll 1
      for (int u = 0; u < 4; ++u) {
        const float lu = u == 0 ? l[0] : u == 1 ? l[1] : u == 2 ? l[2] : l[3];
        if (lu > up) continue;
        const double cand = __dadd_rn(L.ps[c][u], r64(u, pos));
        if (dless(cand, best)) {
          best = cand;
          s = u;
        }
      }
      up = f64_up(best);
    }
    if (dless(best, L.d[c][pos])) {
      L.d[c][pos] = best;
      L.hi[c][pos] = up;
      L.pk[c][pos] = (unsigned char)(4 * kq + s);
    }
  }
  __syncwarp();
}

// K1: phase 1 on block (r,r) by one cluster of eight CTAs of four row warps, as
// the FP32 path's: a warp owns four adjacent rows, lane l their columns
// 4l..4l+3, and takes the four steps of a quad together.  The quad's own rows
// are brought to their steps by four helper warps of the owning CTA (a column a
// lane) while the others bring their pivots up; the helpers also pass the quads
// around the ring of CTAs by st.async.  The buffers hold eight quads (so that
// the kernel leaves room beside phase-4 CTAs): a CTA's four quads reuse the
// space of the quads eight before, which every CTA has left behind by then (a
// split cluster barrier per four quads).
// Bound: the chain of 32 quads (up to six dependent FP64 adds each), and while
// many elements still improve the FP64 adds of their candidates.  Measured per
// launch at n = 1000, real weights: 61-95 us, 1.9 us a quad (one CTA that took
// each flagged element in a serial loop per step: 245-600 us; this split with
// the row warps doing the helpers' work: 65-105 us, the whole solve 1.14 ms
// against 1.08); taking a lane's own flagged elements in place instead of
// listing them for the warp 125-218 us.
namespace k1 {
constexpr int CTAS = 8, WARPS = 4, RING = 2 * WARPS;  // WARPS: that own rows; as many help
constexpr int THREADS = 64 * WARPS;
struct Smem {
  double r64[RING][4][T];              // row s of the quad at its step
  unsigned long long rlo[RING][2][T];  // their lower bounds, rows (0, 1) and (2, 3)
  WarpLines wl[WARPS];
  double es[3][4];                     // the own quad's rows at its columns, at their steps
  float eslo[3][4];                    // their lower bounds
  uint64_t bar[QUADS];
};
constexpr uint32_t QUAD_BYTES = 4 * T * 8 + 2 * T * 8;
}  // namespace k1

__global__ void __cluster_dims__(k1::CTAS, 1, 1) __launch_bounds__(k1::THREADS, 2)
    fw64_diag(double *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int vec, int first,
              DiagOps64 ops, unsigned *__restrict__ range) {
  using namespace k1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const int base = r * T, m = min(T, n - base), nquad = (m + 3) / 4;
  const int cta = (int)cluster_cta_rank(), tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool helper = w >= WARPS;
  const int own = helper ? -1 : cta * WARPS + w;  // this warp's row quad
  const int i0 = 4 * own, j0 = 4 * lane, ht = tid - 32 * WARPS;  // ht: a helper's column
  if (tid < QUADS) {
    mbar_init(&sm.bar[tid], 1);
    fence_mbar_init();
    if (tid / WARPS != cta) mbar_expect_tx(&sm.bar[tid], QUAD_BYTES);
  }
  WarpLines &L = sm.wl[w % WARPS];
#pragma unroll
  for (int rr = 0; rr < 4 && !helper; ++rr) {
    const double *row = D + (int64_t)(base + i0 + rr) * ld + base;
    *reinterpret_cast<unsigned *>(&L.pk[rr][j0]) = 0xFFFFFFFFu;
#pragma unroll
    for (int c = 0; c < 4; c += 2) {
      double2 t = make_double2(inf<double>(), inf<double>());
      if (i0 + rr < m) {
        if (vec && j0 + c + 1 < m) {
          t = *reinterpret_cast<const double2 *>(row + j0 + c);
        } else {
          if (j0 + c < m) t.x = row[j0 + c];
          if (j0 + c + 1 < m) t.y = row[j0 + c + 1];
        }
      }
      *reinterpret_cast<double2 *>(&L.d[rr][j0 + c]) = t;
      *reinterpret_cast<float2 *>(&L.hi[rr][j0 + c]) = make_float2(f64_up(t.x), f64_up(t.y));
    }
  }
  __syncwarp();
  cluster_sync();  // every barrier of the cluster is set up before anyone publishes
  bool ok = true;
  const unsigned next = (unsigned)(cta + 1) % CTAS;
  const uint32_t next_base = cluster_map(smem_addr(smem_raw), next) - smem_addr(smem_raw);
#pragma unroll 1
  for (int kq = 0; kq < nquad; ++kq) {
    const int g = kq / WARPS, ow = kq % WARPS, slot = kq % RING;
    const bool mine = kq == own;
    double v = 0.0;
    float vlo;
    auto keep_pivots = [&]() {
      if (lane < 16) {
        (&L.ps[0][0])[lane] = v;
        (&L.plo[0][0])[lane] = vlo;
      }
    };
    if (!helper) v = L.d[(lane >> 2) & 3][4 * kq + (lane & 3)];
    if (cta == g) {
      if (mine) {
        double e[3];
        quad_pivots_own(v, vlo, e, lane);
        if (lane < 4) {
#pragma unroll
          for (int u = 0; u < 3; ++u) {
            sm.es[u][lane] = e[u];
            sm.eslo[u][lane] = f64_down(e[u]);
          }
        }
        keep_pivots();
      }
      __syncthreads();
      if (helper) {  // column ht: the quad's rows at their steps
        double q[4];
        float qlo[4];
        bool may = false;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          q[s] = sm.wl[ow].d[s][ht];
          qlo[s] = f64_down(q[s]);
#pragma unroll
          for (int u = 0; u < 3; ++u)
            if (u < s) may |= __fadd_rd(sm.wl[ow].plo[s][u], qlo[u]) < sm.wl[ow].hi[s][ht];
        }
        if (may) {  // (a column whose rows cannot improve keeps its values)
#pragma unroll
          for (int s = 1; s < 4; ++s) {
#pragma unroll
            for (int u = 0; u < 3; ++u)
              if (u < s) {
                const double cand = __dadd_rn(sm.wl[ow].ps[s][u], q[u]);
                if (dless(cand, q[s])) q[s] = cand;
              }
            qlo[s] = f64_down(q[s]);
          }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) sm.r64[slot][s][ht] = q[s];
        sm.rlo[slot][0][ht] = packf2(qlo[0], qlo[1]);
        sm.rlo[slot][1][ht] = packf2(qlo[2], qlo[3]);
      } else if (!mine) {
        const float elo[3] = {sm.eslo[0][lane & 3], sm.eslo[1][lane & 3], sm.eslo[2][lane & 3]};
        quad_pivots(v, vlo, elo, lane, [&](int s) { return sm.es[s][lane & 3]; });
        keep_pivots();
      }
      __syncthreads();
    } else {
      if (ok) ok = mbar_spin(&sm.bar[kq], 0);
    }
    if (helper) {
      if (next != (unsigned)g) {  // pass the quad on to the next CTA of the ring
        const uint32_t bar = next_base + smem_addr(&sm.bar[kq]);
        const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(&sm.r64[slot][0][0]);
        const ulonglong2 *srl = reinterpret_cast<const ulonglong2 *>(&sm.rlo[slot][0][0]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const ulonglong2 t = src[ht + 128 * u];
          st_async16(next_base + smem_addr(src + ht + 128 * u), t.x, t.y, bar);
        }
        const ulonglong2 t = srl[ht];
        st_async16(next_base + smem_addr(srl + ht), t.x, t.y, bar);
      }
    } else {
      if (cta != g) {
        const int t = 4 * kq + (lane & 3);
        const unsigned long long e01 = sm.rlo[slot][0][t], e23 = sm.rlo[slot][1][t];
        const float elo[3] = {__uint_as_float((unsigned)e01), __uint_as_float((unsigned)(e01 >> 32)),
                              __uint_as_float((unsigned)e23)};
        quad_pivots(v, vlo, elo, lane, [&](int s) { return sm.r64[slot][s][t]; });
        keep_pivots();
      }
      __syncwarp();
      relax_lines(L, kq, mine, lane, sm.rlo[slot][0], sm.rlo[slot][1],
                  [&](int s, int pos) { return sm.r64[slot][s][pos]; });
    }
    if (ow == WARPS - 1 || kq + 1 == nquad) {  // done with CTA g's quads
      if (g > 0) cluster_wait();               // and so is everyone with CTA g-1's, whose space comes next
      cluster_arrive();
    }
  }
  cluster_wait();  // no CTA leaves while another may still write its buffers
  if (!ok) {       // D and P stay as they are
    report_wait_timeout();
    drain_ring(sm.bar, nquad, WARPS, cta);
    return;
  }
  if (helper) return;
  double d[4][4];
#pragma unroll
  for (int rr = 0; rr < 4; ++rr)
#pragma unroll
    for (int c = 0; c < 4; ++c) d[rr][c] = L.d[rr][j0 + c];
  if (range) {  // of the lower bounds
    unsigned hi = 0u, lo = 0u;
#pragma unroll
    for (int rr = 0; rr < 4; ++rr)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float x = f64_down(d[rr][c]);
        if (x < inf<float>()) {
          hi = max(hi, fkey(x));
          lo = max(lo, fkey(-x));
        }
      }
    screen_range(range, hi, lo);
  }
  if (ops.Alo) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        ops.Blo[(2 * own + h) * T + j0 + c] = packf2(f64_down(d[2 * h][c]), f64_down(d[2 * h + 1][c]));
        ops.Alo[(2 * lane + h) * T + i0 + c] = packf2(f64_down(d[c][2 * h]), f64_down(d[c][2 * h + 1]));
      }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 4; c += 2) {
        *reinterpret_cast<double2 *>(&ops.B64[(i0 + a) * T + j0 + c]) = make_double2(d[a][c], d[a][c + 1]);
        *reinterpret_cast<double2 *>(&ops.A64[(j0 + a) * T + i0 + c]) = make_double2(d[c][a], d[c + 1][a]);
      }
  }
#pragma unroll
  for (int rr = 0; rr < 4; ++rr)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = i0 + rr, j = j0 + c;
      if (i >= m || j >= m) continue;
      const unsigned k = L.pk[rr][j];
      const int64_t e = (int64_t)(base + i) * ld + base + j;
      if (k != 0xFFu) D[e] = d[rr][c];
      // the first round's block is not initialised: every entry is written
      if (P && (first || k != 0xFFu)) P[e] = k != 0xFFu ? base + (int)k : -1;
    }
}

// K2: phases 2 and 3, k sequential in the paper's order (as the FP32 path):
// within a row block (r,J) every column j evolves on its own,
//   own[i][j] <- min(own[i][j], diag[i][k] + own[k][j])   (k ascending),
// within a column block (I,r) every row i does,
//   own[i][j] <- min(own[i][j], own[i][k] + diag[k][j]),
// with the diagonal block final after K1.  A warp keeps four such lines, lane
// l their positions 4l..4l+3, and takes the four steps of a quad together
// against the diagonal block's lower bounds in shared memory (one bulk copy);
// the values are read from global memory only where a candidate may improve.
// Then D and P are written where improved, and the blocks packed as phase-4
// operands.  Four warps a CTA, so that few blocks still use many SMs.
// Bound: the chain of 32 quads, as K1.  Measured per launch at n = 1000, real
// weights: 31-66 us (one step at a time, each flagged element in a serial
// loop: 94-156 us).
namespace k2 {
constexpr int WARPS = 4, LINES = 4 /* of a WarpLines */, CTA_LINES = WARPS * LINES, PARTS = T / CTA_LINES;
struct Smem {
  unsigned long long M[PAIRS][T];
  WarpLines wl[WARPS];
  uint64_t bar;
};
}  // namespace k2

__global__ void __launch_bounds__(32 * k2::WARPS, 2)
    fw64_lines(double *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, int vec,
               DiagOps64 ops, Panels64 pan, Screen scr) {
  using namespace k2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const int b = blockIdx.x / PARTS, part = blockIdx.x % PARTS;
  const bool is_row = b < R - 1;
  int other = is_row ? b : b - (R - 1);
  other += (other >= r);
  const int base_r = r * T, m_r = min(T, n - base_r);
  const int base_o = other * T, m_o = min(T, n - base_o);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) {
    mbar_init(&sm.bar, 1);
    fence_mbar_init();
    mbar_expect_tx(&sm.bar, sizeof(sm.M));
    fence_proxy_async_global();
    bulk_g2s(&sm.M[0][0], is_row ? ops.Alo : ops.Blo, sizeof(sm.M), &sm.bar);
  }
  const double *M64 = is_row ? ops.A64 : ops.B64;  // [k][pos]
  const int line0 = part * CTA_LINES + w * LINES, p0 = 4 * lane;
  // Element (line, pos) of the own block sits at D[g0 + line * sl + pos * sp].
  const int64_t g0 = is_row ? (int64_t)base_r * ld + base_o : (int64_t)base_o * ld + base_r;
  const int64_t sl = is_row ? 1 : ld, sp = is_row ? ld : 1;
  WarpLines &L = sm.wl[w];
  double v[LINES][4];
  // pairs along a line (column blocks) or across two lines (row blocks)
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int u = 0; u < 4; u += 2) {
      const int c = is_row ? u : a, q = is_row ? a : u;  // first element of the pair
      const int dc = is_row ? 1 : 0, dq = is_row ? 0 : 1;
      const bool in0 = line0 + c < m_o && p0 + q < m_r, in1 = line0 + c + dc < m_o && p0 + q + dq < m_r;
      const double *src = D + g0 + (line0 + c) * sl + (p0 + q) * sp;
      double2 t = make_double2(inf<double>(), inf<double>());
      if (vec && in1) {
        t = *reinterpret_cast<const double2 *>(src);
      } else {
        if (in0) t.x = src[0];
        if (in1) t.y = src[1];
      }
      if (is_row) {
        v[u][a] = t.x, v[u + 1][a] = t.y;
      } else {
        v[a][u] = t.x, v[a][u + 1] = t.y;
      }
    }
#pragma unroll
  for (int c = 0; c < LINES; ++c) {
    *reinterpret_cast<unsigned *>(&L.pk[c][p0]) = 0xFFFFFFFFu;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      L.d[c][p0 + q] = v[c][q];
      L.hi[c][p0 + q] = f64_up(v[c][q]);
    }
  }
  __syncthreads();
  const bool ok = mbar_wait(&sm.bar, 0);
  if (__syncthreads_or(!ok)) {  // the diagonal block never arrived: leave D, P and the operands as they are
    if (tid == 0) give_up(&sm.bar, 0);
    return;
  }
#pragma unroll 1
  for (int kq = 0; kq < QUADS; ++kq) {
    double x = L.d[(lane >> 2) & 3][4 * kq + (lane & 3)];
    {
      const int t = 4 * kq + (lane & 3);
      const unsigned long long e01 = sm.M[2 * kq][t], e23 = sm.M[2 * kq + 1][t];
      const float elo[3] = {__uint_as_float((unsigned)e01), __uint_as_float((unsigned)(e01 >> 32)),
                            __uint_as_float((unsigned)e23)};
      float xlo;
      quad_pivots(x, xlo, elo, lane, [&](int s) { return M64[(4 * kq + s) * T + t]; });
      if (lane < 16) {
        (&L.ps[0][0])[lane] = x;
        (&L.plo[0][0])[lane] = xlo;
      }
    }
    __syncwarp();
    relax_lines(L, kq, false, lane, sm.M[2 * kq], sm.M[2 * kq + 1], [&](int s, int pos) { return M64[(4 * kq + s) * T + pos]; });
  }
#pragma unroll
  for (int c = 0; c < LINES; ++c)
#pragma unroll
    for (int q = 0; q < 4; ++q) v[c][q] = L.d[c][p0 + q];
  // The phase-4 operands everywhere (padded), D and P where the line improved.
  const int64_t blk = other;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int kp = 2 * lane + h;
    unsigned long long *dst = is_row ? &pan.B[((blk * 2 + (line0 >> 6)) * PAIRS + kp) * (T / 2) + (line0 & 63)]
                                     : &pan.A[(blk * PAIRS + kp) * T + line0];
#pragma unroll
    for (int c = 0; c < LINES; c += 2)
      *reinterpret_cast<ulonglong2 *>(dst + c) =
          make_ulonglong2(packf2(f64_down(v[c][2 * h]), f64_down(v[c][2 * h + 1])),
                          packf2(f64_down(v[c + 1][2 * h]), f64_down(v[c + 1][2 * h + 1])));
  }
  double *rows = is_row ? pan.B64 : pan.A64;
#pragma unroll
  for (int c = 0; c < LINES; ++c)
#pragma unroll
    for (int q = 0; q < 4; q += 2)
      *reinterpret_cast<double2 *>(&rows[(blk * T + line0 + c) * T + p0 + q]) = make_double2(v[c][q], v[c][q + 1]);
  if (scr.EA) {
    const float inv = screen_scale(scr.range);
    uint32_t *E = (is_row ? scr.EB : scr.EA) + blk * (T * T / 2);
    float *rlo = is_row ? pan.Blo : pan.Alo;
    bool whole = true;
#pragma unroll
    for (int c = 0; c < LINES; ++c) {
      const int line = line0 + c;
      float lo[4], e[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) lo[q] = f64_down(v[c][q]);
      *reinterpret_cast<float4 *>(&rlo[(blk * T + line) * T + p0]) = make_float4(lo[0], lo[1], lo[2], lo[3]);
      const float least = screen_least(lo[0], lo[1], lo[2], lo[3]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        e[q] = screen_weight(lo[q], least, inv);
        whole = whole && screen_whole(lo[q]) && lo[q] == f64_up(v[c][q]);
      }
      // k = 4 lane .. 4 lane + 3: half of chunk lane / 2
      *reinterpret_cast<uint2 *>(&E[line * (T / 2) + ((lane >> 1) ^ (line & 7)) * 4 + 2 * (lane & 1)]) =
          make_uint2(bf16x2(e[0], e[1]), bf16x2(e[2], e[3]));
      if (lane == 0) (is_row ? scr.base_b : scr.base_a)[blk * T + line] = least;
    }
    whole = __syncthreads_and(whole);
    if (tid == 0) (is_row ? scr.whole_b : scr.whole_a)[blk * PARTS + part] = whole;
  }
#pragma unroll
  for (int c = 0; c < LINES; ++c)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned k = L.pk[c][p0 + q];
      if (k == 0xFFu) continue;  // improved: inside the matrix
      const int64_t g = g0 + (line0 + c) * sl + (p0 + q) * sp;
      D[g] = v[c][q];
      if (P) P[g] = base_r + (int)k;
    }
}

// ---------------------------------------------------------------- K3
// Phase 4: one CTA computes a 32 x 64 piece of an output block from the lower
// bounds of all 128 k in shared memory, thread tile 4 x 2 (as the FP32 path's
// pieces).  Per output and group of k only the group's minimum is
// kept, merged into
//   X = min lo, with the group it came from (the first that reached it), and
//   Y = min lo over all other groups.
// Afterwards an output with X < ru(old) finds the first k with lo = X in its
// group and adds that candidate in FP64 (s).  No other candidate can be as
// small when s = X, or when neither Y nor the group's other sums are <= ru(s);
// otherwise every candidate with lo <= ru(s) is added in FP64, k ascending.
// Bound: the FP32 pipes where a launch fills the chip, latency below.  Measured
// per solve: n = 1000, real weights, 0.41 ms (6.8 ms with every improved output
// settled by a whole warp over all 128 k, which is what lower bounds alone ask
// for when no sum is a float); n = 4096 / 8192, integers, 11.0 / 66.7 ms with
// the overlapped chain's share (11.4 / 64.5 with a 128 x 64 tile, whose solves
// took 14.1 / 65.7 ms against 9.8 / 63.6).
namespace k3 {
constexpr int THREADS = 256, TR = 32, TC = 64, PER_BLOCK = (T / TR) * (T / TC);
constexpr int GP = 8;  // k-pairs per group
struct Smem {
  unsigned long long A[PAIRS][TR];
  unsigned long long B[PAIRS][TC];
  uint64_t bar;
};
}  // namespace k3

// False if the wait for the operands ran out: the CTA must then not set the
// barrier up again.
__device__ __forceinline__ bool piece64(double *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r,
                                        int I, int J, int sub, const Panels64 &pan) {
  using namespace k3;
  constexpr int CW = 2;  // columns per thread
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const int si = sub >> 1, hJ = sub & 1;
  const int baseI = I * T + si * TR, baseJ = J * T + hJ * TC, baseK = r * T;
  const int mI = min(TR, n - baseI), mJ = min(TC, n - baseJ), mK = min(T, n - baseK);
  if (mI <= 0 || mJ <= 0) return true;  // past the matrix (uniform exit)
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  // Whole groups: the operands are +inf past the matrix.
  const int ng = (mK + 2 * GP - 1) / (2 * GP);
  if (tid == 0) {
    mbar_init(&sm.bar, 1);
    fence_mbar_init();
    mbar_expect_tx(&sm.bar, (uint32_t)(GP * ng * (TR + TC) * 8));
    fence_proxy_async_global();
    bulk_g2s(&sm.B[0][0], pan.B + ((int64_t)J * 2 + hJ) * PAIRS * TC, (uint32_t)(GP * ng * TC * 8), &sm.bar);
  }
  __syncthreads();
  if (w == 0) {
    const unsigned long long *srcA = pan.A + (int64_t)I * PAIRS * T + si * TR;
    fence_proxy_async_global();
    for (int kp = lane; kp < GP * ng; kp += 32) bulk_g2s(&sm.A[kp][0], srcA + (int64_t)kp * T, TR * 8, &sm.bar);
  }
  // Outputs of a lane as in the FP32 pieces: rows r0 + (a & 1) + 8 (a >> 1),
  // columns c0 + (c & 1) + 16 (c >> 1).
  constexpr int WC = TC / (8 * CW);
  const int r0 = (w / WC) * 16 + 2 * (lane >> 3), c0 = (w % WC) * 8 * CW + 2 * (lane & 7);
  const float FINF = inf<float>();
  float X[4][CW], Y[4][CW];
  unsigned grp[CW];  // byte a of grp[c]: the group X[a][c] came from
#pragma unroll
  for (int c = 0; c < CW; ++c) {
    grp[c] = 0u;
#pragma unroll
    for (int a = 0; a < 4; ++a) X[a][c] = Y[a][c] = FINF;
  }
  __syncwarp();
  const bool ok = mbar_wait(&sm.bar, 0);
  if (__syncthreads_or(!ok)) {  // the operands never arrived: the block stays as it is
    if (tid == 0) give_up(&sm.bar, 0);
    return false;
  }
  if (tid == 0) mbar_inval(&sm.bar);  // its one phase is over: the next piece may set it up again
#pragma unroll 1
  for (int g = 0; g < ng; ++g) {
    float m[4][CW];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < CW; ++c) m[a][c] = FINF;
#pragma unroll 8
    for (int u = 0; u < GP; ++u) {
      const int kp = GP * g + u;
      const ulonglong2 a01 = *reinterpret_cast<const ulonglong2 *>(&sm.A[kp][r0]);
      const ulonglong2 a23 = *reinterpret_cast<const ulonglong2 *>(&sm.A[kp][r0 + 8]);
#pragma unroll
      for (int c = 0; c < CW; c += 2) {
        const ulonglong2 bb = *reinterpret_cast<const ulonglong2 *>(&sm.B[kp][c0 + 8 * c]);
        relax2_rm(m[0][c], a01.x, bb.x);
        relax2_rm(m[0][c + 1], a01.x, bb.y);
        relax2_rm(m[1][c], a01.y, bb.x);
        relax2_rm(m[1][c + 1], a01.y, bb.y);
        relax2_rm(m[2][c], a23.x, bb.x);
        relax2_rm(m[2][c + 1], a23.x, bb.y);
        relax2_rm(m[3][c], a23.y, bb.x);
        relax2_rm(m[3][c + 1], a23.y, bb.y);
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        if (m[a][c] < X[a][c]) grp[c] = __byte_perm(grp[c], (unsigned)g, byte_sel64(a));
        Y[a][c] = fminf(Y[a][c], fmaxf(X[a][c], m[a][c]));
        X[a][c] = fminf(X[a][c], m[a][c]);
      }
  }
  double old[4][CW];
  unsigned left = 0u;  // bit 4 c + a: output (a, c) may improve
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      const int i = r0 + (a & 1) + 8 * (a >> 1), j = c0 + c;
      old[a][c] = i < mI && j < mJ ? D[(int64_t)(baseI + i) * ld + baseJ + j] : -inf<double>();
    }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < CW; ++c) left |= (X[a][c] < f64_up(old[a][c]) ? 1u : 0u) << (4 * c + a);
  // Each lane takes its own next output, so that the warp runs the rest as
  // often as its fullest lane needs and not once per output.
#pragma unroll 1
  for (; left; left &= left - 1) {
    const int t = __ffs(left) - 1, a = t & 3, c = t >> 2;
    float x = X[0][0], second = Y[0][0];
    double was = old[0][0];
#pragma unroll
    for (int u = 1; u < 4 * CW; ++u) {
      x = t == u ? X[u & 3][u >> 2] : x;
      second = t == u ? Y[u & 3][u >> 2] : second;
      was = t == u ? old[u & 3][u >> 2] : was;
    }
    const int g = (int)(((c ? grp[1] : grp[0]) >> (8 * a)) & 0xFFu);
    const int i = r0 + (a & 1) + 8 * (a >> 1), j = c0 + c;
    int k = -1;
#pragma unroll
    for (int u = 0; u < GP; ++u) {
      const float2 l = sum2_rm(sm.A[GP * g + u][i], sm.B[GP * g + u][j]);
      const bool h0 = k < 0 && l.x == x;
      k = h0 ? 2 * (GP * g + u) : k;
      second = h0 ? second : fminf(second, l.x);
      const bool h1 = k < 0 && l.y == x;
      k = h1 ? 2 * (GP * g + u) + 1 : k;
      second = h1 ? second : fminf(second, l.y);
    }
    const double *ra = pan.A64 + ((int64_t)I * T + si * TR + i) * T, *rb = pan.B64 + ((int64_t)J * T + hJ * TC + j) * T;
    double best = __dadd_rn(__ldcg(ra + k), __ldcg(rb + k));
    if (best != f32_as_f64(x)) {
      const float up = f64_up(best);
      if (second <= up) {
        best = inf<double>();
#pragma unroll 1
        for (int h = 0; h < ng; ++h) {
          unsigned bits = 0u;
#pragma unroll
          for (int u = 0; u < GP; ++u) {
            const float2 l = sum2_rm(sm.A[GP * h + u][i], sm.B[GP * h + u][j]);
            bits |= (l.x <= up ? 1u : 0u) << (2 * u) | (l.y <= up ? 1u : 0u) << (2 * u + 1);
          }
#pragma unroll 1
          for (; bits; bits &= bits - 1) {
            const int kk = 2 * GP * h + __ffs(bits) - 1;
            const double cand = __dadd_rn(__ldcg(ra + kk), __ldcg(rb + kk));
            if (dless(cand, best)) {
              best = cand;
              k = kk;
            }
          }
        }
      }
    }
    if (dless(best, was)) {
      const int64_t e = (int64_t)(baseI + i) * ld + baseJ + j;
      D[e] = best;
      if (P) P[e] = baseK + k;
    }
  }
  return true;
}

template <int CTAS_PER_SM>
__global__ void __launch_bounds__(k3::THREADS, CTAS_PER_SM)
    fw64_pieces(double *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, Panels64 pan,
                int set) {
  int I, J;
  block_of(set, blockIdx.x / k3::PER_BLOCK, r, R, I, J);
  piece64(D, ld, P, n, r, I, J, blockIdx.x % k3::PER_BLOCK, pan);
}

// K3 screened (screen.cuh), on the lower bounds of the panels and the upper
// bounds of the old values: a candidate below the old value has a lower-bound
// sum below its upper bound.  Eight lanes settle a flagged output, four outputs
// a warp: lane s takes entries 4 (s + 8 u) + q (u, q < 4) of the row of Alo and
// the row of Blo; the candidate of the least sum is added in FP64 first, then
// those whose lower-bound sum its value does not exclude.
// Bound: as the FP32 screen, the latency of the loads; at n = 4096 the next
// round's chain (K1 90, K2 75, row and column r+1 50 us) sets the pace.  n =
// 4096 / 6000 with P, integers: 9.8 / 27.3 -> 8.6 / 20.2 ms.
template <bool PROBE>
__global__ void __launch_bounds__(k3x::THREADS, 4)
    fw64_screen(double *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, int vec, Panels64 pan,
                Screen scr, int set) {
  using namespace k3x;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const float FINF = inf<float>();
  Tile tile;
  const int count = screen_tile<k2::PARTS, PROBE>(sm, tile, n, r, R, scr, set, vec != 0,
                                                  [&](int i, int j, int left, auto whole_tile) {
    const double *p = D + (int64_t)i * ld + j;
    if constexpr (decltype(whole_tile)::value) {
      const double2 t = *reinterpret_cast<const double2 *>(p);
      return make_float2(f64_up(t.x), f64_up(t.y));
    }
    return make_float2(left > 0 ? f64_up(p[0]) : 0.0f, left > 1 ? f64_up(p[1]) : 0.0f);
  });
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, s8 = lane & 7;
  const float4 *alo = reinterpret_cast<const float4 *>(pan.Alo + (int64_t)tile.baseI * T);
  const float4 *blo = reinterpret_cast<const float4 *>(pan.Blo + (int64_t)tile.baseJ * T);
#pragma unroll 1
  for (int g = 4 * w; g < count; g += THREADS / 32 * 4) {
    const int it = g + (lane >> 3), e = sm.list[min(it, count - 1)], i = e / H, j = e % H;
    double *out = D + (int64_t)(tile.baseI + i) * ld + tile.baseJ + j;
    float4 av[4], bv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      av[u] = alo[i * (T / 4) + s8 + 8 * u];
      bv[u] = blo[j * (T / 4) + s8 + 8 * u];
    }
    const double was = *out;
    float c[16], m = FINF;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      c[4 * u] = __fadd_rd(av[u].x, bv[u].x);
      c[4 * u + 1] = __fadd_rd(av[u].y, bv[u].y);
      c[4 * u + 2] = __fadd_rd(av[u].z, bv[u].z);
      c[4 * u + 3] = __fadd_rd(av[u].w, bv[u].w);
      m = min3f(min3f(m, c[4 * u], c[4 * u + 1]), c[4 * u + 2], c[4 * u + 3]);
    }
    float least = m;
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) least = fminf(least, __shfl_xor_sync(kFullMask, least, d));
    const bool may = it < count && least < f64_up(was);
    if (!__any_sync(kFullMask, may)) continue;
    const double *ra = pan.A64 + (int64_t)(tile.baseI + i) * T, *rb = pan.B64 + (int64_t)(tile.baseJ + j) * T;
    // k of this lane's entry t: 4 (s8 + 8 (t / 4)) + t % 4, ascending with t
    auto k_of = [&](int t) { return 4 * (s8 + 8 * (t >> 2)) + (t & 3); };
    double best = inf<double>();
    int k = T;
    if (may && m == least) {
      int t = 0;
#pragma unroll
      for (int u = 15; u >= 0; --u) t = c[u] == m ? u : t;
      k = k_of(t);
      best = __dadd_rn(ra[k], rb[k]);
    }
    __syncwarp();
    auto reduce = [&]() {  // the least value of the output's lanes, the first k that has it
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) {
        const double v = __shfl_xor_sync(kFullMask, best, d);
        const int kv = __shfl_xor_sync(kFullMask, k, d);
        if (dless(v, best) || (!dless(best, v) && kv < k)) best = v, k = kv;
      }
    };
    const int first = k;
    reduce();
    const float up = f64_up(best);
    unsigned bits = 0u;
#pragma unroll
    for (int u = 0; u < 16; ++u) bits |= (c[u] <= up && k_of(u) != first ? 1u : 0u) << u;
    if (!may) bits = 0u;
    if (__any_sync(kFullMask, bits != 0u)) {
#pragma unroll 1
      for (; bits; bits &= bits - 1) {
        const int kk = k_of(__ffs(bits) - 1);
        const double v = __dadd_rn(ra[kk], rb[kk]);
        if (dless(v, best) || (!dless(best, v) && kk < k)) best = v, k = kk;
      }
      __syncwarp();
      reduce();
    }
    if (may && s8 == 0 && dless(best, was)) {
      *out = best;
      if (P) P[out - D] = r * T + k;
    }
  }
}

// The tiles the screen listed, relaxed densely: CTAs take pieces in turn.
__global__ void __launch_bounds__(k3::THREADS, 4)
    fw64_listed(double *__restrict__ D, int64_t ld, int32_t *__restrict__ P, int n, int r, int R, Panels64 pan,
                Screen scr, int set) {
  constexpr int PER = k3x::H / k3::TR;  // pieces a tile, one above the other
  const k3x::Listed listed(scr, set, R);
  const int pieces = PER * listed.count;
#pragma unroll 1
  for (int t = blockIdx.x; t < pieces; t += gridDim.x) {
    const int tile = listed.tile(t / PER), q = tile % k3x::PER_BLOCK;
    int I, J;
    block_of(set, tile / k3x::PER_BLOCK, r, R, I, J);
    fence_proxy_async_smem();
    __syncthreads();  // everyone is done with the previous piece's shared memory
    if (!piece64(D, ld, P, n, r, I, J, 2 * ((q >> 1) * PER + t % PER) + (q & 1), pan)) return;
  }
}

static int g_smem_k1[64], g_smem_k2[64], g_smem_k3[2][64], g_smem_k3x[2][64], g_smem_k3l[64];

// Four CTAs of 64 registers per SM where phase 4 has many waves (n = 4096 /
// 8192: 8.56 / 41.0 ms against 8.63 / 41.2 with three), three of 80 up to 24 blocks
// a side, where K1 must find room beside them (int32 n = 2048: 2.88 against 2.99 ms).
constexpr int kFewBlocks = 24;
// Phase 4 is screened from round 16 on from 32 blocks a side (n = 4096: 8.56 against
// 9.83 ms unscreened, 6000: 20.2 / 27.3; n = 3328: 5.66 / 5.83, 3840: 7.65 / 8.31,
// integers, but where most outputs improve screening costs up to 3 % at every
// size).  From round 8 on 3 % more at n = 4096, since settling an output costs more
// here.
constexpr int kScreenMinR = 32, kScreenFrom = 16;
// (As FP32 with P; limits of 12 to 14 within 1 % at n = 4096 and 6000.)
constexpr ScreenCost kCost{18, 15};

}  // namespace f64

// Host side of FP64 (called by apsp_fw_f64); init(stream) sets P to -1 outside
// its first block.
int run_fw_f64_interval(double *D, int n, int64_t ld, int32_t *P, cudaStream_t s,
                        void (*path_init)(int32_t *, int64_t, int64_t, int64_t, cudaStream_t)) {
  using namespace f64;
  const int R = (n + T - 1) / T;
  int st;
  if ((st = ensure_smem(fw64_diag, (int)sizeof(k1::Smem), g_smem_k1))) return st;
  if ((st = ensure_smem(fw64_lines, (int)sizeof(k2::Smem), g_smem_k2))) return st;
  const auto pieces = R <= kFewBlocks ? fw64_pieces<3> : fw64_pieces<4>;
  if ((st = ensure_smem(pieces, (int)sizeof(k3::Smem), g_smem_k3[R <= kFewBlocks]))) return st;
  if ((st = ensure_smem(fw64_screen<false>, (int)sizeof(k3x::Smem), g_smem_k3x[0]))) return st;
  if ((st = ensure_smem(fw64_screen<true>, (int)sizeof(k3x::Smem), g_smem_k3x[1]))) return st;
  if ((st = ensure_smem(fw64_listed, (int)sizeof(k3::Smem), g_smem_k3l))) return st;
  // Phase-4 operands: two sets by round parity, each R blocks of A and of B;
  // then K1's copies of the closed diagonal block.  With screened rounds the
  // sets also hold the rows of lower bounds and the screen's share.
  Panels64 pan[2]{};
  DiagOps64 ops{};
  char *scratch = nullptr;
  const bool screened = R >= kScreenMinR;
  ScreenSets scr(R, k2::PARTS);
  if (R > 1) {
    const size_t elems = (size_t)R * T * T, plain = elems * (4 + 4 + 8 + 8);
    const size_t set = plain + (screened ? elems * (4 + 4) + scr.set_bytes() : 0);
    if (scratch_alloc((void **)&scratch, 2 * set + (size_t)T * T * 24 + (screened ? scr.list_bytes() : 0), s) !=
        cudaSuccess) {
      cudaGetLastError();
      return APSP_ENOMEM;
    }
    for (int q = 0; q < 2; ++q) {
      char *base = scratch + q * set;
      pan[q].A64 = reinterpret_cast<double *>(base);
      pan[q].B64 = pan[q].A64 + elems;
      pan[q].A = reinterpret_cast<unsigned long long *>(pan[q].B64 + elems);
      pan[q].B = pan[q].A + elems / 2;
      if (!screened) continue;
      pan[q].Alo = reinterpret_cast<float *>(base + plain);
      pan[q].Blo = pan[q].Alo + elems;
      scr.place_set(q, pan[q].Blo + elems);
    }
    ops.A64 = reinterpret_cast<double *>(scratch + 2 * set);
    ops.B64 = ops.A64 + T * T;
    ops.Alo = reinterpret_cast<unsigned long long *>(ops.B64 + T * T);
    ops.Blo = ops.Alo + T * T / 2;
    if (screened && scr.place_lists(ops.Blo + T * T / 2, s) != cudaSuccess) {
      cudaFreeAsync(scratch, s);
      cudaGetLastError();
      return APSP_ECUDA;
    }
  }
  bool capturing = false;
  if ((st = stream_capturing(s, &capturing))) {
    if (scratch) cudaFreeAsync(scratch, s);
    return st;
  }
  const int probed = set_blocks(capturing ? kSetAll : kSetRest, R);
  auto screen_of = [&](int r) { return screened && r >= kScreenFrom ? scr.round(r, kScreenFrom, probed, kCost) : Screen{}; };
  const int vec = ld % 2 == 0 && (reinterpret_cast<uintptr_t>(D) & 15) == 0;
  auto init = [&](cudaStream_t stm) {
    if (P) path_init(P, n, ld, T, stm);
  };
  auto diag = [&](int r, cudaStream_t stm) {
    PhaseScope sc(1, stm);
    fw64_diag<<<k1::CTAS, k1::THREADS, sizeof(k1::Smem), stm>>>(D, ld, P, n, r, vec, (int)(P && r == 0), ops,
                                                                screen_of(r).range);
  };
  auto panels = [&](int r, cudaStream_t stm) {
    PhaseScope sc(2, stm);
    fw64_lines<<<2 * (R - 1) * k2::PARTS, 32 * k2::WARPS, sizeof(k2::Smem), stm>>>(D, ld, P, n, r, R, vec, ops,
                                                                                   pan[r & 1], screen_of(r));
  };
  auto phase4 = [&](int r, int set, int blocks, cudaStream_t stm) {
    if (blocks <= 0) return;
    const bool screen = screened && r >= kScreenFrom;
    PhaseScope sc(3, stm, screen ? 2 : 1);
    if (screen) {
      const Screen sr = screen_of(r);
      (sr.cost ? fw64_screen<true> : fw64_screen<false>)<<<k3x::PER_BLOCK * blocks, k3x::THREADS, sizeof(k3x::Smem), stm>>>(
          D, ld, P, n, r, R, vec, pan[r & 1], sr, set);
      fw64_listed<<<std::min(k3::PER_BLOCK * blocks, kListedCtas * kSms), k3::THREADS, sizeof(k3::Smem), stm>>>(
          D, ld, P, n, r, R, pan[r & 1], sr, set);
      return;
    }
    pieces<<<k3::PER_BLOCK * blocks, k3::THREADS, sizeof(k3::Smem), stm>>>(D, ld, P, n, r, R, pan[r & 1], set);
  };
  st = run_rounds(R, s, capturing, init, diag, panels, phase4);
  cudaError_t e = cudaGetLastError();
  if (scratch) {
    cudaError_t f = cudaFreeAsync(scratch, s);
    if (e == cudaSuccess) e = f;
  }
  return st ? st : status_from(e);
}

int take_device_error_f64() { return take_tu_device_error(); }

}  // namespace apsp
