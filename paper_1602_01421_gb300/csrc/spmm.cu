// SpMM, Y = A X for a 0/1 pattern matrix A (Section 3.3): every non-zero (i, j) adds row j
// of the dense block X to row i of Y.  X and Y are row-major n x b (Section 3.3.2).
//
// GB300 layout of A, built once per handle from the CSR (Section 3.3.1 / 3.3.3 motives: the
// paper fights branchy single-entry rows with SCSR+COO tiles and power-law load imbalance
// with work stealing; here the same two problems are solved by degree binning):
//   * tail rows (degree <= tail_max, default 128; 97% of the scale-22 R-MAT rows): grouped by
//     exact degree into 32-row slices whose column indices are stored transposed
//     ("SELL-32"): step t of row l is ell[t*32 + l]; a lane owns a row (above degree 32, two or
//     four lanes share one, slice_pieces), with coalesced index loads and no divergence or masked
//     lane, since all 32 rows of a slice have the same degree;
//   * mid rows (tail_max < degree <= hub_min): one warp per row (a "task"; long ones of smaller
//     matrices are shared by two or four warps of a CTA, plan_wide), 32 consecutive
//     column indices per coalesced load, each lane gathering up to 32 bytes of an X row
//     (one 256-bit load when X is 32-byte aligned), partial sums combined by a
//     reduce-scatter butterfly;
//   * hub rows (degree > hub_min): split into tasks of hub_chunk non-zeros; each task writes
//     a partial row, and a second kernel adds a hub's partials in a fixed order (deterministic,
//     no atomics).
// Tasks are ordered longest first so the block scheduler handles them like a longest-
// processing-time list; tail slices follow in the same launch.  The task rows' column
// indices are stored either as int32 or, in the packed format, as per-task gap fields that a
// warp decodes with a prefix sum (fewer bytes to stream from host memory).
// FP32 sums are compensated per lane (Kahan) before the lane tree, and the warps of a shared task
// and (compensated) hub chunks are added in FP64, so the FP32 error bound (9 * 2^-24 * A|X| per entry) does not grow with the
// degree or depend on the signs of X.
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "fe_internal.cuh"
#include "vec.cuh"

namespace fe {

static_assert(sizeof(Task) == 16, "Task must be 16 bytes");
static_assert(sizeof(PTask) == 32, "PTask must be 32 bytes");

// FP64 blocks whose sums the FP64 adds would bind (b = 1 is bound by its gathers): they are added in
// integers for the most part (Fx below) and gathered 16 bytes a lane.
template <typename T, int B>
constexpr bool kUseFx = sizeof(T) == 8 && B >= 2;
// Per (type, b, fragment width) geometry: a lane moves NE elements (<= FB bytes: 16, or 32
// with 256-bit loads when X is 32-byte aligned) per load; an X row of b elements spans C lanes
// in a warp task (P = 32 / C rows gathered per warp instruction) and C chunks in a tail lane.
template <typename T, int B, bool V32>
struct Geo {
  static constexpr int FB = V32 && !kUseFx<T, B> ? 32 : 16;
  static constexpr int ROWB = B * (int)sizeof(T);
  static constexpr int NE = ROWB <= FB ? B : FB / (int)sizeof(T);
  static constexpr int C = B / NE;
  static constexpr int P = 32 / C;
  static constexpr int UNROLL = C >= 4 ? 1 : 4 / C;
  static constexpr int LNE = NE >= 8 ? 3 : NE >= 4 ? 2 : NE >= 2 ? 1 : 0;  // log2(NE)
  // lane bits summed by the plain butterfly levels after the scatter levels (C .. 16 >> LNE)
  static constexpr int PLAIN_MASK = (16 >> LNE) >= C ? ((16 >> LNE) << 1) - C : 0;
};

struct SpmmParams {
  const int32_t* colidx;
  const uint32_t* tbits;
  const Task* tasks;
  const PTask* ptasks;
  int64_t ntasks, nhub_tasks;
  // tasks [0, wide4) run on four warps each, [wide4, wide2) on two, the rest on one; CTA ranges
  int64_t wide4, wide2, ctas4, ctas2, task_ctas;
  const int32_t* slice_rows;
  const int32_t* ell;
  int nbuckets, shared;   // shared: lanes share rows of the slices
  int32_t bucket_deg[kMaxBuckets];
  int32_t bucket_slice_begin[kMaxBuckets + 1];
  uint32_t bucket_warp_begin[kMaxBuckets + 1];  // first warp (after the tasks') of each bucket's slices
  int64_t bucket_ell_base[kMaxBuckets];
};

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarpsPerCta = 8;

// Warps of a CTA that share a task: a warp takes up to 128 non-zeros a round, so a task of 4096 on
// one warp is a serial chain of 32 rounds of two dependent loads, 35 to 50 us whatever the size of
// the graph.  In plans for at most kWideCols columns, and in streamed panels, hub chunks and rows
// above 2048 take four warps and rows above kWideLen two (R-MAT with 16384 vertices: FP32 b = 4 35
// -> 14 us, FP64 b = 4 48 -> 19 us; 131072 vertices: 58 -> 27 and 80 -> 70 us).  With more columns
// there are long rows enough to hide the chain, and four places of X read at once for one row
// cost locality (4.2 million vertices: FP32 b = 4 446 -> 467 us, b = 16 1.50 -> 1.57 ms; even at a
// million, 105 -> 109 us).  The rule uses the columns, which the parts of a row partition share with
// the whole matrix, so that a row's order of summation is the same in both.
constexpr int64_t kWideCols = 1 << 19;
constexpr int kWideLen = 1024;

// Lanes that share a row of a slice of degree d, each taking a run of its steps, and warps that
// share the slice (32 / pieces rows each): one lane per row makes a slice of 128 steps a serial
// chain of 32 dependent rounds of gathers (and 128 FP64 adds per column), the last thing that a
// launch waits for (R-MAT with 2^20 vertices, FP32 b = 4: 138 -> 105 us, FP64 b = 1 120 -> 107 us;
// 1000 vertices, FP64 b = 8 79 -> 29 us).  By the degree only, like the warps per task; FP64 b = 1
// with more than kSharedCols columns keeps one lane per row (its adds are all FP64, and the lanes'
// sums are more of them; 4.2 million vertices: 416 against 423 us).
constexpr int64_t kSharedCols = 1 << 20;
__host__ __device__ __forceinline__ int slice_pieces(int deg, int shared) {
  return deg <= 32 || !shared ? 1 : (deg <= 64 ? 2 : 4);
}

// Per-lane running sums.  FP32: Kahan's compensated summation (Kahan 1965; Higham, "Accuracy
// and Stability of Numerical Algorithms", 2nd ed., Thm. 4.8): c carries the rounding error of
// the last addition, so a lane's sum of m terms is within (2u + O(m u^2)) sum |x| of the exact
// sum (u = 2^-24), whatever the number of terms and their signs, instead of (m - 1) u sum |x|.
// Four FP32 adds per term; nvcc does not reassociate floating-point adds, so the correction
// survives compilation.  FP64: plain adds (m u with u = 2^-53 is already far below the FP64
// bound).  kahan_add(s, c, x) adds x; kahan_value(s, c) is the compensated sum.
__device__ __forceinline__ void kahan_add(float& s, float& c, float x) {
  const float y = x - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}
__device__ __forceinline__ void kahan_add(double& s, double&, double x) { s += x; }
__device__ __forceinline__ float kahan_value(float s, float c) { return s - c; }
__device__ __forceinline__ double kahan_value(double s, double) { return s; }
// The sum of this lane's (s, c), `keep`, and its partner's, `send` of the lane `off` away (TwoSum: the sums
// of lanes that share a row are compensated too).
__device__ __forceinline__ void kahan_merge(float keep, float ckeep, float send, float csend, int off, float& s, float& c) {
  const float x = __shfl_xor_sync(0xffffffffu, send, off), cx = __shfl_xor_sync(0xffffffffu, csend, off);
  const float t = keep + x, z = t - keep;
  const float d = (ckeep + cx) - ((keep - (t - z)) + (x - z));
  c = d == d ? d : 0.f;   // an infinite sum has no error term
  s = t;
}
__device__ __forceinline__ void kahan_merge(double keep, double, double send, double, int off, double& s, double&) {
  s = keep + __shfl_xor_sync(0xffffffffu, send, off);
}

// FP64 sums in integers.  An FP64 add occupies the FP64 pipe of an SM for 16 clocks per warp; the
// 32-bit integer units take the 16 instructions of an aligned integer add in half of that, beside it.
// So of every four gathered values one is added in FP64 and three as integers: an Fx holds
// a * 2^((e >> 20) - 1080), e the largest biased exponent so far (in its place in the high word),
// and a value's 53-bit significand, shifted left by 5 and right by its distance to e, is added to a.
// Bits below 2^-57 of the largest value are dropped (of a value towards zero, of a, when e rises,
// downwards): between two flushes, 24 values (4.6 bits, so a stays within 63) and at most 8 rises of
// e, an error below 2^-52 of the largest value, no more than that of as many FP64 adds; where no bit
// is dropped (whole numbers, say) the sum is exact.  Values with exponents near the ends of the range
// (infinities, NaN, below 2^-943) set `bad`, and the sums are formed again with FP64 adds.  Measured
// against FP64 adds alone (R-MAT, X 32-byte aligned): 4.2 million vertices b = 2 585 -> 520 us, b = 4
// 1085 -> 707, b = 8 2068 -> 1352, b = 16 4.18 -> 2.34 ms; a million, b = 4 288 -> 172 us.  The gathers
// bind then (FP32 b = 8, rows of the same 32 bytes: 615 us).
struct Fx {
  long long a;
  unsigned e;
};
constexpr int kFxGroups = 8;   // groups of four values between flushes
// t or, for sign = -1, -t - 1: fx_add3 takes the signs off again
__device__ __forceinline__ long long fx_align(unsigned hi, unsigned lo, unsigned ev, unsigned e, int sign) {
  const unsigned m = (hi & 0xfffffu) | min(ev, 0x100000u);   // implicit bit (0 for zeros, subnormals)
  unsigned long long t = (((unsigned long long)m << 32) | lo) << 5;
  asm("shr.u64 %0, %0, %1;" : "+l"(t) : "r"((e - ev) >> 20));   // shifts of 64 and more give 0
  return (long long)t ^ sign;
}
__device__ __forceinline__ void fx_add3(Fx& f, double x, double y, double z) {
  const unsigned hx = __double2hiint(x), hy = __double2hiint(y), hz = __double2hiint(z);
  const unsigned ex = hx & 0x7ff00000u, ey = hy & 0x7ff00000u, ez = hz & 0x7ff00000u;
  const unsigned e = max(max(ex, ey), max(ez, f.e));
  const int sx = (int)hx >> 31, sy = (int)hy >> 31, sz = (int)hz >> 31;
  asm("shr.s64 %0, %0, %1;" : "+l"(f.a) : "r"((e - f.e) >> 20));
  f.e = e;
  f.a += fx_align(hx, __double2loint(x), ex, e, sx) + fx_align(hy, __double2loint(y), ey, e, sy) +
         fx_align(hz, __double2loint(z), ez, e, sz) - (sx + sy + sz);
}
// s += f, f = 0
__device__ __forceinline__ void fx_flush(double& s, Fx& f, bool& bad) {
  bad = bad || f.e >= 0x7d000000u || (f.e < 0x05000000u && f.a != 0);
  const double v = __ll2double_rn(f.a);
  const unsigned hi = (unsigned)__double2hiint(v) + f.e - (1080u << 20);   // the exponent's change, modulo 2^32
  const double x = __hiloint2double((int)hi, __double2loint(v));
  s += f.a != 0 ? x : 0.0;
  f.a = 0;
  f.e = 0;
}
// Lanes of a slice that share a row by its columns, without 256-bit gathers: 16 bytes of it each.
// With Fx sums a column takes 13 registers (four gathers in flight), and the warps that fit decide
// (b = 4 at 4.2 million vertices: 950 us with four columns a lane, 80 registers).
template <typename T, int B, bool V32>
constexpr int kColLanes = V32 || B * sizeof(T) <= 16 || (sizeof(T) == 8 && !kUseFx<T, B>) ? 1 : B * (int)sizeof(T) / 16;
// Plans with shorter slice rows than this (packed ones, by default 16) take FP64 adds at b = 2: most of their
// tasks are rows of few entries a lane, whose flushes cost more than the adds, and a packed task's decoding
// takes the integer units too (packed, 4.2 million vertices: 813 us with FP64 adds, 1042 with Fx; a million 209
// and 258).  By tail_max, so that both index formats of one split give the same sums.
constexpr int kFxTailMax = 64;
constexpr int kFxMinDegree = 12;   // slices of shorter rows: the flush would cost more than it saves

// Gap field k (w bits) of a packed task's bit stream.
__device__ __forceinline__ int gap_field(const uint32_t* __restrict__ tb, int k, int w, uint32_t wmask) {
  const int64_t bit = (int64_t)k * w;
  const int64_t wi = bit >> 5;
  return (int)(__funnelshift_r(__ldcs(tb + wi), __ldcs(tb + wi + 1), (int)(bit & 31)) & wmask);
}

// Task ti on W warps of the CTA (this one takes piece `piece`); W > 1: all warps of the CTA call it
// (ti past the range: nothing to do but the barriers).
template <typename T, int B, bool V32, bool PACKED, bool FX, int W>
__device__ __forceinline__ void run_task(const SpmmParams& p, int64_t ti, int64_t tend, const T* __restrict__ X,
                                         T* __restrict__ Y, double* __restrict__ partial, int warp, int lane, double* red) {
  using G = Geo<T, B, V32>;
  const int piece = warp % W;
  int64_t start = 0;
  int row = 0, len = 0;
  int cbase = 0, w = 1;
  if (W == 1 || ti < tend) {
    if constexpr (PACKED) {
      const int4 r0 = __ldg(reinterpret_cast<const int4*>(p.ptasks + ti));
      const int4 r1 = __ldg(reinterpret_cast<const int4*>(p.ptasks + ti) + 1);
      start = (int64_t)(uint32_t)r0.x | ((int64_t)r0.y << 32);  // word offset
      row = r0.z;
      len = r0.w;
      cbase = r1.x;
      w = r1.y;
    } else {
      const int4 raw = __ldg(reinterpret_cast<const int4*>(p.tasks + ti));
      start = (int64_t)(uint32_t)raw.x | ((int64_t)raw.y << 32);
      row = raw.z;
      len = raw.w;
    }
  }
  // this warp's entries [k0, len)
  const int plen = W == 1 ? len : ((len + W - 1) / W + 31) & ~31;
  const int k0 = min(len, piece * plen), klen = W == 1 ? len : min(len, k0 + plen);
  const int chunk = lane % G::C;
  const int slot = lane / G::C;
  T acc[G::NE], cmp[G::NE];
#pragma unroll
  for (int e = 0; e < G::NE; ++e) acc[e] = cmp[e] = T(0);
  const int32_t* __restrict__ ci = p.colidx + start;
  const uint32_t* __restrict__ tb = p.tbits + start;
  const uint32_t wmask = (1u << w) - 1u;  // 1 <= w <= 31
  int carry = cbase;  // packed: the column reached by the previous round
  if constexpr (PACKED && W > 1) {
    // the columns that the earlier pieces cover: every warp adds up its own gaps first
    __shared__ int span[kWarpsPerCta];
    int sum = 0;
#pragma unroll 4
    for (int k = k0 + lane; k < klen; k += 32) sum += gap_field(tb, k, w, wmask);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(kFull, sum, off);
    if (lane == 0) span[warp] = sum;
    __syncthreads();
    for (int i = 0; i < piece; ++i) carry += span[warp - piece + i];
  }
  // the column of entry base + lane (-1 past the end); packed: calls in order, all lanes
  auto load_col = [&](int base) {
    const int k = base + lane;
    if constexpr (PACKED) {
      // field k of w bits, then an inclusive prefix sum of the gaps across the warp
      if (base >= klen) return -1;
      int g = 0;
      if (k < klen) g = gap_field(tb, k, w, wmask);
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, g, off);
        if (lane >= off) g += y;
      }
      const int col = carry + g;
      carry = __shfl_sync(kFull, col, 31);
      return k < klen ? col : -1;
    } else {
      return k < klen ? __ldcs(ci + k) : -1;
    }
  };
  auto plain = [&]() {
    for (int base = k0; base < klen; base += 32 * G::UNROLL) {
      int cols[G::UNROLL];
#pragma unroll
      for (int u = 0; u < G::UNROLL; ++u) cols[u] = load_col(base + u * 32);
#pragma unroll
      for (int u = 0; u < G::UNROLL; ++u) {
#pragma unroll
        for (int g = 0; g < 32; g += G::P) {
          // rounds whose P slots all lie past the row's end are skipped (warp-uniform test)
          if (base + u * 32 + g < klen) {
            int col = __shfl_sync(kFull, cols[u], g + slot);
            if (col >= 0) {
              T f[G::NE];
              ld_frag<T, G::NE>(X + (int64_t)col * B + chunk * G::NE, f);
#pragma unroll
              for (int e = 0; e < G::NE; ++e) kahan_add(acc[e], cmp[e], f[e]);
            }
          }
        }
      }
    }
  };
  if constexpr (FX) {
    constexpr int PER = 32 / G::P, NG = G::UNROLL * PER;   // gathers of a lane per 32 columns, per round
    const int carry0 = carry;
    Fx fa[G::NE];
    bool bad = false;
#pragma unroll
    for (int e = 0; e < G::NE; ++e) fa[e] = Fx{0, 0u};
    int groups = 0;
    int cols[G::UNROLL];   // of the coming round, loaded a round ahead
#pragma unroll
    for (int u = 0; u < G::UNROLL; ++u) cols[u] = load_col(k0 + u * 32);
    for (int base = k0; base < klen; base += 32 * G::UNROLL) {
#pragma unroll
      for (int v0 = 0; v0 < NG; v0 += 4) {
        T f[4][G::NE];   // four gathers of the lane (zero past the row's end)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int col = __shfl_sync(kFull, cols[(v0 + v) / PER], (v0 + v) % PER * G::P + slot);
#pragma unroll
          for (int e = 0; e < G::NE; ++e) f[v][e] = T(0);
          if (col >= 0) ld_frag<T, G::NE>(X + (int64_t)col * B + chunk * G::NE, f[v]);
        }
        if (v0 + 4 == NG) {
#pragma unroll
          for (int u = 0; u < G::UNROLL; ++u) cols[u] = load_col(base + (G::UNROLL + u) * 32);
        }
#pragma unroll
        for (int e = 0; e < G::NE; ++e) {
          acc[e] += f[0][e];
          fx_add3(fa[e], f[1][e], f[2][e], f[3][e]);
        }
      }
      if (++groups == kFxGroups * 4 / NG) {
#pragma unroll
        for (int e = 0; e < G::NE; ++e) fx_flush(acc[e], fa[e], bad);
        groups = 0;
      }
    }
#pragma unroll
    for (int e = 0; e < G::NE; ++e) fx_flush(acc[e], fa[e], bad);
    if (__any_sync(kFull, bad)) {
#pragma unroll
      for (int e = 0; e < G::NE; ++e) acc[e] = T(0);
      carry = carry0;
      plain();
    }
  } else {
    plain();
  }
  // Sum the P slot partials of each chunk.  The first LNE butterfly levels (offsets 16, 8, ..)
  // also scatter the NE elements -- a lane keeps half of what it holds and adds its partner's
  // copy of that half -- so every level after them adds one value per lane.  Where warps share the
  // task the lanes' sums stay compensated, so that the warps' add no more than the last rounding.
  constexpr bool kPairs = sizeof(T) == 4 && W > 1;
  if constexpr (!kPairs) {
#pragma unroll
    for (int e = 0; e < G::NE; ++e) acc[e] = kahan_value(acc[e], cmp[e]);
  }
  int ebase = 0;
#pragma unroll
  for (int lvl = 0; lvl < G::LNE; ++lvl) {
    const int h = G::NE >> (lvl + 1);
    const int off = 16 >> lvl;
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < (G::NE >> (lvl + 1)); ++i) {
      const T send = up ? acc[i] : acc[i + h];
      const T keep = up ? acc[i + h] : acc[i];
      if constexpr (kPairs) kahan_merge(keep, up ? cmp[i + h] : cmp[i], send, up ? cmp[i] : cmp[i + h], off, acc[i], cmp[i]);
      else acc[i] = keep + __shfl_xor_sync(kFull, send, off);
    }
    if (up) ebase += h;
  }
#pragma unroll
  for (int off = 16 >> G::LNE; off >= G::C; off >>= 1) {
    if constexpr (kPairs) kahan_merge(acc[0], cmp[0], acc[0], cmp[0], off, acc[0], cmp[0]);
    else acc[0] += __shfl_xor_sync(kFull, acc[0], off);
  }
  // column c of the row, or of a hub chunk: its sum stays in FP64 until the hub's chunks are added
  auto put = [&](int c, auto v) {
    if constexpr (sizeof(T) == 8) {
      T* dst = ti < p.nhub_tasks ? partial + ti * B : Y + (int64_t)row * B;
      dst[c] = v;
    } else if (ti < p.nhub_tasks) {
      partial[ti * B + c] = (double)v;
    } else {
      Y[(int64_t)row * B + c] = (T)v;
    }
  };
  if constexpr (W == 1) {
    if ((lane & G::PLAIN_MASK) == 0) put(chunk * G::NE + ebase, acc[0]);
  } else {
    // the pieces in order, in FP64: one more rounding to T however many there are
    if ((lane & G::PLAIN_MASK) == 0)
      red[warp * B + chunk * G::NE + ebase] = kPairs ? (double)acc[0] - (double)cmp[0] : (double)acc[0];
    __syncthreads();
    if (piece == 0 && lane < B && ti < tend) {
      double s = red[warp * B + lane];
#pragma unroll
      for (int i = 1; i < W; ++i) s += red[(warp + i) * B + lane];
      put(lane, s);
    }
  }
}

// Warp `wi` of the slices.
template <typename T, int B, bool V32, bool FX>
__device__ __forceinline__ void run_slice(const SpmmParams& p, unsigned wi, const T* __restrict__ X,
                                          T* __restrict__ Y, int lane) {
  constexpr int SC = kColLanes<T, B, V32>, K = B / SC;   // lanes per row for its columns, columns of each
  constexpr int NE = Geo<T, B, V32>::NE < K ? Geo<T, B, V32>::NE : K;
  // bucket = last one whose first warp is <= wi (buckets are non-empty, so strictly increasing)
  int lo = 0, hi = p.nbuckets - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.bucket_warp_begin[mid] <= wi) lo = mid;
    else hi = mid - 1;
  }
  const int bkt = lo;
  const int deg = p.bucket_deg[bkt];
  const int pieces = slice_pieces(deg, p.shared), nrows = 32 / (pieces * SC);
  const int unit = (int)(wi - p.bucket_warp_begin[bkt]);
  const int in_bucket = unit / (pieces * SC), piece = lane / (nrows * SC), cl = lane % SC;
  const int srow = (unit % (pieces * SC)) * nrows + lane / SC % nrows;   // row of the slice
  const int64_t si = (int64_t)p.bucket_slice_begin[bkt] + in_bucket;
  const int64_t off = p.bucket_ell_base[bkt] + in_bucket * 32 * (int64_t)deg;
  const int len = ((deg + pieces - 1) / pieces + 3) & ~3;    // steps of a piece
  const int t1 = min(deg, (piece + 1) * len);
  int row = -1;
  if constexpr (!FX) row = __ldcs(p.slice_rows + si * 32 + srow);
  T acc[K], cmp[K];
#pragma unroll
  for (int q = 0; q < K; ++q) acc[q] = cmp[q] = T(0);
  const int32_t* __restrict__ e = p.ell + off + srow;
  const T* __restrict__ x = X + cl * K;
  auto add_row = [&](int c) {
#pragma unroll
    for (int ch = 0; ch < K; ch += NE) {
      T f[NE];
      ld_frag<T, NE>(x + (int64_t)c * B + ch, f);
#pragma unroll
      for (int q = 0; q < NE; ++q) kahan_add(acc[ch + q], cmp[ch + q], f[q]);
    }
  };
  auto plain = [&](int t) {   // steps [t, t1)
    for (; t + 4 <= t1; t += 4) {
      int c[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) c[u] = __ldcs(e + (t + u) * 32);
#pragma unroll
      for (int u = 0; u < 4; ++u) add_row(c[u]);
    }
    for (; t < t1; ++t) add_row(__ldcs(e + t * 32));
  };
  bool done = false;
  if constexpr (FX) {
    if (deg >= kFxMinDegree) {
      Fx fa[K];
      bool bad = false;
#pragma unroll
      for (int q = 0; q < K; ++q) fa[q] = Fx{0, 0u};
      int t = piece * len, groups = 0;
      int c[4];   // the next round's columns, loaded a round ahead
#pragma unroll
      for (int u = 0; u < 4; ++u) c[u] = t + 4 <= t1 ? __ldcs(e + (t + u) * 32) : 0;
      for (; t + 4 <= t1; t += 4) {
        T f[4][K];
#pragma unroll
        for (int u = 0; u < 4; ++u) ld_frag<T, K>(x + (int64_t)c[u] * B, f[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = t + 8 <= t1 ? __ldcs(e + (t + 4 + u) * 32) : 0;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          acc[q] += f[0][q];
          fx_add3(fa[q], f[1][q], f[2][q], f[3][q]);
        }
        if (++groups == kFxGroups) {
#pragma unroll
          for (int q = 0; q < K; ++q) fx_flush(acc[q], fa[q], bad);
          groups = 0;
        }
      }
      for (; t < t1; ++t) add_row(__ldcs(e + t * 32));
#pragma unroll
      for (int q = 0; q < K; ++q) fx_flush(acc[q], fa[q], bad);
      done = !bad;
      if (bad) {
#pragma unroll
        for (int q = 0; q < K; ++q) acc[q] = T(0);
      }
    }
  }
  if (!done) plain(piece * len);
  if constexpr (FX) row = __ldcs(p.slice_rows + si * 32 + srow);   // late: one register less
  T* y = Y + (int64_t)row * B + cl * K;
  if (pieces == 1) {
    if (row >= 0) {
#pragma unroll
      for (int q = 0; q < K; ++q) acc[q] = kahan_value(acc[q], cmp[q]);
      st_row<T, K>(y, acc);
    }
    return;
  }
  // the pieces' sums: lanes 16 apart, then (four pieces) 8 apart, each level also dividing the
  // columns between the two lanes while there are two
  constexpr int H1 = K >= 2 ? K / 2 : 1, H2 = H1 >= 2 ? H1 / 2 : 1;
  bool writer = row >= 0;
  const bool up1 = (lane & 16) != 0, up2 = (lane & 8) != 0;
#pragma unroll
  for (int i = 0; i < H1; ++i) {
    const int j = (i + H1) % K;   // i for a single column, which both lanes keep
    kahan_merge(up1 ? acc[j] : acc[i], up1 ? cmp[j] : cmp[i], up1 ? acc[i] : acc[j], up1 ? cmp[i] : cmp[j], 16, acc[i], cmp[i]);
  }
  if (K >= 2) y += up1 ? H1 : 0;
  else writer = writer && !up1;
  if (pieces == 2) {
    if (writer) {
#pragma unroll
      for (int q = 0; q < H1; ++q) acc[q] = kahan_value(acc[q], cmp[q]);
      st_row<T, H1>(y, acc);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < H2; ++i) {
    const int j = (i + H2) % H1;
    kahan_merge(up2 ? acc[j] : acc[i], up2 ? cmp[j] : cmp[i], up2 ? acc[i] : acc[j], up2 ? cmp[i] : cmp[j], 8, acc[i], cmp[i]);
  }
  if (H1 >= 2) y += up2 ? H2 : 0;
  else writer = writer && !up2;
  if (writer) {
#pragma unroll
    for (int q = 0; q < H2; ++q) acc[q] = kahan_value(acc[q], cmp[q]);
    st_row<T, H2>(y, acc);
  }
}

template <typename T, int B>
constexpr bool kWide = B * sizeof(T) >= 32 && !kUseFx<T, B>;
// Resident CTAs to compile for.  Packed tasks decode besides: FP32 b = 4 spills 144 bytes at 8 CTAs, 24 at
// 6 (4.2 million vertices 879 and 801 us, a million 216 and 192).
template <typename T, int B, bool V32, bool PACKED, bool FX>
constexpr int kMinCtas = FX ? 5
                         : B * sizeof(T) <= 16 ? (PACKED && sizeof(T) == 4 && B == 4 ? 6 : 8)
                                               : (B == 8 ? 5 : (V32 ? 3 : 7));
template <typename T, int B, bool V32, bool PACKED, bool FX>
__global__ void __launch_bounds__(256, (kMinCtas<T, B, V32, PACKED, FX>))
    spmm_main_kernel(const SpmmParams p, const T* __restrict__ X, T* __restrict__ Y, double* __restrict__ partial) {
  __shared__ double red[kWarpsPerCta * B];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t cta = blockIdx.x;
  if (cta < p.ctas4) {
    run_task<T, B, V32, PACKED, FX, 4>(p, cta * 2 + warp / 4, p.wide4, X, Y, partial, warp, lane, red);
  } else if (cta < p.ctas2) {
    run_task<T, B, V32, PACKED, FX, 2>(p, p.wide4 + (cta - p.ctas4) * 4 + warp / 2, p.wide2, X, Y, partial, warp, lane, red);
  } else if (cta < p.task_ctas) {
    const int64_t ti = p.wide2 + (cta - p.ctas2) * kWarpsPerCta + warp;
    if (ti < p.ntasks) run_task<T, B, V32, PACKED, FX, 1>(p, ti, p.ntasks, X, Y, partial, warp, lane, red);
  } else {
    const unsigned wi = (unsigned)(cta - p.task_ctas) * kWarpsPerCta + warp;
    if (wi < p.bucket_warp_begin[p.nbuckets]) run_slice<T, B, V32, FX>(p, wi, X, Y, lane);
  }
}

// s + e <- (s + e) + x exactly up to the rounding of e (Neumaier 1974: the error of every add is
// collected separately).  The larger one by the high words: equal ones have one exponent, which is all
// that the error's formula needs, and the FP64 pipe is spared a comparison.
__device__ __forceinline__ void neumaier_add(double& s, double& e, double x) {
  const double u = s + x;
  const bool up = (__double2hiint(x) & 0x7fffffff) > (__double2hiint(s) & 0x7fffffff);
  const double a = up ? x : s, b = up ? s : x;
  e += (a - u) + b;
  s = u;
}

// Y[hub_rows[h]] = sum of the hub's task partials in compensated FP64, then one rounding to T: an error
// of about 2^-53 |sum| + O(k 2^-106) sum |partial| for any number k of partials (FP64 in both types),
// so a hub adds one rounding to its chunks' errors.  One warp per hub row: lane l adds column l % B of tasks l / B, l / B +
// 32 / B, .. in order, then the lanes of a column are added in a fixed tree (R-MAT with 2^20 vertices,
// FP32 b = 4: 8.4 us with a thread per entry over all of a row's partials, 3.1 us now).
template <typename T, int B>
__global__ void __launch_bounds__(256) hub_reduce_kernel(const int32_t* __restrict__ hub_rows,
                                                         const int32_t* __restrict__ hub_task_begin,
                                                         int64_t nhub, const double* __restrict__ partial,
                                                         T* __restrict__ Y) {
  const int64_t h = (int64_t)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
  if (h >= nhub) return;
  const int lane = threadIdx.x & 31, c = lane % B, slot = lane / B;
  const int t0 = hub_task_begin[h], t1 = hub_task_begin[h + 1];
  const double* src = partial + (int64_t)t0 * B + lane;   // task t0 + slot, column c
  const int steps = (t1 - t0 - slot + 32 / B - 1) / (32 / B);
  double s = steps > 0 ? src[0] : 0.0, e = 0.0;
#pragma unroll 4
  for (int t = 1; t < steps; ++t) neumaier_add(s, e, src[(int64_t)t * 32]);
#pragma unroll
  for (int off = B; off < 32; off <<= 1) {
    const double s2 = __shfl_xor_sync(kFull, s, off), e2 = __shfl_xor_sync(kFull, e, off);
    neumaier_add(s, e, s2);
    e += e2;
  }
  // an infinite partial makes the error term NaN: the plain sum is the result then
  const double r = s + e;
  if (lane < B) Y[(int64_t)hub_rows[h] * B + c] = (T)(r == r ? r : s);
}

// Window size for an L2 access-policy window over `bytes` of X: the device's largest window,
// the persisting set-aside (raised once per device, in this process's context, to the device's
// maximum) bounding it so that the whole window can persist.
static int l2_window_bytes(size_t bytes, size_t* win) {
  static std::mutex mu;
  static size_t maxwin[kMaxDevices], persist[kMaxDevices];
  const int dev = cur_device();
  if (dev < 0) return dev;
  std::lock_guard<std::mutex> lock(mu);
  if (maxwin[dev] == 0) {
    int mw = 0, mp = 0;
    FE_CUDA(cudaDeviceGetAttribute(&mw, cudaDevAttrMaxAccessPolicyWindowSize, dev));
    FE_CUDA(cudaDeviceGetAttribute(&mp, cudaDevAttrMaxPersistingL2CacheSize, dev));
    FE_ARG(mw > 0 && mp > 0, "spmm: this device has no L2 persistence control");
    FE_CUDA(cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, (size_t)mp));
    maxwin[dev] = (size_t)mw;
    persist[dev] = (size_t)mp;
  }
  *win = std::min(bytes, std::min(maxwin[dev], persist[dev]));
  return FE_OK;
}

template <typename T, int B>
static int launch_spmm(const PlanView& pv, const T* X, T* Y, double* partial, cudaStream_t s) {
  SpmmParams p;
  memset(&p, 0, sizeof(p));
  p.colidx = pv.colidx;
  p.tbits = pv.tbits;
  p.tasks = reinterpret_cast<const Task*>(pv.tasks);
  p.ptasks = reinterpret_cast<const PTask*>(pv.tasks);
  p.ntasks = pv.ntasks;
  p.nhub_tasks = pv.nhub_tasks;
  p.slice_rows = pv.slice_rows;
  p.ell = pv.ell;
  p.nbuckets = pv.nbuckets;
  // 256-bit gathers (FP32 rows of at least 32 bytes on a 32-byte boundary): fewer rounds than with
  // 16-byte fragments (R-MAT with 16384 vertices, b = 16: 23 against 37 us; 4.2 million, b = 8: 0.62
  // against 0.64 ms); b = 16 with many columns takes the fragments and four lanes per slice row,
  // whose registers allow seven CTAs instead of three (4.2 million: 1.50 -> 1.03 ms)
  bool v32 = false;
  if constexpr (kWide<T, B>) v32 = ((uintptr_t)X % 32) == 0 && (B < 16 || pv.x_rows <= kWideCols);
  const int col_lanes = v32 ? kColLanes<T, B, true> : kColLanes<T, B, false>;
  p.shared = B > 1 || sizeof(T) == 4 || pv.x_rows <= kSharedCols;
  int64_t warps = 0;
  for (int i = 0; i < pv.nbuckets; ++i) {
    p.bucket_deg[i] = pv.deg_of_bucket[i];
    p.bucket_slice_begin[i] = pv.deg_slice_begin[i];
    p.bucket_warp_begin[i] = (uint32_t)warps;
    p.bucket_ell_base[i] = pv.deg_ell_base[i];
    const int64_t end = i + 1 < pv.nbuckets ? pv.deg_slice_begin[i + 1] : pv.nslices;
    warps += (end - pv.deg_slice_begin[i]) * slice_pieces(pv.deg_of_bucket[i], p.shared) * col_lanes;
  }
  p.bucket_slice_begin[pv.nbuckets] = (int32_t)pv.nslices;
  p.bucket_warp_begin[pv.nbuckets] = (uint32_t)warps;
  p.wide4 = pv.wide4;
  p.wide2 = pv.wide2;
  p.ctas4 = ceil_div(pv.wide4, 2);
  p.ctas2 = p.ctas4 + ceil_div(pv.wide2 - pv.wide4, 4);
  p.task_ctas = p.ctas2 + ceil_div(pv.ntasks - pv.wide2, kWarpsPerCta);
  const int64_t ctas = p.task_ctas + ceil_div(warps, kWarpsPerCta);
  if (ctas > 0) {
    void (*kern)(const SpmmParams, const T*, T*, double*) = nullptr;
    if (v32) {
      if constexpr (kWide<T, B>)
        kern = pv.packed ? spmm_main_kernel<T, B, true, true, false> : spmm_main_kernel<T, B, true, false, false>;
    } else {
      constexpr bool FX = kUseFx<T, B>;
      kern = pv.packed ? spmm_main_kernel<T, B, false, true, FX> : spmm_main_kernel<T, B, false, false, FX>;
      if constexpr (FX && B == 2)
        if (pv.tail_max < kFxTailMax)
          kern = pv.packed ? spmm_main_kernel<T, B, false, true, false> : spmm_main_kernel<T, B, false, false, false>;
    }
    if (pv.l2_persist) {
      // L2 access-policy window on X: its lines are kept (persisting) while the streamed index
      // arrays pass through as streaming accesses (Section 3.3.3's cache-resident dense tiles,
      // with the GPU's L2 as the cache)
      size_t win = 0;
      FE_TRY(l2_window_bytes((size_t)pv.x_rows * B * sizeof(T), &win));
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
      attr[0].val.accessPolicyWindow.base_ptr = const_cast<T*>(X);
      attr[0].val.accessPolicyWindow.num_bytes = win;
      attr[0].val.accessPolicyWindow.hitRatio = 1.0f;
      attr[0].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
      attr[0].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)ctas);
      cfg.blockDim = dim3(256);
      cfg.dynamicSmemBytes = 0;
      cfg.stream = s;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      FE_CUDA(cudaLaunchKernelEx(&cfg, kern, p, X, Y, partial));
    } else {
      kern<<<(unsigned)ctas, 256, 0, s>>>(p, X, Y, partial);
    }
    count_launch();
    FE_CUDA(cudaGetLastError());
  }
  if (pv.nhub > 0) {
    hub_reduce_kernel<T, B><<<(unsigned)ceil_div(pv.nhub, kWarpsPerCta), 256, 0, s>>>(
        pv.hub_rows, pv.hub_task_begin, pv.nhub, partial, Y);
    count_launch();
    FE_CUDA(cudaGetLastError());
  }
  return FE_OK;
}

PlanView resident_view(fe_csr h) {
  const fe_spmm_plan& pl = h->plan;
  PlanView v;
  memset(&v, 0, sizeof(v));
  v.colidx = h->d_colidx;
  v.tbits = pl.d_tbits;
  v.packed = pl.packed;
  v.tasks = pl.d_tasks;
  v.ntasks = pl.ntasks;
  v.nhub_tasks = pl.nhub_tasks;
  v.tail_max = pl.tail_max;
  v.wide4 = pl.wide4;
  v.wide2 = pl.wide2;
  v.slice_rows = pl.d_slice_rows;
  v.ell = pl.d_ell;
  v.nslices = pl.nslices;
  v.nbuckets = pl.nbuckets;
  for (int i = 0; i < pl.nbuckets; ++i) {
    v.deg_of_bucket[i] = pl.deg_of_bucket[i];
    v.deg_slice_begin[i] = pl.deg_slice_begin[i];
    v.deg_ell_base[i] = pl.deg_ell_base[i];
  }
  v.hub_rows = pl.d_hub_rows;
  v.hub_task_begin = pl.d_hub_task_begin;
  v.nhub = pl.nhub;
  v.x_rows = h->ncols;
  v.l2_persist = pl.l2_persist;
  return v;
}

int spmm_view(const PlanView& v, const void* X, void* Y, void* partial, int b, fe_dtype dt,
              cudaStream_t s) {
  if (dt == FE_F32) {
    const float* x = static_cast<const float*>(X);
    float* y = static_cast<float*>(Y);
    double* pa = static_cast<double*>(partial);
    switch (b) {
      case 1: return launch_spmm<float, 1>(v, x, y, pa, s);
      case 2: return launch_spmm<float, 2>(v, x, y, pa, s);
      case 4: return launch_spmm<float, 4>(v, x, y, pa, s);
      case 8: return launch_spmm<float, 8>(v, x, y, pa, s);
      case 16: return launch_spmm<float, 16>(v, x, y, pa, s);
    }
  } else {
    const double* x = static_cast<const double*>(X);
    double* y = static_cast<double*>(Y);
    double* pa = static_cast<double*>(partial);
    switch (b) {
      case 1: return launch_spmm<double, 1>(v, x, y, pa, s);
      case 2: return launch_spmm<double, 2>(v, x, y, pa, s);
      case 4: return launch_spmm<double, 4>(v, x, y, pa, s);
      case 8: return launch_spmm<double, 8>(v, x, y, pa, s);
      case 16: return launch_spmm<double, 16>(v, x, y, pa, s);
    }
  }
  return set_error(FE_ERR_INVALID, "spmm: unsupported b = %d", b);
}

int spmm_resident(fe_csr h, const void* X, void* Y, int b, fe_dtype dt, cudaStream_t s) {
  return spmm_view(resident_view(h), X, Y, h->partials.p, b, dt, s);
}

// ---------------------------------------------------------------- plan (host, at create)

static int dev_upload(fe_csr h, void** dst, const void* src, size_t bytes) {
  *dst = nullptr;
  if (bytes == 0) return FE_OK;
  cudaError_t e = cudaMalloc(dst, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *dst = nullptr;
    return set_error(FE_ERR_OOM, "cudaMalloc(%zu) for the CSR failed: %s", bytes, cudaGetErrorString(e));
  }
  h->allocations.push_back(*dst);
  h->device_bytes += (int64_t)bytes;
  if (src) FE_CUDA(cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice));
  return FE_OK;
}

// Plan of rows [r0, r1): task starts are offsets into hp.tcol, the column indices of the
// panel's task rows only (tail rows are read from the ELL slices); row ids are global.
static int bit_length(uint32_t x) { return x == 0 ? 0 : 32 - __builtin_clz(x); }

size_t plan_row_index_bytes(const int32_t* cols, int64_t d, int tail_max, int hub_chunk, bool packed) {
  if (d <= tail_max || !packed) return 4 * (size_t)d;
  // packed: every chunk of hub_chunk entries is a segment of one gap width, word-aligned
  std::vector<int32_t> sorted;
  const int32_t* c = cols;
  if (!std::is_sorted(cols, cols + d)) {
    sorted.assign(cols, cols + d);
    std::sort(sorted.begin(), sorted.end());
    c = sorted.data();
  }
  size_t bytes = 0;
  for (int64_t s0 = 0; s0 < d; s0 += hub_chunk) {
    const int64_t s1 = std::min<int64_t>(d, s0 + hub_chunk);
    int w = 1;
    for (int64_t k = s0 + 1; k < s1; ++k) w = std::max(w, bit_length((uint32_t)(c[k] - c[k - 1])));
    bytes += 4 * (size_t)ceil_div((s1 - s0) * w, 32) + 16;  // + the larger task record
  }
  return bytes;
}

// Packed index format: each task's sorted columns become gap fields of the task's width w
// (g_0 = 0, g_k = c_k - c_{k-1}) in a word-aligned segment of the bit stream, so that tasks can
// be encoded in parallel; two zero words pad the end (the decoder reads a two-word window).
static void pack_tasks(HostPlan& hp) {
  const int64_t nt = hp.ntasks;
  hp.ptasks.resize(nt);
  std::vector<int64_t> words(nt + 1, 0);
  #pragma omp parallel for schedule(dynamic, 256)
  for (int64_t t = 0; t < nt; ++t) {
    const Task& tk = hp.tasks[t];
    const int32_t* c = hp.tcol.data() + tk.start;
    int w = 1;
    for (int k = 1; k < tk.len; ++k) w = std::max(w, bit_length((uint32_t)(c[k] - c[k - 1])));
    hp.ptasks[t] = PTask{0, tk.row, tk.len, c[0], w, 0, 0};
    words[t + 1] = ceil_div((int64_t)tk.len * w, 32);
  }
  for (int64_t t = 0; t < nt; ++t) words[t + 1] += words[t];
  hp.tbits.assign(words[nt] + 2, 0u);
  #pragma omp parallel for schedule(dynamic, 256)
  for (int64_t t = 0; t < nt; ++t) {
    PTask& pt = hp.ptasks[t];
    pt.woff = words[t];
    const int32_t* c = hp.tcol.data() + hp.tasks[t].start;
    uint32_t* out = hp.tbits.data() + words[t];
    const int w = pt.w;
    for (int k = 1; k < pt.len; ++k) {
      const uint32_t g = (uint32_t)(c[k] - c[k - 1]);
      const int64_t bit = (int64_t)k * w;
      const int64_t wi = bit >> 5;
      const int sh = (int)(bit & 31);
      out[wi] |= g << sh;
      if (sh + w > 32) out[wi + 1] |= g >> (32 - sh);
    }
  }
  hp.tcol.clear();
  hp.tcol.shrink_to_fit();
  hp.tasks.clear();
  hp.tasks.shrink_to_fit();
  hp.packed = true;
}

void plan_wide(const HostPlan& hp, int64_t ncols, bool streamed, int64_t* wide4, int64_t* wide2) {
  *wide4 = *wide2 = 0;
  if (ncols > kWideCols && !streamed) return;
  // the tasks after the hub chunks are rows by descending degree
  int64_t t = hp.nhub_tasks;
  auto len = [&](int64_t i) { return hp.packed ? hp.ptasks[i].len : hp.tasks[i].len; };
  while (t < hp.ntasks && len(t) > 2 * kWideLen) ++t;
  *wide4 = t;
  while (t < hp.ntasks && len(t) > kWideLen) ++t;
  *wide2 = t;
}

int build_host_plan(const int64_t* rowptr, const int32_t* colidx, int64_t r0, int64_t r1,
                    int tail_max, int hub_min, int hub_chunk, bool packed, HostPlan& hp) {
  hp = HostPlan();
  std::vector<int64_t> tail_cnt(tail_max + 1, 0);
  std::vector<int64_t> mid_cnt(hub_min + 1, 0);
  int64_t nhub = 0, nhub_tasks = 0;
  for (int64_t i = r0; i < r1; ++i) {
    const int64_t d = rowptr[i + 1] - rowptr[i];
    hp.max_degree = std::max(hp.max_degree, d);
    if (d <= tail_max) tail_cnt[d]++;
    else if (d <= hub_min) mid_cnt[d]++;
    else { nhub++; nhub_tasks += ceil_div(d, hub_chunk); }
  }
  hp.rows_empty = tail_cnt[0];
  for (int d = 1; d <= tail_max; ++d) hp.rows_tail += tail_cnt[d];
  for (int d = tail_max + 1; d <= hub_min; ++d) hp.rows_mid += mid_cnt[d];
  hp.rows_hub = nhub;
  FE_ARG(nhub_tasks < INT32_MAX, "spmm plan: too many hub tasks");
  // tail slices: buckets by degree, descending, empty buckets dropped
  int64_t nslices = 0, ell_total = 0;
  std::vector<int> bucket_of_deg(tail_max + 1, -1);
  for (int d = tail_max; d >= 0; --d) {
    if (tail_cnt[d] == 0) continue;
    const int bk = hp.nbuckets++;
    bucket_of_deg[d] = bk;
    hp.deg_of_bucket[bk] = d;
    hp.deg_slice_begin[bk] = (int32_t)nslices;
    hp.deg_ell_base[bk] = ell_total;
    const int64_t sl = ceil_div(tail_cnt[d], 32);
    nslices += sl;
    ell_total += sl * 32 * d;
  }
  FE_ARG(nslices < INT32_MAX / 4, "spmm plan: too many tail slices");
  hp.nslices = nslices;
  hp.slice_rows.assign(nslices * 32, -1);
  std::vector<int64_t> cursor(tail_max + 1, 0);
  for (int d = 0; d <= tail_max; ++d)
    if (bucket_of_deg[d] >= 0) cursor[d] = (int64_t)hp.deg_slice_begin[bucket_of_deg[d]] * 32;
  // tasks: hub chunks first, then mid rows by degree descending (stable in row order)
  std::vector<int64_t> mid_pos(hub_min + 2, 0);
  {
    int64_t acc = nhub_tasks;
    for (int d = hub_min; d > tail_max; --d) { mid_pos[d] = acc; acc += mid_cnt[d]; }
  }
  hp.ntasks = nhub_tasks + hp.rows_mid;
  hp.nhub_tasks = nhub_tasks;
  hp.nhub = nhub;
  hp.tasks.resize(hp.ntasks);
  hp.hub_rows.resize(nhub);
  hp.hub_task_begin.resize(nhub + 1);
  int64_t ht = 0, hi = 0, tpos = 0;
  {
    int64_t tnnz = 0;
    for (int64_t i = r0; i < r1; ++i) {
      const int64_t d = rowptr[i + 1] - rowptr[i];
      if (d > tail_max) tnnz += d;
    }
    hp.tcol.resize(tnnz > 0 ? tnnz : 1);
  }
  for (int64_t i = r0; i < r1; ++i) {
    const int64_t d = rowptr[i + 1] - rowptr[i];
    if (d <= tail_max) {
      hp.slice_rows[cursor[d]++] = (int32_t)i;
      continue;
    }
    memcpy(hp.tcol.data() + tpos, colidx + rowptr[i], sizeof(int32_t) * (size_t)d);
    if (packed && !std::is_sorted(hp.tcol.data() + tpos, hp.tcol.data() + tpos + d))
      std::sort(hp.tcol.data() + tpos, hp.tcol.data() + tpos + d);
    if (d <= hub_min) {
      hp.tasks[mid_pos[d]++] = Task{tpos, (int32_t)i, (int32_t)d};
    } else {
      hp.hub_rows[hi] = (int32_t)i;
      hp.hub_task_begin[hi] = (int32_t)ht;
      for (int64_t c = 0; c < d; c += hub_chunk)
        hp.tasks[ht++] = Task{tpos + c, (int32_t)i, (int32_t)std::min<int64_t>(hub_chunk, d - c)};
      ++hi;
    }
    tpos += d;
  }
  hp.tcol_total = tpos;
  hp.hub_task_begin[nhub] = (int32_t)ht;
  // ELL fill (transposed per slice; padding lanes read column 0 and are not written)
  hp.ell.assign(ell_total > 0 ? ell_total : 1, 0);
  for (int bk = 0; bk < hp.nbuckets; ++bk) {
    const int d = hp.deg_of_bucket[bk];
    if (d == 0) continue;
    const int64_t s0 = hp.deg_slice_begin[bk];
    const int64_t s1 = (bk + 1 < hp.nbuckets) ? hp.deg_slice_begin[bk + 1] : nslices;
    int32_t* ell = hp.ell.data();
    const int32_t* srows = hp.slice_rows.data();
    const int64_t ebase = hp.deg_ell_base[bk];
    #pragma omp parallel for schedule(static)
    for (int64_t sl = s0; sl < s1; ++sl) {
      int32_t* e = ell + ebase + (sl - s0) * 32 * d;
      for (int lane = 0; lane < 32; ++lane) {
        const int32_t r = srows[sl * 32 + lane];
        for (int t = 0; t < d; ++t) e[t * 32 + lane] = r >= 0 ? colidx[rowptr[r] + t] : 0;
      }
    }
  }
  hp.ell_total = ell_total;
  if (packed) pack_tasks(hp);
  return FE_OK;
}

int spmm_build_plan(fe_csr h, const int64_t* rowptr, const int32_t* colidx_raw, int tail_max,
                    int hub_min, int hub_chunk, bool packed) {
  const int64_t n = h->n;
  const int32_t* colidx = colidx_raw;
  fe_spmm_plan& pl = h->plan;
  pl.tail_max = tail_max;
  pl.hub_min = hub_min;
  pl.hub_chunk = hub_chunk;
  HostPlan hp;
  FE_TRY(build_host_plan(rowptr, colidx, 0, n, tail_max, hub_min, hub_chunk, packed, hp));
  pl.packed = packed ? 1 : 0;
  h->max_degree = hp.max_degree;
  h->rows_empty = hp.rows_empty;
  h->rows_tail = hp.rows_tail;
  h->rows_mid = hp.rows_mid;
  h->rows_hub = hp.rows_hub;
  pl.nbuckets = hp.nbuckets;
  for (int i = 0; i < hp.nbuckets; ++i) {
    pl.deg_of_bucket[i] = hp.deg_of_bucket[i];
    pl.deg_slice_begin[i] = hp.deg_slice_begin[i];
    pl.deg_ell_base[i] = hp.deg_ell_base[i];
  }
  pl.nslices = hp.nslices;
  pl.ntasks = hp.ntasks;
  pl.nhub_tasks = hp.nhub_tasks;
  plan_wide(hp, h->ncols, false, &pl.wide4, &pl.wide2);
  pl.nhub = hp.nhub;
  if (packed) {
    FE_TRY(dev_upload(h, (void**)&pl.d_tbits, hp.tbits.data(), sizeof(uint32_t) * hp.tbits.size()));
    FE_TRY(dev_upload(h, &pl.d_tasks, hp.ptasks.data(), sizeof(PTask) * hp.ntasks));
    pl.index_bytes = (int64_t)(sizeof(uint32_t) * hp.tbits.size() + sizeof(int32_t) * hp.ell_total);
  } else {
    FE_TRY(dev_upload(h, (void**)&h->d_colidx, hp.tcol.data(), sizeof(int32_t) * hp.tcol_total));
    FE_TRY(dev_upload(h, &pl.d_tasks, hp.tasks.data(), sizeof(Task) * hp.ntasks));
    pl.index_bytes = (int64_t)(sizeof(int32_t) * (hp.tcol_total + hp.ell_total));
  }
  FE_TRY(dev_upload(h, (void**)&pl.d_slice_rows, hp.slice_rows.data(), sizeof(int32_t) * hp.slice_rows.size()));
  FE_TRY(dev_upload(h, (void**)&pl.d_ell, hp.ell.data(), sizeof(int32_t) * hp.ell_total));
  FE_TRY(dev_upload(h, (void**)&pl.d_hub_rows, hp.hub_rows.data(), sizeof(int32_t) * hp.nhub));
  FE_TRY(dev_upload(h, (void**)&pl.d_hub_task_begin, hp.hub_task_begin.data(), sizeof(int32_t) * (hp.nhub + 1)));
  if (hp.nhub_tasks > 0) {
    FE_TRY(h->partials.alloc(sizeof(double) * 16 * hp.nhub_tasks));
    h->device_bytes += (int64_t)h->partials.bytes;
  }
  return FE_OK;
}

}  // namespace fe
