// Rayleigh-Ritz on the projected matrix (Algorithm 1 steps (2)-(4)) and the Krylov-Schur
// restart of the small matrix, on the device.
//
// T = (H_m + H_m^T) / 2 (m x m) is diagonalised, the Ritz values are ordered by `which`, and each
// Ritz pair gets its residual estimate rho_c = ||H[m:m+b, 0:m] y_c|| (the coupling of the last
// block to the next basis block, since A V_m = V_m H_m + V_{NB} H[m:m+b, :]).
//
// m <= 160 (ritz_cluster_kernel): FP64 runs at 1/64 of the FP32 rate here, so FP64 is spent on
// matrix products only, and those are spread over a thread-block cluster.  One iteration turns
// the FP64 vectors Q (T ~ Q D Q^T) into better ones:
//   G = Q^T Q, W = T Q, S = Q^T W                                    (FP64, all CTAs)
//   R = I - G;  d = diag S + R_ii theta_i,
//   N_ij = S_ij + R_ij (theta_i + theta_j) / 2                       (FP64, then N in FP32)
//     -- to first order in R the projection onto the orthonormalised Q (I + R / 2);
//   E: the rotation that diagonalises D + N, relative to I           (FP32, one CTA)
//   Q <- Q + Q (R / 2 + E)                                           (FP64, all CTAs)
// N and E are small, so their FP32 rounding is relative to something small: the error of an
// iteration is about 1e-7 of the previous one (and the square of the previous one where E is
// taken to first order).  The first iteration has Q = I and S = T: a whole FP32 Jacobi
// diagonalisation.  The second finds N ~ 1e-7 |T| and runs one or two sweeps; the third finds
// |N_ij / (d_j - d_i)| below 1e-8, takes E_ij = N_ij / (d_j - d_i) and is the last.  The
// iterative refinement with matrix products and the treatment of R follow Ogita & Aishima,
// "Iterative refinement for symmetric eigenvalue decomposition", Japan J. Indust. Appl. Math. 35
// (2018); solving for E by Jacobi in FP32 makes close eigenvalues no special case.
// Measured per call on a GB300 against FP32 and FP64 Jacobi sweeps on one CTA: m = 32 590 -> 110
// us (seven FP32 sweeps of 9 us, FP64 18 us), m = 128 14.65 -> 1.15 ms (eight sweeps of 99 us,
// FP64 0.23 ms).  What bounds it now: the sweeps' two barriers and dependent chains per step (31
// steps of 0.29 us at m = 32), at m = 128 their shared-memory traffic.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "fe_internal.cuh"
#include "ritz_layout.cuh"

namespace fe {

// tan of the Jacobi angle that diagonalises [app apq; apq aqq] (Golub & Van Loan Section
// 8.5.2), evaluated in FP32.  FP64 entries are first scaled by a power of two and the diagonal
// difference is taken in FP64, so only the final quotient and square root are FP32.  Returns
// 0 when apq is negligible at FP32 range.  Any t gives an exactly orthogonal rotation once c
// and s are formed from it (jacobi_cs), so an inexact t only leaves a small (p,q) entry for
// the next sweep.
__device__ __forceinline__ float jacobi_tan(float app, float apq, float aqq) {
  if (apq == 0.f) return 0.f;
  const float tau = (aqq - app) / (2.f * apq);
  if (fabsf(tau) > 1e18f) return 0.5f / tau;
  return (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
}
__device__ __forceinline__ float jacobi_tan(double app, double apq, double aqq) {
  if (apq == 0.0) return 0.f;
  const double mx = fmax(fmax(fabs(app), fabs(aqq)), fabs(apq));
  int e;
  frexp(mx, &e);
  const double sc = ldexp(1.0, -e);
  const float d = (float)((aqq - app) * sc), f = (float)(apq * sc);
  if (f == 0.f) return 0.f;
  const float tau = d / (2.f * f);
  if (fabsf(tau) > 1e18f) return 0.5f / tau;
  return (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
}
// c = 1 / sqrt(1 + t^2), s = t c in T: FP32 estimate, then (FP64) two Newton steps for the
// reciprocal square root, so that c^2 + s^2 = 1 to T's rounding.
__device__ __forceinline__ void jacobi_cs(float t, float& c, float& s) {
  c = rsqrtf(1.f + t * t);
  s = t * c;
}
__device__ __forceinline__ void jacobi_cs(float t32, double& c, double& s) {
  const double t = (double)t32, u = 1.0 + t * t;
  double r = (double)rsqrtf((float)u);
  r = r * (1.5 - 0.5 * u * r * r);
  r = r * (1.5 - 0.5 * u * r * r);
  c = r;
  s = t * r;
}

// Sum over the block of one value per thread (all threads call it).
__device__ double ritz_block_sum(double v, double* red) {
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < (nth + 31) / 32; ++w) s += red[w];
    red[0] = s;
  }
  __syncthreads();
  const double s = red[0];
  __syncthreads();
  return s;
}

// e / d for 0 <= e < 2^22 and 1 <= d < 2^11, with inv = 1 / d: an FP32 estimate corrected once
// (an integer division would be a long instruction sequence inside the work loops).
__device__ __forceinline__ int small_div(int e, int d, float inv) {
  int q = (int)((float)e * inv);
  const int r = e - q * d;
  q += r < 0 ? -1 : (r >= d ? 1 : 0);
  return q;
}

// The e-th of the pairs (k, k2), k <= k2 < np (the upper triangle of the step's 2 x 2 blocks,
// np (np + 1) / 2 of them), from a triangular-number inversion in FP32 corrected in integers.
__device__ __forceinline__ void tri_pair(int e, int np, int& k, int& k2) {
  const int f = np * (np + 1) / 2 - 1 - e;   // reversed index: row r holds r + 1 items
  int r = (int)((sqrtf(8.f * (float)f + 1.f) - 1.f) * 0.5f);
  if ((r + 1) * (r + 2) / 2 <= f) ++r;
  if (r * (r + 1) / 2 > f) --r;
  const int o = f - r * (r + 1) / 2;
  k = np - 1 - r;
  k2 = np - 1 - o;
}

// Parallel cyclic Jacobi sweeps on the symmetric mp x mp matrix A (row stride ld), with
// Q <- Q J accumulated, until the off-diagonal Frobenius norm squared is <= thresh or after
// max_sweeps.  Returns the sweeps run; *conv tells whether the threshold was met.
template <typename T>
__device__ int jacobi_sweeps(T* A, T* Q, int ld, int m, int mp, double thresh, int max_sweeps,
                             T* cs, T* sn, int* pp, int* pq, double* red, bool* conv) {
  const int tid = threadIdx.x, nth = blockDim.x;
  const int np = mp / 2;
  const float inv_mp = 1.f / (float)mp, inv_np = 1.f / (float)np;
  const int ntri = np * (np + 1) / 2;
  int sweeps = 0;
  while (true) {
    double v = 0.0;
    for (int e = tid; e < mp * mp; e += nth) {
      const int i = small_div(e, mp, inv_mp), j = e - i * mp;
      if (i != j) v += (double)A[i * ld + j] * (double)A[i * ld + j];
    }
    const double off2 = ritz_block_sum(v, red);
    if (off2 <= thresh || sweeps >= max_sweeps) {
      *conv = off2 <= thresh;
      return sweeps;
    }
    ++sweeps;
    for (int step = 0; step < mp - 1; ++step) {
      // circle method: position 0 fixed, positions 1..mp-1 rotate by `step`
      for (int k = tid; k < np; k += nth) {
        auto pos = [&](int i) { return i == 0 ? 0 : ((i - 1 + step) % (mp - 1)) + 1; };
        int p = pos(k), q = pos(mp - 1 - k);
        if (p > q) { int t = p; p = q; q = t; }
        T c = T(1), sv = T(0);
        if (q < m) {
          const float t = jacobi_tan(A[p * ld + p], A[p * ld + q], A[q * ld + q]);
          if (t != 0.f) jacobi_cs(t, c, sv);
        }
        pp[k] = p;
        pq[k] = q;
        cs[k] = c;
        sn[k] = sv;
      }
      __syncthreads();
      // A <- J^T A J as independent 2 x 2 blocks (rows of pair k, columns of pair k2, k <= k2,
      // mirrored to the lower triangle), and Q <- Q J by column pairs: the step's pairs are
      // disjoint, so no two work items touch the same entry and one barrier suffices.
      for (int e = tid; e < ntri + mp * np; e += nth) {
        if (e < ntri) {
          int k, k2;
          tri_pair(e, np, k, k2);
          const T s1 = sn[k], s2 = sn[k2];
          if (s1 == T(0) && s2 == T(0)) continue;
          const T c1 = cs[k], c2 = cs[k2];
          const int p1 = pp[k], q1 = pq[k];
          if (k == k2) {
            // the pair's own block: full transform (t need not be exact)
            const T app = A[p1 * ld + p1], aqq = A[q1 * ld + q1], apq = A[p1 * ld + q1];
            const T cc = c1 * c1, ss = s1 * s1, cs2 = c1 * s1;
            A[p1 * ld + p1] = cc * app - T(2) * cs2 * apq + ss * aqq;
            A[q1 * ld + q1] = ss * app + T(2) * cs2 * apq + cc * aqq;
            const T npq = cs2 * (app - aqq) + (cc - ss) * apq;
            A[p1 * ld + q1] = npq;
            A[q1 * ld + p1] = npq;
          } else {
            const int p2 = pp[k2], q2 = pq[k2];
            const T x00 = A[p1 * ld + p2], x01 = A[p1 * ld + q2];
            const T x10 = A[q1 * ld + p2], x11 = A[q1 * ld + q2];
            const T y00 = c1 * x00 - s1 * x10, y01 = c1 * x01 - s1 * x11;
            const T y10 = s1 * x00 + c1 * x10, y11 = s1 * x01 + c1 * x11;
            const T z00 = c2 * y00 - s2 * y01, z01 = s2 * y00 + c2 * y01;
            const T z10 = c2 * y10 - s2 * y11, z11 = s2 * y10 + c2 * y11;
            A[p1 * ld + p2] = z00;
            A[p1 * ld + q2] = z01;
            A[q1 * ld + p2] = z10;
            A[q1 * ld + q2] = z11;
            A[p2 * ld + p1] = z00;
            A[q2 * ld + p1] = z01;
            A[p2 * ld + q1] = z10;
            A[q2 * ld + q1] = z11;
          }
        } else {
          const int e2 = e - ntri;
          const int i = small_div(e2, np, inv_np), k = e2 - i * np;
          const T sk = sn[k];
          if (sk == T(0)) continue;
          const T ck = cs[k];
          const int p = pp[k], q = pq[k];
          const T vp = Q[i * ld + p], vq = Q[i * ld + q];
          Q[i * ld + p] = ck * vp - sk * vq;
          Q[i * ld + q] = sk * vp + ck * vq;
        }
      }
      __syncthreads();
    }
  }
}

// ------------------------------------------------------------ m <= 160: one cluster
constexpr int kRitzMaxIter = 8;        // refinement iterations (three are the rule)
constexpr float kTinyAngle = 1e-8f;    // first-order E: its error is the angle's square

// Global workspace (L2-resident): six mp x mp FP64 matrices, N in FP32, two diagonals, the
// rotation logs of two sweeps, control words.
struct RitzWork {
  double *T, *Q, *Q2, *G, *W, *X, *d0, *d1;
  float* N;
  float2* log;     // [2][(mp - 1) * np]: (cos - 1, sin) of the step's pairs
  unsigned* ctl;   // [0] max |R| (float bits), [1] mode, [2] done, [3..4] another sweep follows
};
constexpr int kRitzCtl = 8;

__host__ __device__ inline size_t ritz_cluster_doubles(int m) {
  const size_t mp = m + (m & 1), np = mp / 2;
  return 6 * mp * mp + 2 * mp + (mp * mp + 1) / 2 + 2 * (mp - 1) * np + kRitzCtl;
}

__device__ inline RitzWork ritz_cluster_work(double* w, int mp) {
  const size_t mat = (size_t)mp * mp, np = mp / 2;
  RitzWork r;
  r.T = w;
  r.Q = w + mat;
  r.Q2 = w + 2 * mat;
  r.G = w + 3 * mat;
  r.W = w + 4 * mat;
  r.X = w + 5 * mat;
  r.d0 = w + 6 * mat;
  r.d1 = r.d0 + mp;
  r.log = reinterpret_cast<float2*>(r.d1 + mp);
  r.ctl = reinterpret_cast<unsigned*>(r.log + 2 * (mp - 1) * np);
  r.N = reinterpret_cast<float*>(r.ctl + 2 * kRitzCtl);
  return r;
}

// All threads of all CTAs of the cluster; global writes before it are visible after it.
__device__ __forceinline__ void ritz_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void ritz_bar(int threads) {
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

// Maximum over the block of one non-negative float per thread.
__device__ float ritz_block_max(float v, float* red) {
  const int tid = threadIdx.x;
  for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  v = (tid & 31) < (int)(blockDim.x >> 5) ? red[tid & 31] : 0.f;
  for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
  __syncthreads();
  return v;
}

// FP64 bits as an integer that orders like the value (for comparisons off the FP64 pipe).
// Negating the value negates the key.
__device__ __forceinline__ long long ritz_key(double x) {
  const long long v = __double_as_longlong(x);
  return v < 0 ? -(v & 0x7fffffffffffffffll) : v;
}

// Hardware approximations, subnormals flushed (an inexact rotation angle only leaves a small
// pivot, and the error of its cosine and sine is part of R in the next iteration).
__device__ __forceinline__ float ritz_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ritz_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// CTA 0's matrix during the sweeps, in shared memory: two copies of the entries (ritz_entry) and
// of the diagonal by slot (unevaluated sums of two floats), and a step's (cos - 1, sin).
struct RitzMat {
  float *n0, *n1;
  float2 *d0, *d1, *cs;
};

__device__ __forceinline__ void ritz_swap(RitzMat& mt) {
  float* tn = mt.n0; mt.n0 = mt.n1; mt.n1 = tn;
  float2* td = mt.d0; mt.d0 = mt.d1; mt.d1 = td;
}

// One sweep of the parallel cyclic Jacobi method ("round-robin" ordering, Brent & Luk 1985: each
// of the mp - 1 steps rotates np = mp / 2 disjoint index pairs), with the threads of warps below
// nact / 32; mt.n0, mt.d0 hold the matrix before and after.  The rotations also go to `log`.
// Blocks item0 + u nact < nitems are this thread's: kk their pairs (k | k2 << 16), to where their
// four entries go.  A pair is left alone when
// |N_pq| <= skip, or when it is below tau (N's own uncertainty) and its angle would not be
// tiny; isc: a power of two that brings |T| near 1.  psum: sum of the squared pivots; tmax:
// largest |tan| (both of this thread).
// What bounds it: two barriers and two dependent chains per step (rotation, block update), each
// thread's addresses fixed; at mp = 128 the 11 shared-memory wavefronts per 32 blocks.
template <int ITEMS>
__device__ __forceinline__ void ritz_sweep(RitzMat& mt, int mp, int nact, int item0, int nitems,
                                           const int (&to)[ITEMS][2], const int (&kk)[ITEMS],
                                           float skip, float tau, float isc, float2* log, float* psum,
                                           float* tmax) {
  const int tid = threadIdx.x, np = mp / 2, nt = nitems;
  float ps = 0.f, tm = 0.f;
  const int sp = tid, sq = mp - 1 - tid;
  const int tp = ritz_shift(sp, mp), tq = ritz_shift(sq, mp);
  const int tres = tid < np ? ritz_entry(tp, tq, mp) : 0;
  for (int step = 0; step < mp - 1; ++step) {
    float cm = 0.f, s = 0.f;
    if (tid < np) {
      const float n = mt.n0[4 * nt + tid];
      const float2 dp = mt.d0[sp], dq = mt.d0[sq];
      const float gap = (dq.x - dp.x) + (dq.y - dp.y);
      const float an = fabsf(n);
      const float g = fabsf(gap) * isc, h = 2.f * isc * n;
      // cos 2a = g / w, sin 2a = h / w with w = |(g, h)|; c^2 = (1 + cos 2a) / 2
      const float iw = ritz_rsqrt(fmaf(g, g, h * h));
      const bool rot = an > skip && (an > tau || an <= kTinyAngle * fabsf(gap));
      const float c2 = rot ? fmaf(0.5f * g, iw, 0.5f) : 1.f, ic = ritz_rsqrt(c2), c = c2 * ic;
      s = rot ? copysignf(0.5f, gap) * h * (iw * ic) : 0.f;
      cm = -s * s * ritz_rcp(1.f + c);
      const float t = s * ic, dn = t * n;
      // the pivot's remainder: c s (d_p - d_q) + (c^2 - s^2) n
      const float left = rot ? c2 * fmaf(fmaf(-t, t, 1.f), n, -t * gap) : n;
      mt.cs[tid] = make_float2(cm, s);
      mt.n1[tres] = left;
      const float lo1 = dp.y - dn, h1 = dp.x + lo1;
      mt.d1[tp] = make_float2(h1, lo1 - (h1 - dp.x));
      const float lo2 = dq.y + dn, h2 = dq.x + lo2;
      mt.d1[tq] = make_float2(h2, lo2 - (h2 - dq.x));
      if (rot) ps = fmaf(n, n, ps);
      tm = fmaxf(tm, fabsf(t));
    }
    ritz_bar(nact);
    if (tid < np) log[step * np + tid] = make_float2(cm, s);
    // N <- J^T N J as independent 2 x 2 blocks (rows of pair k, columns of pair k2, k < k2); all
    // loads of the thread's blocks are issued before the first store
    float2 r1[ITEMS], r2[ITEMS];
    float x[ITEMS][4];
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      const int e = ritz_read(item0 + u * nact, nitems);
      r1[u] = mt.cs[kk[u] & 0xffff];
      r2[u] = mt.cs[kk[u] >> 16];
#pragma unroll
      for (int v = 0; v < 4; ++v) x[u][v] = mt.n0[v * nt + e];
    }
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      const float y00 = x[u][0] + fmaf(r1[u].x, x[u][0], -r1[u].y * x[u][2]);
      const float y01 = x[u][1] + fmaf(r1[u].x, x[u][1], -r1[u].y * x[u][3]);
      const float y10 = x[u][2] + fmaf(r1[u].x, x[u][2], r1[u].y * x[u][0]);
      const float y11 = x[u][3] + fmaf(r1[u].x, x[u][3], r1[u].y * x[u][1]);
      if (item0 + u * nact < nitems) {
        mt.n1[to[u][0] & 0xffff] = y00 + fmaf(r2[u].x, y00, -r2[u].y * y01);
        mt.n1[to[u][0] >> 16] = y01 + fmaf(r2[u].x, y01, r2[u].y * y00);
        mt.n1[to[u][1] & 0xffff] = y10 + fmaf(r2[u].x, y10, -r2[u].y * y11);
        mt.n1[to[u][1] >> 16] = y11 + fmaf(r2[u].x, y11, r2[u].y * y10);
      }
    }
    ritz_bar(nact);
    ritz_swap(mt);
  }
  *psum = ps;
  *tmax = tm;
}

__device__ __forceinline__ int ritz_next(int p, int mp) { return p == 0 ? 0 : (p == mp - 1 ? 1 : p + 1); }

// One row of E <- (I + E) J - I over a sweep's logged rotations, one warp; row: mp floats of
// shared memory.  np <= 32: lane k keeps the entries of slots k and mp - 1 - k in registers and
// the slots move by shuffles; otherwise the entries stay in shared memory.
__device__ void ritz_apply_row(float* row, int i, int mp, const float2* log) {
  const int lane = threadIdx.x & 31, np = mp / 2;
  constexpr int D = 8;   // steps whose rotations are in flight
  if (np <= 32) {
    const bool on = lane < np;
    int p = lane, q = mp - 1 - lane;
    float ep = on ? row[p] : 0.f, eq = on ? row[q] : 0.f;
    for (int s0 = 0; s0 < mp - 1; s0 += D) {
      float2 r[D];
#pragma unroll
      for (int t = 0; t < D; ++t)
        r[t] = (s0 + t < mp - 1 && on) ? log[(s0 + t) * np + lane] : make_float2(0.f, 0.f);
#pragma unroll
      for (int t = 0; t < D; ++t) {
        if (s0 + t >= mp - 1) break;
        const float vp = ep + (i == p ? 1.f : 0.f), vq = eq + (i == q ? 1.f : 0.f);
        const float np_ = ep + fmaf(r[t].x, vp, -r[t].y * vq), nq_ = eq + fmaf(r[t].x, vq, r[t].y * vp);
        const float dn = __shfl_down_sync(0xffffffffu, np_, 1), up = __shfl_up_sync(0xffffffffu, nq_, 1);
        ep = lane == 0 ? np_ : (lane == np - 1 ? nq_ : dn);
        eq = lane == 0 ? (np == 1 ? nq_ : dn) : up;
        p = ritz_next(p, mp);
        q = ritz_next(q, mp);
      }
    }
    if (on) {
      row[lane] = ep;
      row[mp - 1 - lane] = eq;
    }
    return;
  }
  constexpr int U = (kRitzOneMax / 2 + 31) / 32;
  int p[U], q[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    p[u] = lane + 32 * u;
    q[u] = mp - 1 - p[u];
  }
  constexpr int D2 = 4;
  for (int s0 = 0; s0 < mp - 1; s0 += D2) {
    float2 r[D2][U];
#pragma unroll
    for (int t = 0; t < D2; ++t)
#pragma unroll
      for (int u = 0; u < U; ++u)
        r[t][u] = (s0 + t < mp - 1 && lane + 32 * u < np) ? log[(s0 + t) * np + lane + 32 * u] : make_float2(0.f, 0.f);
#pragma unroll
    for (int t = 0; t < D2; ++t) {
      if (s0 + t >= mp - 1) break;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (lane + 32 * u < np) {
          const float ep = row[p[u]], eq = row[q[u]];
          const float vp = ep + (i == p[u] ? 1.f : 0.f), vq = eq + (i == q[u] ? 1.f : 0.f);
          row[p[u]] = ep + fmaf(r[t][u].x, vp, -r[t][u].y * vq);
          row[q[u]] = eq + fmaf(r[t][u].x, vq, r[t][u].y * vp);
          p[u] = ritz_next(p[u], mp);
          q[u] = ritz_next(q[u], mp);
        }
      }
      __syncwarp();
    }
  }
}

// Shared memory: CTA 0 holds the sweep's matrix, the others their rows of E.  ITEMS: 2 x 2 blocks
// per thread of CTA 0.
template <int ITEMS>
__global__ void __launch_bounds__(512, 1)
    ritz_cluster_kernel(const double* __restrict__ H, int m, int b, int which, int max_sweeps, double tol,
                        double* __restrict__ theta_out, double* __restrict__ Y_out,
                        double* __restrict__ rho_out, int* __restrict__ info, double* work) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int mp = m + (m & 1);  // even size; index m (if odd) is a zero dummy never rotated
  const int np = mp / 2;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x, ncta = gridDim.x;   // the grid is one cluster
  const int nth = blockDim.x, nwarps = nth / 32;
  RitzWork w = ritz_cluster_work(work, mp);
  __shared__ float red[32];
  __shared__ double redd[32];
  __shared__ int order[kRitzOneMax];
  __shared__ int s_mode, s_done, s_more;
  float* sm = reinterpret_cast<float*>(smem_raw);
  // this thread's 2 x 2 blocks (pairs k < k2) of CTA 0's sweeps
  const int nitems = ritz_items(np);
  const int nact = ritz_active(np, nth);
  RitzMat mt;
  mt.cs = reinterpret_cast<float2*>(sm);
  mt.d0 = mt.cs + np;
  mt.d1 = mt.d0 + mp;
  mt.n0 = reinterpret_cast<float*>(mt.d1 + mp);
  mt.n1 = mt.n0 + ritz_copy(np);
  int to[ITEMS][2], kk[ITEMS];
#pragma unroll
  for (int u = 0; u < ITEMS; ++u) {
    const int e = tid + u * nact;
    to[u][0] = to[u][1] = kk[u] = 0;
    if (rank == 0 && tid < nact && e < nitems) {
      int k = 0, left = e;
      while (left >= np - 1 - k) { left -= np - 1 - k; ++k; }
      const int k2 = k + 1 + left;
      const int p1 = ritz_shift(k, mp), q1 = ritz_shift(mp - 1 - k, mp);
      const int p2 = ritz_shift(k2, mp), q2 = ritz_shift(mp - 1 - k2, mp);
      kk[u] = k | (k2 << 16);
      to[u][0] = ritz_entry(p1, p2, mp) | (ritz_entry(p1, q2, mp) << 16);
      to[u][1] = ritz_entry(q1, p2, mp) | (ritz_entry(q1, q2, mp) << 16);
    }
  }
  // T, its FP32 off-diagonal and its diagonal, shared by the CTAs
  for (int e = rank * nth + tid; e < mp * mp; e += ncta * nth) {
    const int i = e / mp, j = e - i * mp;
    double a = 0.0;
    if (i < m && j < m) a = 0.5 * (H[i * m + j] + H[j * m + i]);
    w.T[e] = a;
    w.N[e] = i == j ? 0.f : (float)a;
    if (i == j) w.d0[i] = a;
  }
  if (rank == 0 && tid < kRitzCtl) w.ctl[tid] = 0u;
  ritz_cluster_sync();
  double *Q = w.Q, *Qn = w.Q2, *d = w.d0, *dprev = w.d1;
  float fro = 0.f, dmax = 0.f, isc = 1.f;
  int sweeps = 0, left = max_sweeps, done = 0, it = 0;
  for (;; ++it) {
    // ---- FP32: E, the rotation that diagonalises D + N (CTA 0; rows of E in the others)
    if (rank == 0) {
      float f2 = 0.f, nu = 0.f, dm = 0.f;
      for (int i = tid; i < mp; i += nth) {
        const double a = d[i];
        const float h = (float)a;
        mt.d0[i] = make_float2(h, (float)(a - (double)h));
        dm = fmaxf(dm, fabsf(h));
        f2 = fmaf(h, h, f2);
      }
      const float rmax = __uint_as_float(w.ctl[0]);
      dmax = ritz_block_max(dm, red);
      // entries of N below tau are rounding (1e-15 |T|) or first-order R left over (R^2 D)
      float tau = fmaxf((float)tol * fro, 0.5f * (float)mp * rmax * rmax * dmax);
      if (it >= 4) tau = fmaxf(tau, 1e-13f * fro);
      float emax = 0.f;
      for (int e = tid; e < mp * mp; e += nth) {
        const int i = e / mp, j = e - i * mp;
        if (i >= j) continue;
        const float n = w.N[e], an = fabsf(n);
        mt.n0[ritz_entry(i, j, mp)] = n;
        nu = fmaxf(nu, an);
        f2 = fmaf(2.f * n, n, f2);
        if (an > 0.f) {
          const float gap = fabsf((mt.d0[j].x - mt.d0[i].x) + (mt.d0[j].y - mt.d0[i].y));
          if (an > tau || an <= kTinyAngle * gap) emax = fmaxf(emax, gap > 0.f ? __fdividef(an, gap) : 1.f);
        }
      }
      if (it == 0) {
        fro = (float)sqrt(ritz_block_sum((double)f2, redd));
        isc = fro > 0.f && fro < 1e38f ? exp2f(-floorf(log2f(fro))) : 1.f;
        tau = (float)tol * fro;
      }
      nu = ritz_block_max(nu, red);
      emax = ritz_block_max(emax, red);
      // late iterations, and those after the last sweep allowed, only repair orthogonality: rotations
      // that are not tiny are left out
      const bool first_order = it > 0 && (emax <= kTinyAngle || it >= kRitzMaxIter - 2 || left == 0);
      if (tid == 0) {
        w.ctl[0] = 0u;
        w.ctl[1] = first_order ? 1u : 0u;
        w.ctl[2] = (first_order && rmax <= kTinyAngle) ? (emax <= kTinyAngle ? 1u : 2u) : 0u;
      }
      if (first_order) {
        ritz_cluster_sync();
      } else {
        const float skip = fmaxf(it == 0 ? 2e-8f * fro : 1e-7f * nu, 1e-17f * fro);
        const int cap = ritz_sweep_cap(it, left);
        for (int s = 0; s < cap; ++s) {
          float ps = 0.f, tm = 0.f;
          if (tid < nact)
            ritz_sweep<ITEMS>(mt, mp, nact, tid, nitems, to, kk, skip, tau, isc, w.log + (size_t)(s & 1) * (mp - 1) * np, &ps, &tm);
          else
            ritz_swap(mt);   // mp - 1 steps, an odd number
          __syncthreads();
          // the pivots met in a sweep bound what the next one would find (quadratic convergence)
          const float v = it == 0 ? (float)ritz_block_sum((double)ps, redd)
                                  : ritz_block_max(tm, red);
          const bool more = s + 1 < cap && v > (it == 0 ? 1e-8f * fro * fro : 1e-4f);
          ++sweeps;
          if (it > 0) --left;
          if (tid == 0) w.ctl[3 + (s & 1)] = more ? 1u : 0u;
          if (!more)
            for (int i = tid; i < mp; i += nth) d[i] = (double)mt.d0[i].x + (double)mt.d0[i].y;
          ritz_cluster_sync();
          if (!more) break;
        }
      }
    } else {
      const int nrows = (mp - rank + ncta - 1) / (ncta - 1);   // rows rank - 1, + ncta - 1, ..
      for (int e = tid; e < nrows * mp; e += nth) sm[e] = 0.f;
      for (int s = 0;; ++s) {
        ritz_cluster_sync();
        if (tid == 0) {
          s_mode = (int)w.ctl[1];
          s_more = (int)w.ctl[3 + (s & 1)];
        }
        __syncthreads();
        const bool more = s_mode == 0 && s_more != 0, sweep = s_mode == 0;
        if (sweep)
          for (int r = warp; r < nrows; r += nwarps) {
            const int i = rank - 1 + r * (ncta - 1);
            if (i < mp) ritz_apply_row(sm + r * mp, i, mp, w.log + (size_t)(s & 1) * (mp - 1) * np);
          }
        __syncthreads();
        if (!more) break;
      }
      // X = R / 2 + E (it = 0: Q = I + E)
      for (int e = tid; e < nrows * mp; e += nth) {
        const int r = e / mp, j = e - r * mp;
        const int i = rank - 1 + r * (ncta - 1);
        if (i >= mp) continue;
        if (it == 0) {
          Q[i * mp + j] = (double)sm[e] + (i == j ? 1.0 : 0.0);
          continue;
        }
        double x = (i == j ? 0.5 : 0.0) - 0.5 * w.G[i <= j ? i * mp + j : j * mp + i];
        if (s_mode != 0) {
          const float n = w.N[i * mp + j];
          const float gap = (float)(d[j] - d[i]);
          if (i != j && fabsf(n) <= kTinyAngle * fabsf(gap) && gap != 0.f) x += (double)(n / gap);
        } else {
          x += (double)sm[e];
        }
        w.X[i * mp + j] = x;
      }
    }
    ritz_cluster_sync();
    if (tid == 0) s_done = (int)w.ctl[2];
    __syncthreads();
    done = s_done;
    // ---- FP64: Q <- Q + Q X
    if (it > 0) {
      const int chunks = (mp * mp + 31) / 32;
      for (int c = rank + ncta * warp; c < chunks; c += ncta * nwarps) {
        const int e = c * 32 + lane;
        if (e < mp * mp) {
          const int i = e / mp, j = e - i * mp;
          const double* q = Q + i * mp;
          const double* x = w.X + j;
          double a = 0.0;
#pragma unroll 8
          for (int l = 0; l < mp; ++l) a = fma(q[l], x[(size_t)l * mp], a);
          Qn[e] = q[j] + a;
        }
      }
      double* t = Q; Q = Qn; Qn = t;
      ritz_cluster_sync();
    }
    if (done || it == kRitzMaxIter) break;
    // ---- FP64: G = Q^T Q (upper triangle) and W = T Q
    {
      const int ntri = np * (mp + 1), total = mp * mp + ntri;
      const int chunks = (total + 31) / 32;
      for (int c = rank + ncta * warp; c < chunks; c += ncta * nwarps) {
        const int e = c * 32 + lane;
        if (e >= total) continue;
        const double *x, *y;
        int i, j;
        if (e < mp * mp) {
          i = e / mp;
          j = e - i * mp;
          x = w.T + i;   // T is symmetric: row i as a column
        } else {
          // rows r and mp - 1 - r of the triangle make one line of mp + 1 entries
          const int f = e - mp * mp, r = f / (mp + 1), col = f - r * (mp + 1);
          i = col < mp - r ? r : mp - 1 - r;
          j = col < mp - r ? r + col : col - 1;
          x = Q + i;
        }
        y = Q + j;
        double a = 0.0;
#pragma unroll 8
        for (int l = 0; l < mp; ++l) a = fma(x[(size_t)l * mp], y[(size_t)l * mp], a);
        if (e < mp * mp) w.W[e] = a;
        else w.G[i * mp + j] = a;
      }
    }
    ritz_cluster_sync();
    // ---- FP64: S = Q^T W (upper triangle), then N, the new diagonal and max |R|
    {
      double* t = d; d = dprev; dprev = t;
      const int ntri = np * (mp + 1), chunks = (ntri + 31) / 32;
      float rm = 0.f;
      for (int c = rank + ncta * warp; c < chunks; c += ncta * nwarps) {
        const int f = c * 32 + lane;
        if (f >= ntri) continue;
        const int r = f / (mp + 1), col = f - r * (mp + 1);
        const int i = col < mp - r ? r : mp - 1 - r;
        const int j = col < mp - r ? r + col : col - 1;
        const double* x = Q + i;
        const double* y = w.W + j;
        double a = 0.0;
#pragma unroll 8
        for (int l = 0; l < mp; ++l) a = fma(x[(size_t)l * mp], y[(size_t)l * mp], a);
        const double R = (i == j ? 1.0 : 0.0) - w.G[i * mp + j];
        rm = fmaxf(rm, fabsf((float)R));
        if (i == j) {
          d[i] = fma(R, dprev[i], a);
          w.N[i * mp + i] = 0.f;
        } else {
          const float n = (float)fma(0.5 * R, dprev[i] + dprev[j], a);
          w.N[i * mp + j] = n;
          w.N[j * mp + i] = n;
        }
      }
      for (int off = 16; off > 0; off >>= 1) rm = fmaxf(rm, __shfl_xor_sync(0xffffffffu, rm, off));
      if (lane == 0 && rm > 0.f) atomicMax(&w.ctl[0], __float_as_uint(rm));
    }
    ritz_cluster_sync();
  }
  // ---- order by `which` (0 = LM: |x| descending, ties larger first; 1 = LA: descending;
  // 2 = SA: ascending; equal values in index order) by counting, then the outputs
  long long* key = reinterpret_cast<long long*>(smem_raw);
  if (tid < m) key[tid] = ritz_key(d[tid]);
  __syncthreads();
  if (tid < m) {
    const long long x = key[tid];
    int pos = 0;
    for (int j = 0; j < m; ++j) {
      const long long y = key[j];
      bool before = y > x;
      if (which == 0) {   // |x| orders like the larger of key and -key
        const long long ax = max(x, -x), ay = max(y, -y);
        before = ay > ax || (ay == ax && y > x);
      } else if (which == 2) {
        before = y < x;
      }
      pos += before || (y == x && j < tid);
    }
    order[pos] = tid;
  }
  if (rank == 0 && tid == 0) info[0] = done == 1 ? sweeps : -1;
  __syncthreads();   // order is complete; key's memory is free
  if (rank == 0)
    for (int c = tid; c < m; c += nth) theta_out[c] = d[order[c]];
  for (int e = rank * nth + tid; e < m * m; e += ncta * nth) {
    const int i = e / m, c = e - i * m;
    Y_out[e] = Q[i * mp + order[c]];
  }
  // rho of columns rank, rank + ncta, ..: one partial square per (column, row of the last block)
  double* sq = reinterpret_cast<double*>(smem_raw);
  const int ncols = m > rank ? (m - rank + ncta - 1) / ncta : 0;
  for (int e = tid; e < ncols * b; e += nth) {
    const int c = rank + (e / b) * ncta, p = e % b;
    const double* h = H + (size_t)(m + p) * m;
    const double* y = Q + order[c];
    double s = 0.0;
#pragma unroll 8
    for (int i = 0; i < m; ++i) s = fma(h[i], y[(size_t)i * mp], s);
    sq[e] = s * s;
  }
  __syncthreads();
  for (int k = tid; k < ncols; k += nth) {
    double r2 = 0.0;
    for (int p = 0; p < b; ++p) r2 += sq[k * b + p];
    rho_out[rank + k * ncta] = sqrt(r2);
  }
}

// ------------------------------------------------------------ large subspaces (m > kRitzOneMax)
// For m up to kRitzMax (512) the m x m matrices no longer fit one SM's shared memory, and FP64
// Jacobi work on one SM (2 DFMA per clock) would take tens of milliseconds per sweep.  So:
//   1. one CTA runs the FP32 Jacobi sweeps (A32, Q32 in global memory, L2-resident) to a
//      relative off-diagonal norm of about 1e-6;
//   2. Q32 is made orthogonal in FP64 by two Newton-Schulz steps Q <- Q (3 I - Q^T Q) / 2
//      (Higham, "Functions of Matrices", 8.3: quadratic convergence to the orthogonal polar
//      factor from ||Q^T Q - I|| ~ 1e-7), and A <- Q^T T Q, all as FP64 matrix products on the
//      whole GPU;
//   3. FP64 parallel Jacobi sweeps on the nearly diagonal A finish it (two or three sweeps), on
//      a cooperative grid: a step's rotations are computed by every CTA from the same entries,
//      then the CTAs share the step's 2 x 2 block updates, with a grid barrier after each half;
//   4. one CTA orders the pairs and writes theta, Y and the residual estimates.
// Workspace layout (ld = mp + 1): A32, Q32 (floats, one mp x ld double-array each pair), A64,
// Q64, W64, S64, then the barrier words and the per-CTA partial sums.
constexpr int kCoopCtas = 64;

struct BigWork {
  float *A32, *Q32;
  double *A, *Q, *W, *S;
  unsigned* bar;      // [0] arrivals, [1] generation, [2] error flag
  double* part;       // kCoopCtas partial sums, then fro2 at [kCoopCtas]
};

__host__ __device__ inline size_t big_mat_doubles(int m) {
  const int mp = m + (m & 1);
  return (size_t)mp * (mp + 1);
}

__host__ __device__ inline BigWork big_work(double* w, int m) {
  const size_t mat = big_mat_doubles(m);
  BigWork b;
  b.A32 = reinterpret_cast<float*>(w);
  b.Q32 = reinterpret_cast<float*>(w) + mat;
  b.A = w + mat;
  b.Q = b.A + mat;
  b.W = b.Q + mat;
  b.S = b.W + mat;
  b.bar = reinterpret_cast<unsigned*>(b.S + mat);
  b.part = b.S + mat + 4;
  return b;
}

size_t ritz_work_doubles(int m) {
  const size_t grid = 5 * big_mat_doubles(m) + 4 + kCoopCtas + 8;
  return m <= kRitzOneMax ? std::max(ritz_cluster_doubles(m), grid) : grid;
}

// 1. FP32 sweeps (one CTA) and the FP64 copies of T and Q32.
__global__ void __launch_bounds__(1024) ritz_big_fp32_kernel(const double* __restrict__ H, int m, double* work) {
  const int mp = m + (m & 1), ld = mp + 1, np = mp / 2;
  BigWork w = big_work(work, m);
  __shared__ float cs[kRitzMax / 2], sn[kRitzMax / 2];
  __shared__ int pp[kRitzMax / 2], pq[kRitzMax / 2];
  __shared__ double red[32];
  __shared__ bool conv;
  const int tid = threadIdx.x, nth = blockDim.x;
  double v = 0.0;
  for (int e = tid; e < mp * mp; e += nth) {
    const int i = e / mp, j = e % mp;
    const double a = (i < m && j < m) ? 0.5 * (H[i * m + j] + H[j * m + i]) : 0.0;
    w.A32[i * ld + j] = (float)a;
    w.Q32[i * ld + j] = (i == j) ? 1.f : 0.f;
    v += a * a;
  }
  const double fro2 = ritz_block_sum(v, red);
  __syncthreads();
  jacobi_sweeps<float>(w.A32, w.Q32, ld, m, mp, 1e-12 * fro2, 20, cs, sn, pp, pq, red, &conv);
  for (int e = tid; e < mp * mp; e += nth) {
    const int i = e / mp, j = e % mp;
    w.Q[i * ld + j] = (double)w.Q32[i * ld + j];
    w.A[i * ld + j] = (i < m && j < m) ? 0.5 * (H[i * m + j] + H[j * m + i]) : 0.0;
  }
  if (tid == 0) w.part[kCoopCtas] = fro2;
  (void)np;
}

// 2. C = alpha op(A) op(B) + beta C for mp x mp FP64 matrices (row stride ld); op = transpose
// when ta / tb.  32 x 32 output tile per CTA, 256 threads with 4 outputs each.
__global__ void __launch_bounds__(256) ritz_dgemm_kernel(const double* __restrict__ A, const double* __restrict__ B,
                                                         double* __restrict__ C, int mp, int ld, int ta, int tb,
                                                         double alpha, double beta) {
  __shared__ double sa[32][33], sb[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int k0 = 0; k0 < mp; k0 += 32) {
    for (int r = ty; r < 32; r += 8) {
      const int i = i0 + r, k = k0 + tx;   // sa[r][tx] = op(A)[i][k]
      sa[r][tx] = (i < mp && k < mp) ? (ta ? A[k * ld + i] : A[i * ld + k]) : 0.0;
      const int kk = k0 + r, j = j0 + tx; // sb[r][tx] = op(B)[kk][j]
      sb[r][tx] = (kk < mp && j < mp) ? (tb ? B[j * ld + kk] : B[kk * ld + j]) : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const double bv = sb[k][tx];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = fma(sa[ty + 8 * u][k], bv, acc[u]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = i0 + ty + 8 * u, j = j0 + tx;
    if (i < mp && j < mp) C[i * ld + j] = alpha * acc[u] + (beta != 0.0 ? beta * C[i * ld + j] : 0.0);
  }
}

// Q <- (3 Q - W) / 2 with W = Q (Q^T Q): one Newton-Schulz step.
__global__ void ritz_ns_kernel(double* __restrict__ Q, const double* __restrict__ W, int mp, int ld) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= mp * mp) return;
  const int i = e / mp, j = e % mp;
  Q[i * ld + j] = 1.5 * Q[i * ld + j] - 0.5 * W[i * ld + j];
}

// Grid-wide barrier for a cooperative launch (all CTAs resident): arrival counter and
// generation word in global memory.  The wait is bounded; on a timeout the error flag is set
// and false returned (the caller then leaves its loops).
__device__ bool coop_barrier(unsigned* bar, unsigned& gen) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    __threadfence();
    const unsigned g = gen;
    if (atomicAdd(&bar[0], 1u) == gridDim.x - 1) {
      atomicExch(&bar[0], 0u);
      __threadfence();
      atomicAdd(&bar[1], 1u);
    } else {
      unsigned spins = 0;
      while (atomicAdd(&bar[1], 0u) == g) {
        if (++spins > (1u << 26) || atomicAdd(&bar[2], 0u) != 0u) {
          atomicExch(&bar[2], 1u);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    gen = g + 1;
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// 3. FP64 parallel Jacobi sweeps on A (nearly diagonal), Q <- Q J, across the grid.
__global__ void __launch_bounds__(512) ritz_big_jacobi64_kernel(double* work, int m, double tol, int max_sweeps,
                                                                int* info) {
  const int mp = m + (m & 1), ld = mp + 1, np = mp / 2;
  BigWork w = big_work(work, m);
  __shared__ double cs[kRitzMax / 2], sn[kRitzMax / 2];
  __shared__ int pp[kRitzMax / 2], pq[kRitzMax / 2];
  __shared__ double red[32];
  const int tid = threadIdx.x, nth = blockDim.x;
  const int gt = blockIdx.x * nth + tid, gn = gridDim.x * nth;
  unsigned gen = 0;
  const double fro2 = w.part[kCoopCtas];
  const double thresh = tol * tol * fro2;
  int sweeps = 0;
  bool conv = false;
  while (true) {
    double v = 0.0;
    for (int e = gt; e < mp * mp; e += gn) {
      const int i = e / mp, j = e % mp;
      if (i != j) v += w.A[i * ld + j] * w.A[i * ld + j];
    }
    v = ritz_block_sum(v, red);
    if (tid == 0) w.part[blockIdx.x] = v;
    if (!coop_barrier(w.bar, gen)) return;
    double off2 = 0.0;
    for (int c = 0; c < (int)gridDim.x; ++c) off2 += w.part[c];   // same order in every CTA
    if (off2 <= thresh || sweeps >= max_sweeps) {
      conv = off2 <= thresh;
      break;
    }
    ++sweeps;
    for (int step = 0; step < mp - 1; ++step) {
      // every CTA forms the step's rotations from the same (stable) entries ...
      for (int k = tid; k < np; k += nth) {
        auto pos = [&](int i) { return i == 0 ? 0 : ((i - 1 + step) % (mp - 1)) + 1; };
        int p = pos(k), q = pos(mp - 1 - k);
        if (p > q) { const int t = p; p = q; q = t; }
        double c = 1.0, sv = 0.0;
        if (q < m) {
          const float t = jacobi_tan(w.A[p * ld + p], w.A[p * ld + q], w.A[q * ld + q]);
          if (t != 0.f) jacobi_cs(t, c, sv);
        }
        pp[k] = p;
        pq[k] = q;
        cs[k] = c;
        sn[k] = sv;
      }
      if (!coop_barrier(w.bar, gen)) return;   // all rotations read before any entry changes
      // ... then the CTAs share the independent 2 x 2 block updates and Q's column pairs
      const int nsq = np * np;
      for (int e = gt; e < nsq + mp * np; e += gn) {
        if (e < nsq) {
          const int k = e / np, k2 = e - k * np;
          if (k > k2) continue;
          const double s1 = sn[k], s2 = sn[k2];
          if (s1 == 0.0 && s2 == 0.0) continue;
          const double c1 = cs[k], c2 = cs[k2];
          const int p1 = pp[k], q1 = pq[k];
          double* A = w.A;
          if (k == k2) {
            const double app = A[p1 * ld + p1], aqq = A[q1 * ld + q1], apq = A[p1 * ld + q1];
            const double cc = c1 * c1, ss = s1 * s1, cs2 = c1 * s1;
            A[p1 * ld + p1] = cc * app - 2.0 * cs2 * apq + ss * aqq;
            A[q1 * ld + q1] = ss * app + 2.0 * cs2 * apq + cc * aqq;
            const double npq = cs2 * (app - aqq) + (cc - ss) * apq;
            A[p1 * ld + q1] = npq;
            A[q1 * ld + p1] = npq;
          } else {
            const int p2 = pp[k2], q2 = pq[k2];
            const double x00 = A[p1 * ld + p2], x01 = A[p1 * ld + q2];
            const double x10 = A[q1 * ld + p2], x11 = A[q1 * ld + q2];
            const double y00 = c1 * x00 - s1 * x10, y01 = c1 * x01 - s1 * x11;
            const double y10 = s1 * x00 + c1 * x10, y11 = s1 * x01 + c1 * x11;
            const double z00 = c2 * y00 - s2 * y01, z01 = s2 * y00 + c2 * y01;
            const double z10 = c2 * y10 - s2 * y11, z11 = s2 * y10 + c2 * y11;
            A[p1 * ld + p2] = z00;
            A[p1 * ld + q2] = z01;
            A[q1 * ld + p2] = z10;
            A[q1 * ld + q2] = z11;
            A[p2 * ld + p1] = z00;
            A[q2 * ld + p1] = z01;
            A[p2 * ld + q1] = z10;
            A[q2 * ld + q1] = z11;
          }
        } else {
          const int e2 = e - nsq;
          const int i = e2 / np, k = e2 - i * np;
          const double sk = sn[k];
          if (sk == 0.0) continue;
          const double ck = cs[k];
          const int p = pp[k], q = pq[k];
          const double vp = w.Q[i * ld + p], vq = w.Q[i * ld + q];
          w.Q[i * ld + p] = ck * vp - sk * vq;
          w.Q[i * ld + q] = sk * vp + ck * vq;
        }
      }
      if (!coop_barrier(w.bar, gen)) return;
    }
  }
  if (blockIdx.x == 0 && tid == 0) info[0] = conv ? sweeps : -1;
}

// 4. Ordering and outputs (one CTA).
__global__ void ritz_big_out_kernel(const double* __restrict__ H, int m, int b, int which, double* work,
                                    double* __restrict__ theta_out, double* __restrict__ Y_out,
                                    double* __restrict__ rho_out, int* __restrict__ info) {
  const int mp = m + (m & 1), ld = mp + 1;
  BigWork w = big_work(work, m);
  __shared__ int order[kRitzMax];
  const int tid = threadIdx.x, nth = blockDim.x;
  if (tid == 0) {
    for (int i = 0; i < m; ++i) order[i] = i;
    for (int i = 1; i < m; ++i) {
      const int x = order[i];
      const double tx = w.A[x * ld + x];
      int j = i - 1;
      while (j >= 0) {
        const double ty = w.A[order[j] * ld + order[j]];
        bool before;
        if (which == 0) before = fabs(tx) > fabs(ty) || (fabs(tx) == fabs(ty) && tx > ty);
        else if (which == 1) before = tx > ty;
        else before = tx < ty;
        if (!before) break;
        order[j + 1] = order[j];
        --j;
      }
      order[j + 1] = x;
    }
    if (w.bar[2] != 0u) info[0] = -2;   // a grid barrier timed out
  }
  __syncthreads();
  for (int c = tid; c < m; c += nth) theta_out[c] = w.A[order[c] * ld + order[c]];
  for (int e = tid; e < m * m; e += nth) {
    const int i = e / m, c = e % m;
    Y_out[e] = w.Q[i * ld + order[c]];
  }
  for (int c = tid; c < m; c += nth) {
    double r2 = 0.0;
    for (int p = 0; p < b; ++p) {
      double s = 0.0;
      for (int i = 0; i < m; ++i) s += H[(m + p) * m + i] * w.Q[i * ld + order[c]];
      r2 += s * s;
    }
    rho_out[c] = sqrt(r2);
  }
}

static int launch_ritz_big(const double* H, int m, int b, int which, int max_sweeps, double tol,
                           double* theta, double* Y, double* rho, int* info, double* work,
                           cudaStream_t s) {
  const int mp = m + (m & 1), ld = mp + 1;
  BigWork w = big_work(work, m);
  FE_CUDA(cudaMemsetAsync(w.bar, 0, 4 * sizeof(unsigned), s));
  ritz_big_fp32_kernel<<<1, 1024, 0, s>>>(H, m, work);
  count_launch();
  FE_CUDA(cudaGetLastError());
  const dim3 gg((mp + 31) / 32, (mp + 31) / 32);
  auto gemm = [&](const double* A, const double* B, double* C, int ta, int tb) -> int {
    ritz_dgemm_kernel<<<gg, 256, 0, s>>>(A, B, C, mp, ld, ta, tb, 1.0, 0.0);
    count_launch();
    FE_CUDA(cudaGetLastError());
    return FE_OK;
  };
  for (int it = 0; it < 2; ++it) {   // Q <- Q (3 I - Q^T Q) / 2
    FE_TRY(gemm(w.Q, w.Q, w.S, 1, 0));
    FE_TRY(gemm(w.Q, w.S, w.W, 0, 0));
    ritz_ns_kernel<<<(mp * mp + 255) / 256, 256, 0, s>>>(w.Q, w.W, mp, ld);
    count_launch();
    FE_CUDA(cudaGetLastError());
  }
  FE_TRY(gemm(w.A, w.Q, w.W, 0, 0));   // W = T Q
  FE_TRY(gemm(w.Q, w.W, w.A, 1, 0));   // A = Q^T T Q
  // cooperative launch: every CTA resident (the grid barrier relies on it)
  static KernelSetup ks;
  int per_sm = 0;
  FE_TRY(kernel_occupancy(ks, reinterpret_cast<const void*>(ritz_big_jacobi64_kernel), 512, 0, 0, &per_sm));
  const int grid = std::min(kCoopCtas, per_sm * num_sms());
  FE_ARG(grid >= 1, "ritz: no resident CTA for the cooperative Jacobi kernel");
  double* wk = work;
  int mm = m, ms = max_sweeps;
  double tl = tol;
  void* args[] = {&wk, &mm, &tl, &ms, &info};
  FE_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(ritz_big_jacobi64_kernel), dim3(grid),
                                      dim3(512), args, 0, s));
  count_launch();
  ritz_big_out_kernel<<<1, 512, 0, s>>>(H, m, b, which, work, theta, Y, rho, info);
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// info[0]: the sweeps run, -1 where the projected matrix is not diagonal to tol, -2 after a barrier that timed
// out.  grid: the sweeps on the grid whatever m is (m <= kRitzOneMax: the second attempt after a -1).
int launch_ritz(const double* H, int m, int b, int which, int max_sweeps, double tol,
                double* theta, double* Y, double* rho, int* info, double* work, bool grid, cudaStream_t s) {
  FE_ARG(m >= 1 && m <= kRitzMax, "ritz: subspace m = %d not in [1, %d]", m, kRitzMax);
  FE_ARG(work != nullptr, "ritz: m = %d needs a global workspace", m);
  if (grid || m > kRitzOneMax)
    return launch_ritz_big(H, m, b, which, max_sweeps, tol, theta, Y, rho, info, work, s);
  static KernelSetup ks[3];
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto shape = [&](const RitzShape& sh) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sh.ncta;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(sh.ncta);
    cfg.blockDim = dim3(sh.threads);
    cfg.dynamicSmemBytes = ritz_cluster_smem(m, b, sh.ncta);
  };
  const RitzShape sh = ritz_shape(m, true);
  const int variant = sh.items == 1 ? 0 : (sh.items == 4 ? 1 : 2);
  auto kern = variant == 0 ? ritz_cluster_kernel<1> : (variant == 1 ? ritz_cluster_kernel<4> : ritz_cluster_kernel<7>);
  const void* fn = reinterpret_cast<const void*>(kern);
  FE_TRY(kernel_configure(ks[variant], fn, 128 * 1024));
  shape(sh);
  if (sh.ncta > kRitzCluster) {
    // asked once per device and kernel: whether the device takes the cluster at all
    static std::mutex mu;
    static signed char wide[3][kMaxDevices];   // 0: not asked, 1: yes, -1: no
    const int dev = cur_device();
    if (dev < 0) return dev;
    std::lock_guard<std::mutex> lock(mu);
    if (wide[variant][dev] == 0) {
      int clusters = 0;
      const bool ok = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                      cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters > 0;
      if (!ok) cudaGetLastError();   // not an error: the smaller cluster does
      wide[variant][dev] = ok ? 1 : -1;
    }
    if (wide[variant][dev] < 0) shape(ritz_shape(m, false));
  }
  FE_CUDA(cudaLaunchKernelEx(&cfg, kern, H, m, b, which, max_sweeps, tol, theta, Y, rho, info, work));
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// Krylov-Schur restart of H ((m+b) x m, row-major): keep k Ritz pairs.
//   B^T = H[m:m+b, 0:m] Y[:, 0:k];  H <- 0;  H[c][c] = theta_c (c < k);  H[k:k+b, 0:k] = B^T
__global__ void restart_h_kernel(double* __restrict__ H, int m, int b, int k,
                                 const double* __restrict__ theta, const double* __restrict__ Y) {
  extern __shared__ double bt[];  // b x k
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int e = tid; e < b * k; e += nth) {
    const int p = e / k, c = e % k;
    double s = 0.0;
    for (int i = 0; i < m; ++i) s += H[(m + p) * m + i] * Y[i * m + c];
    bt[e] = s;
  }
  __syncthreads();
  for (int e = tid; e < (m + b) * m; e += nth) H[e] = 0.0;
  __syncthreads();
  for (int c = tid; c < k; c += nth) H[c * m + c] = theta[c];
  for (int e = tid; e < b * k; e += nth) H[(k + e / k) * m + e % k] = bt[e];
}

int launch_restart_h(double* H, int m, int b, int k, const double* theta, const double* Y,
                     cudaStream_t s) {
  restart_h_kernel<<<1, 256, sizeof(double) * b * k, s>>>(H, m, b, k, theta, Y);
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// ------------------------------------------------------------ sign of eigenvectors
// For each column c of the column-major n x ncols matrix X: find the entry of largest
// magnitude (first index on ties) and flip the column if it is negative.  The partials carry
// the signed value of each block's best entry, so the flip decision never re-reads X (which
// other blocks of the flipping kernel may already have changed).
__global__ void colmax_partial_kernel(const double* __restrict__ X, int64_t n, int ncols,
                                      double* __restrict__ pval, int64_t* __restrict__ pidx) {
  const int c = blockIdx.y;
  double best = -1.0, bval = 0.0;
  int64_t bi = INT64_MAX;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    const double x = X[(int64_t)c * n + r];
    const double a = fabs(x);
    if (a > best || (a == best && r < bi)) { best = a; bi = r; bval = x; }
  }
  __shared__ double sv[256], sx[256];
  __shared__ int64_t si[256];
  sv[threadIdx.x] = best;
  sx[threadIdx.x] = bval;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      const double a = sv[threadIdx.x + w];
      const int64_t i = si[threadIdx.x + w];
      if (a > sv[threadIdx.x] || (a == sv[threadIdx.x] && i < si[threadIdx.x])) {
        sv[threadIdx.x] = a;
        si[threadIdx.x] = i;
        sx[threadIdx.x] = sx[threadIdx.x + w];
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    pval[(int64_t)c * gridDim.x + blockIdx.x] = sx[0];   // signed value of the best entry
    pidx[(int64_t)c * gridDim.x + blockIdx.x] = si[0];
  }
}

__global__ void colsign_kernel(double* __restrict__ X, int64_t n, int ncols, int nparts,
                               const double* __restrict__ pval, const int64_t* __restrict__ pidx) {
  const int c = blockIdx.y;
  __shared__ double sgn;
  if (threadIdx.x == 0) {
    double best = -1.0, bval = 0.0;
    int64_t bi = INT64_MAX;
    for (int p = 0; p < nparts; ++p) {
      const double x = pval[(int64_t)c * nparts + p];
      const double a = fabs(x);
      const int64_t i = pidx[(int64_t)c * nparts + p];
      if (a > best || (a == best && i < bi)) { best = a; bi = i; bval = x; }
    }
    sgn = bval < 0.0 ? -1.0 : 1.0;
  }
  __syncthreads();
  if (sgn > 0.0) return;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
    X[(int64_t)c * n + r] = -X[(int64_t)c * n + r];
}

int normalize_signs(double* X, int64_t n, int ncols, cudaStream_t s) {
  const int parts = (int)std::min<int64_t>(ceil_div(n, 256), 64);
  double* pval = small_scratch(12, (size_t)parts * ncols);
  double* pidx = small_scratch(13, (size_t)parts * ncols);
  if (!pval || !pidx) return FE_ERR_OOM;
  dim3 grid(parts, ncols);
  colmax_partial_kernel<<<grid, 256, 0, s>>>(X, n, ncols, pval, reinterpret_cast<int64_t*>(pidx));
  count_launch();
  FE_CUDA(cudaGetLastError());
  colsign_kernel<<<grid, 256, 0, s>>>(X, n, ncols, parts, pval, reinterpret_cast<const int64_t*>(pidx));
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

}  // namespace fe
