// Launch shape, slot order and shared-memory layout of the one-cluster Rayleigh-Ritz kernel: plain
// index arithmetic for host and device, so that it can be checked without a GPU.
#pragma once
#include <stddef.h>

#include <algorithm>

namespace fe {

// Subspaces up to kRitzOneMax are diagonalised by one cluster of kRitzCluster or kRitzClusterMax CTAs.
constexpr int kRitzOneMax = 160;
constexpr int kRitzCluster = 8, kRitzClusterMax = 16;

// FP64 products take m^3 / ncta / 2 clocks each: 16 CTAs where that outweighs the wider cluster's
// barriers (m = 128: 0.43 ms of products on 8, 0.22 ms on 16); threads enough for one, four or
// seven 2 x 2 blocks each (items; 128 registers a thread: more threads with fewer spill).
struct RitzShape {
  int ncta, items, threads;
};
// wide: clusters of kRitzClusterMax can be launched (more than 8 CTAs is a non-portable size).
inline RitzShape ritz_shape(int m, bool wide) {
  return {m > 64 && wide ? kRitzClusterMax : kRitzCluster, m <= 64 ? 1 : (m <= 128 ? 4 : 7), m <= 46 ? 256 : 512};
}

// Most sweeps of iteration `it`: kRitzFirstSweeps FP32 ones of the projected matrix itself, then, over all later
// iterations, as many as the caller's max_sweeps (`left` of them are left), at most six at a time.
constexpr int kRitzFirstSweeps = 15;
__host__ __device__ __forceinline__ int ritz_sweep_cap(int it, int left) {
  return it == 0 ? kRitzFirstSweeps : (left < 6 ? left : 6);
}

// 2 x 2 blocks (pairs k < k2 of np), and the threads that take part in a sweep.
__host__ __device__ __forceinline__ int ritz_items(int np) { return np * (np - 1) / 2; }
__host__ __device__ __forceinline__ int ritz_active(int np, int threads) {
  const int need = ritz_items(np) > np ? ritz_items(np) : np, up = (need + 31) & ~31;
  return up < threads ? up : threads;
}
// Floats of one copy of the matrix: four planes of the blocks' entries, then the pivots.
__host__ __device__ __forceinline__ int ritz_copy(int np) { return 4 * ritz_items(np) + np; }
// Where a thread reads its block e in a plane: threads past the last block read entry 0 (for no
// blocks at all, m <= 2, that is the pivot) and drop it.
__host__ __device__ __forceinline__ int ritz_read(int e, int nitems) { return e < nitems ? e : 0; }

// The circle method in slots: the index in slot i of a step is in slot ritz_shift(i) of the next
// one (slot 0 stays), and pair k of a step is slots k and mp - 1 - k.  Data that moves with its
// slot is at addresses that do not depend on the step, and after mp - 1 steps slot i holds
// index i again.
__host__ __device__ __forceinline__ int ritz_shift(int i, int mp) { return i == 0 ? 0 : (i == 1 ? mp - 1 : i - 1); }
// Offset of the entry of slots a != b: the 2 x 2 block of pairs k < k2 is entry tri(k, k2) of four
// planes (row of pair k from slot k or mp - 1 - k, column likewise); the pivots follow.
__host__ __device__ __forceinline__ int ritz_entry(int a, int b, int mp) {
  const int np = mp / 2, nt = ritz_items(np);
  int ka = a < np ? a : mp - 1 - a, ra = a < np ? 0 : 1;
  int kb = b < np ? b : mp - 1 - b, rb = b < np ? 0 : 1;
  if (ka == kb) return 4 * nt + ka;
  if (ka > kb) {
    int t = ka; ka = kb; kb = t;
    t = ra; ra = rb; rb = t;
  }
  return (ra * 2 + rb) * nt + ka * np - ka * (ka + 1) / 2 + kb - ka - 1;
}

// Bytes of dynamic shared memory: CTA 0's rotations (np float2), two diagonals (mp float2 each) and two
// copies of the matrix; the other CTAs' rows of E; the residual sums.
inline size_t ritz_cluster_smem(int m, int b, int ncta) {
  const size_t mp = m + (m & 1), np = mp / 2;
  const size_t head = (2 * np + 4 * mp + 2 * (size_t)ritz_copy((int)np)) * sizeof(float);
  const size_t rows = ((mp + ncta - 3) / (ncta - 1) + 1) * mp * sizeof(float);
  const size_t rho = std::max<size_t>(m, (size_t)((m + ncta - 1) / ncta) * b) * sizeof(double);
  return std::max(head, std::max(rows, rho));
}

}  // namespace fe
