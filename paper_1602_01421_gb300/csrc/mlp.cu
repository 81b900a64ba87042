// Learned start block (not in the paper; an extension of its random start, Table 1 MvRandom):
// features from SpMM powers (Section 3.3's operation), a 3-layer MLP that maps them to an
// n x b block, its training kernels (loss, gradient, Adam), and the start block fe_eigs uses.
//
// Features (8 per vertex; rms(x) = sqrt(mean(x^2)), 1 when 0):
//   d = A 1; f0 = log(1+d), f1 = d/rms(d), f2 = A d/rms, f3 = A^2 d/rms;
//   R = N(0,1) n x 4 (counter RNG, stream 6); q_p = mean_c (A^p R)_{:,c}^2 (p = 2, 3, 4);
//   f4 = q2/rms(q2), f5 = q3/rms(q3), f6 = q4/rms(q4), f7 = log(1 + q2/mean(q2)).
// Network: h1 = relu(F W1 + b1), h2 = relu(h1 W2 + b2), Z = h2 W3 + b3; parameters packed
// [W1 (8 x H), b1, W2 (H x H), b2, W3 (H x b), b3], FP32.
// Loss against unit reference columns U: L = sum_j (1 - (z_j . u_j)^2 / |z_j|^2).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "fe_internal.cuh"
#include "vec.cuh"

namespace fe {

constexpr int kNFeat = 8;
constexpr uint64_t kStreamProbe = 6;

int64_t mlp_param_count(int H, int b) {
  return (int64_t)kNFeat * H + H + (int64_t)H * H + H + (int64_t)H * b + b;
}

// ---------------------------------------------------------------- features
__global__ void fill_kernel(double* x, int64_t n, double v) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) x[i] = v;
}

// q[i] = mean over the 4 columns of P[i][c]^2
__global__ void rowmeansq_kernel(const double* __restrict__ P, int64_t n, double* __restrict__ q) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double a = P[4 * i], b = P[4 * i + 1], c = P[4 * i + 2], d = P[4 * i + 3];
    q[i] = 0.25 * (a * a + b * b + c * c + d * d);
  }
}

// sums[k] = sum_i x_k[i]^2 for the 6 vectors, sums[6] = sum_i q2[i]; per-CTA partials.
struct FeatVecs {
  const double* v[6];
  const double* q2;
};
__global__ void feat_sums_kernel(const FeatVecs fv, int64_t n, double* __restrict__ partial) {
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const double x = fv.v[k][i];
      acc[k] += x * x;
    }
    acc[6] += fv.q2[i];
  }
  __shared__ double red[7][256];
#pragma unroll
  for (int k = 0; k < 7; ++k) red[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int k = 0; k < 7; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 7) partial[blockIdx.x * 7 + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void feat_scales_kernel(const double* __restrict__ partial, int nctas, int64_t n,
                                   double* __restrict__ scale) {
  const int k = threadIdx.x;
  if (k >= 7) return;
  double s = 0.0;
  for (int c = 0; c < nctas; ++c) s += partial[c * 7 + k];
  const double m = s / (double)n;
  if (k < 6) {
    const double r = sqrt(m);
    scale[k] = r > 0.0 ? r : 1.0;   // rms
  } else {
    scale[k] = m > 0.0 ? m : 1.0;   // mean(q2)
  }
}

__global__ void feat_assemble_kernel(const FeatVecs fv, int64_t n, const double* __restrict__ scale,
                                     float* __restrict__ F) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double d = fv.v[0][i];
    float* f = F + i * kNFeat;
    f[0] = (float)log1p(d);
    f[1] = (float)(d / scale[0]);
    f[2] = (float)(fv.v[1][i] / scale[1]);
    f[3] = (float)(fv.v[2][i] / scale[2]);
    f[4] = (float)(fv.v[3][i] / scale[3]);
    f[5] = (float)(fv.v[4][i] / scale[4]);
    f[6] = (float)(fv.v[5][i] / scale[5]);
    f[7] = (float)log1p(fv.q2[i] / scale[6]);
  }
}

static int spmm_any(fe_csr h, const void* X, void* Y, int b, cudaStream_t s) {
  if (h->semi_external) return semiext_spmm(h, X, Y, b, FE_F64, s);
  return spmm_resident(h, X, Y, b, FE_F64, s);
}

int vertex_features(fe_csr h, uint64_t seed, float* F, cudaStream_t s) {
  const int64_t n = h->n;
  DevBuf buf;
  // d, ad, a2d, q2, q3, q4 (n each) + R/P ping-pong (2 x 4n)
  FE_TRY(buf.alloc(sizeof(double) * (size_t)n * 14));
  double* d = buf.as<double>();
  double* ad = d + n;
  double* a2d = ad + n;
  double* q2 = a2d + n;
  double* q3 = q2 + n;
  double* q4 = q3 + n;
  double* P0 = q4 + n;
  double* P1 = P0 + 4 * n;
  double* ones = P1;  // scratch before the probes use it
  const int ctas = (int)std::min<int64_t>(ceil_div(n, 256), 4 * num_sms());
  fill_kernel<<<ctas, 256, 0, s>>>(ones, n, 1.0);
  count_launch();
  FE_CUDA(cudaGetLastError());
  FE_TRY(spmm_any(h, ones, d, 1, s));
  FE_TRY(spmm_any(h, d, ad, 1, s));
  FE_TRY(spmm_any(h, ad, a2d, 1, s));
  FE_TRY(random_normal(P0, n, 4, 4, FE_F64, seed, kStreamProbe, 0, s));
  FE_TRY(spmm_any(h, P0, P1, 4, s));   // A R
  FE_TRY(spmm_any(h, P1, P0, 4, s));   // A^2 R
  rowmeansq_kernel<<<ctas, 256, 0, s>>>(P0, n, q2);
  count_launch();
  FE_TRY(spmm_any(h, P0, P1, 4, s));   // A^3 R
  rowmeansq_kernel<<<ctas, 256, 0, s>>>(P1, n, q3);
  count_launch();
  FE_TRY(spmm_any(h, P1, P0, 4, s));   // A^4 R
  rowmeansq_kernel<<<ctas, 256, 0, s>>>(P0, n, q4);
  count_launch();
  FE_CUDA(cudaGetLastError());
  FeatVecs fv;
  fv.v[0] = d;
  fv.v[1] = ad;
  fv.v[2] = a2d;
  fv.v[3] = q2;
  fv.v[4] = q3;
  fv.v[5] = q4;
  fv.q2 = q2;
  const int rctas = (int)std::min<int64_t>(ceil_div(n, 256), 2 * num_sms());
  double* part = small_scratch(14, (size_t)rctas * 7 + 8);
  if (!part) return FE_ERR_OOM;
  double* scale = part + (size_t)rctas * 7;
  feat_sums_kernel<<<rctas, 256, 0, s>>>(fv, n, part);
  count_launch();
  feat_scales_kernel<<<1, 32, 0, s>>>(part, rctas, n, scale);
  count_launch();
  feat_assemble_kernel<<<ctas, 256, 0, s>>>(fv, n, scale, F);
  count_launch();
  FE_CUDA(cudaGetLastError());
  FE_CUDA(cudaStreamSynchronize(s));  // buf is freed on return
  return FE_OK;
}

// ---------------------------------------------------------------- forward
template <int H, int B>
struct MlpParams {
  static constexpr int W1 = 0, B1 = kNFeat * H, W2 = B1 + H, B2 = W2 + H * H, W3 = B2 + H,
                       B3 = W3 + H * B, COUNT = B3 + B;
};

// The network runs on tiles of kTile rows per CTA of kThr threads, as products of shared-memory
// operands with register accumulators.  Activations lie transposed (unit, row), kLd floats per
// unit: a thread's output tile is 8 rows (two runs of four) x H / 16 units, read with two 16-byte
// loads of activations and one of weights per inner index for 8 H / 16 FMAs.  Shared-memory bandwidth
// bounds the products all the same (H = 64, the gradient kernel: its data pipe 79% busy, the FMA pipes
// 46%, issue 59%).
constexpr int kTile = 128, kThr = 256, kLd = kTile + 4;   // kLd: units 4 banks apart

struct TileMap {   // the thread's rows r0 .. r0 + 3, r0 + 64 .. r0 + 67 and units c0 ..
  int r0, cg;
  __device__ TileMap() {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    r0 = 4 * (lane % 8 + 8 * (warp & 1));
    cg = lane / 8 + 4 * (warp >> 1);
  }
};

template <int CT>
__device__ __forceinline__ void ld_units(const float* p, float* w) {
  if constexpr (CT == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
  } else {
    const float2 v = *reinterpret_cast<const float2*>(p);
    w[0] = v.x; w[1] = v.y;
  }
}

// acc[i][c] += sum over k < K of act[k][row i] w[k][unit c] (w: K x H)
template <int H, int K>
__device__ __forceinline__ void tile_gemm(const float* act, const float* w, const TileMap& tm,
                                          float (&acc)[8][H / 16]) {
  constexpr int CT = H / 16;
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const float4 a0 = *reinterpret_cast<const float4*>(act + k * kLd + tm.r0);
    const float4 a1 = *reinterpret_cast<const float4*>(act + k * kLd + tm.r0 + 64);
    float wv[CT];
    ld_units<CT>(w + k * H + tm.cg * CT, wv);
    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < CT; ++c) acc[i][c] = fmaf(av[i], wv[c], acc[i][c]);
  }
}

template <int H>
__device__ __forceinline__ void tile_store(float* act, const TileMap& tm, const float (&v)[8][H / 16]) {
  constexpr int CT = H / 16;
#pragma unroll
  for (int c = 0; c < CT; ++c) {
    float* d = act + (tm.cg * CT + c) * kLd + tm.r0;
    *reinterpret_cast<float4*>(d) = make_float4(v[0][c], v[1][c], v[2][c], v[3][c]);
    *reinterpret_cast<float4*>(d + 64) = make_float4(v[4][c], v[5][c], v[6][c], v[7][c]);
  }
}

// relu in place; bit i * CT + c of the result: unit positive
template <int CT>
__device__ __forceinline__ unsigned tile_relu(float (&v)[8][CT]) {
  unsigned mask = 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      const bool on = v[i][c] > 0.f;
      mask |= (on ? 1u : 0u) << (i * CT + c);
      v[i][c] = fmaxf(v[i][c], 0.f);
    }
  return mask;
}

// Shared-memory layout (floats): features, h1, h2, z (later dz), packed parameters.  Up to B = 8
// two gradient CTAs fit an SM.
template <int H, int B>
struct FwdSmem {
  static constexpr int F = 0, H1 = F + kNFeat * kLd, H2 = H1 + H * kLd, Z = H2 + H * kLd,
                       PAR = Z + B * kLd, END = (PAR + MlpParams<H, B>::COUNT + 3) & ~3;
};

// Rows [r0, r0 + kTile) of F (zero past n) into the tile, then h1, h2 and z; m1, m2: the thread's relu masks.  Ends with a barrier.
template <int H, int B>
__device__ __forceinline__ void tile_forward(float* sm, const float* __restrict__ F, int64_t r0, int64_t n,
                                             const TileMap& tm, unsigned* m1, unsigned* m2) {
  using P = MlpParams<H, B>;
  using S = FwdSmem<H, B>;
  constexpr int CT = H / 16;
  const float* sp = sm + S::PAR;
  {
    const int r = threadIdx.x >> 1, i0 = 4 * (threadIdx.x & 1);
    float f[4] = {0.f, 0.f, 0.f, 0.f};
    if (r0 + r < n) {
#pragma unroll
      for (int i = 0; i < 4; ++i) f[i] = F[(r0 + r) * kNFeat + i0 + i];
    }
    __syncthreads();   // the previous tile is consumed
#pragma unroll
    for (int i = 0; i < 4; ++i) sm[S::F + (i0 + i) * kLd + r] = f[i];
  }
  __syncthreads();
  float v[8][CT];
  auto bias = [&](int off) {
    float bv[CT];
    ld_units<CT>(sp + off + tm.cg * CT, bv);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < CT; ++c) v[i][c] = bv[c];
  };
  bias(P::B1);
  tile_gemm<H, kNFeat>(sm + S::F, sp + P::W1, tm, v);
  *m1 = tile_relu<CT>(v);
  tile_store<H>(sm + S::H1, tm, v);
  __syncthreads();
  bias(P::B2);
  tile_gemm<H, H>(sm + S::H1, sp + P::W2, tm, v);
  *m2 = tile_relu<CT>(v);
  tile_store<H>(sm + S::H2, tm, v);
  __syncthreads();
  {
    // two neighbouring lanes per row, one for the even units and one for the odd ones
    const int r = threadIdx.x >> 1, half = threadIdx.x & 1;
    float z[B];
#pragma unroll
    for (int j = 0; j < B; ++j) z[j] = half == 0 ? sp[P::B3 + j] : 0.f;
#pragma unroll 8
    for (int q = half; q < H; q += 2) {
      const float h = sm[S::H2 + q * kLd + r];
#pragma unroll
      for (int j = 0; j < B; ++j) z[j] = fmaf(h, sp[P::W3 + q * B + j], z[j]);
    }
#pragma unroll
    for (int j = 0; j < B; ++j) {
      z[j] += __shfl_xor_sync(0xffffffffu, z[j], 1);
      if (half == 0) sm[S::Z + j * kLd + r] = z[j];
    }
  }
  __syncthreads();
}

template <int H, int B>
__global__ void __launch_bounds__(kThr, 2) mlp_forward_kernel(const float* __restrict__ F, int64_t n,
                                                              const float* __restrict__ params,
                                                              float* __restrict__ Z) {
  using P = MlpParams<H, B>;
  using S = FwdSmem<H, B>;
  extern __shared__ __align__(16) float sm[];
  for (int e = threadIdx.x; e < P::COUNT; e += kThr) sm[S::PAR + e] = params[e];
  const TileMap tm;
  unsigned m1, m2;
  for (int64_t r0 = (int64_t)blockIdx.x * kTile; r0 < n; r0 += (int64_t)gridDim.x * kTile) {
    tile_forward<H, B>(sm, F, r0, n, tm, &m1, &m2);
    const int rows = (int)min((int64_t)kTile, n - r0);
    for (int e = threadIdx.x; e < rows * B; e += kThr) {
      const int r = e / B, j = e % B;
      Z[r0 * B + e] = sm[S::Z + j * kLd + r];
    }
  }
}

// ---------------------------------------------------------------- loss statistics
// TT = 0 (column form): partial[cta] = [s_j = sum_i z_ij u_ij (B), q_j = sum_i z_ij^2 (B)].
// TT > 0 (subspace form, U is n x TT): partial[cta] = [S_tj = sum_i u_it z_ij (TT x B), q_j (B)].
// SPAN: the second block holds the full Gram M = Z^T Z (B x B) instead of its diagonal q.
template <int TT, int B, bool SPAN = false> struct StatsShape {
  static constexpr int NS = TT == 0 ? B : TT * B;
  static constexpr int NQ = SPAN ? B * B : B;
  static constexpr int NP = NS + NQ;
};

// The tile's z and target rows are widened to FP64 in shared memory once (by integer operations:
// the conversion instruction would share the FP64 pipe with the sums); thread (e, slice) then adds
// the products of output e over the rows of its slice in FP64.
template <int H, int B, int TT, bool SPAN = false>
struct StatsSmem {
  static constexpr int NU = TT == 0 ? B : TT, LDD = kTile + 1;   // doubles per column, odd
  static constexpr int ZD = (FwdSmem<H, B>::END + 1) & ~1;       // floats before the doubles
  static constexpr size_t BYTES = ZD * sizeof(float) + (size_t)(B + NU) * LDD * sizeof(double);
};

template <int H, int B, int TT, bool SPAN = false>
__global__ void __launch_bounds__(kThr, 2) mlp_stats_kernel(const float* __restrict__ F, int64_t n,
                                                            const float* __restrict__ params,
                                                            const float* __restrict__ U,
                                                            double* __restrict__ partial) {
  using P = MlpParams<H, B>;
  using S = FwdSmem<H, B>;
  using SS = StatsShape<TT, B, SPAN>;
  using SM = StatsSmem<H, B, TT, SPAN>;
  constexpr int NU = SM::NU, LDD = SM::LDD;
  constexpr int SL = kThr / SS::NP;   // slices of a tile's rows
  static_assert(SL >= 1, "one output per thread at most");
  extern __shared__ __align__(16) float sm[];
  double* zd = reinterpret_cast<double*>(sm + SM::ZD);   // [B][LDD], then the targets [NU][LDD]
  double* ud = zd + B * LDD;
  for (int e = threadIdx.x; e < P::COUNT; e += kThr) sm[S::PAR + e] = params[e];
  const TileMap tm;
  unsigned m1, m2;
  const int out = threadIdx.x % SS::NP, sl = threadIdx.x / SS::NP;
  // output `out` is the sum over the rows of x[r] y[r]
  const double *x, *y;
  if (out < SS::NS) {
    x = zd + (TT == 0 ? out : out % B) * LDD;
    y = ud + (TT == 0 ? out : out / B) * LDD;
  } else {
    const int q = out - SS::NS;
    x = zd + (SPAN ? q / B : q) * LDD;
    y = zd + (SPAN ? q % B : q) * LDD;
  }
  double acc = 0.0;
  for (int64_t r0 = (int64_t)blockIdx.x * kTile; r0 < n; r0 += (int64_t)gridDim.x * kTile) {
    tile_forward<H, B>(sm, F, r0, n, tm, &m1, &m2);
    const int rows = (int)min((int64_t)kTile, n - r0);
    for (int e = threadIdx.x; e < rows * B; e += kThr) {
      const int r = e % rows, j = e / rows;
      zd[j * LDD + r] = f32_to_f64(sm[S::Z + j * kLd + r]);
    }
    for (int e = threadIdx.x; e < rows * NU; e += kThr)
      ud[(e % NU) * LDD + e / NU] = f32_to_f64(U[r0 * NU + e]);
    __syncthreads();
    if (sl < SL) {
      double a = 0.0;
#pragma unroll 4
      for (int r = sl; r < rows; r += SL) a = fma(x[r], y[r], a);
      acc += a;
    }
  }
  __syncthreads();
  double* red = zd;   // SL x NP
  if (sl < SL) red[sl * SS::NP + out] = acc;
  __syncthreads();
  if ((int)threadIdx.x < SS::NP) {
    double t = 0.0;
    for (int k = 0; k < SL; ++k) t += red[k * SS::NP + threadIdx.x];
    partial[(int64_t)blockIdx.x * SS::NP + threadIdx.x] = t;
  }
}

// ---------------------------------------------------------------- backward
// Per tile: forward, dz from the statistics, then
//   gW3 = h2^T dz, dh2 = (dz W3^T) [h2 > 0], gW2 = h1^T dh2, dh1 = (dh2 W2^T) [h1 > 0],
//   gW1 = F^T dh1 and the bias sums,
// with h2's memory reused for dh2 and then dh1.  A gradient entry belongs to one thread, which
// sums a tile in one accumulator and the tiles in another (FP32; deterministic).  Shared-memory
// bandwidth bounds it: 3 H^2 of the (3 (8 H + H B) + 3 H^2) FMAs per row are the three products above.
// Measured at n = 262141, H = 64, b = 4, t = 8 against one row per thread with shared-memory
// operands (loss and gradient, all kernels): 1.98 -> 0.37 ms, of which this
// kernel 1.07 -> 0.21 ms and the statistics 0.20 -> 0.09 ms.
template <int H, int B, int TT, bool SPAN = false>
struct GradSmem {
  static constexpr int W2T = FwdSmem<H, B>::END, COEF = W2T + H * H,
                       TOTAL = COEF + StatsShape<TT, B, SPAN>::NP;
};

// dz_ij: column form ca_j u_ij + cb_j z_ij; subspace form sum_t u_it A_tj + c_j z_ij; span form
// sum_t u_it A_tj + sum_k z_ik C_kj, with the coefficients in shared memory.
template <int H, int B, int TT, bool SPAN = false>
__global__ void __launch_bounds__(kThr, 2) mlp_grad_kernel(const float* __restrict__ F, int64_t n,
                                                           const float* __restrict__ params,
                                                           const float* __restrict__ U,
                                                           const double* __restrict__ coef,
                                                           double* __restrict__ partial) {
  using P = MlpParams<H, B>;
  using S = FwdSmem<H, B>;
  using G = GradSmem<H, B, TT, SPAN>;
  using SS = StatsShape<TT, B, SPAN>;
  constexpr int CT = H / 16;
  constexpr int N3 = (H * B + kThr - 1) / kThr, N1 = kNFeat * H / kThr;   // W3, W1 entries per thread
  extern __shared__ __align__(16) float sm[];
  float* sp = sm + S::PAR;
  float* w2t = sm + G::W2T;
  float* sc = sm + G::COEF;
  const int tid = threadIdx.x;
  for (int e = tid; e < P::COUNT; e += kThr) sp[e] = params[e];
  for (int e = tid; e < H * H; e += kThr) w2t[(e % H) * H + e / H] = params[P::W2 + e];
  for (int e = tid; e < SS::NP; e += kThr) sc[e] = (float)coef[e];
  const TileMap tm;
  const int pg = tm.r0 / 4;   // W2 entries (pg + 16 i, cg + 16 j)
  float a1[N1], a2[CT][CT], a3[N3], ab[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < N1; ++k) a1[k] = 0.f;
#pragma unroll
  for (int k = 0; k < N3; ++k) a3[k] = 0.f;
#pragma unroll
  for (int i = 0; i < CT; ++i)
#pragma unroll
    for (int j = 0; j < CT; ++j) a2[i][j] = 0.f;
  // sum over the tile's rows of x[r] y[r] and of x[r]
  auto dot = [](const float* x, const float* y) {
    float t = 0.f;
#pragma unroll 8
    for (int r = 0; r < kTile; r += 4) {
      const float4 u = *reinterpret_cast<const float4*>(x + r), v = *reinterpret_cast<const float4*>(y + r);
      t = fmaf(u.x, v.x, t);
      t = fmaf(u.y, v.y, t);
      t = fmaf(u.z, v.z, t);
      t = fmaf(u.w, v.w, t);
    }
    return t;
  };
  auto sum = [](const float* x) {
    float t = 0.f;
#pragma unroll 8
    for (int r = 0; r < kTile; r += 4) {
      const float4 u = *reinterpret_cast<const float4*>(x + r);
      t += (u.x + u.y) + (u.z + u.w);
    }
    return t;
  };
  for (int64_t r0 = (int64_t)blockIdx.x * kTile; r0 < n; r0 += (int64_t)gridDim.x * kTile) {
    unsigned m1, m2;
    tile_forward<H, B>(sm, F, r0, n, tm, &m1, &m2);
    // dz (zero past n, where h1 and h2 are not)
    if (tid < kTile) {
      float z[B], dz[B];
      const bool on = r0 + tid < n;
#pragma unroll
      for (int j = 0; j < B; ++j) z[j] = sm[S::Z + j * kLd + tid];
      if (SPAN) {
#pragma unroll
        for (int j = 0; j < B; ++j) {
          float a = 0.0f;
#pragma unroll
          for (int k = 0; k < B; ++k) a = fmaf(z[k], sc[SS::NS + (k * B + j) % SS::NQ], a);
          dz[j] = a;
        }
      } else {
#pragma unroll
        for (int j = 0; j < B; ++j) dz[j] = sc[SS::NS + j] * z[j];
      }
      if (on) {
        const int64_t i = r0 + tid;
        if (TT == 0) {
#pragma unroll
          for (int j = 0; j < B; ++j) dz[j] = fmaf(sc[j], U[i * B + j], dz[j]);
        } else {
#pragma unroll
          for (int tt = 0; tt < (TT == 0 ? 1 : TT); ++tt) {
            const float u = U[i * (TT == 0 ? 1 : TT) + tt];
#pragma unroll
            for (int j = 0; j < B; ++j) dz[j] = fmaf(u, sc[tt * B + j], dz[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < B; ++j) sm[S::Z + j * kLd + tid] = on ? dz[j] : 0.f;
    }
    __syncthreads();
    // gW3, gb3 (h2 and dz), then dh2 over h2
#pragma unroll
    for (int k = 0; k < N3; ++k) {
      const int e = tid + k * kThr;
      if (e < H * B) a3[k] += dot(sm + S::H2 + (e / B) * kLd, sm + S::Z + (e % B) * kLd);
    }
    if (tid < B) ab[2] += sum(sm + S::Z + tid * kLd);
    float v[8][CT];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < CT; ++c) v[i][c] = 0.f;
#pragma unroll
    for (int j = 0; j < B; ++j) {
      const float4 d0 = *reinterpret_cast<const float4*>(sm + S::Z + j * kLd + tm.r0);
      const float4 d1 = *reinterpret_cast<const float4*>(sm + S::Z + j * kLd + tm.r0 + 64);
      const float dv[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        const float w = sp[P::W3 + (tm.cg * CT + c) * B + j];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i][c] = fmaf(dv[i], w, v[i][c]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < CT; ++c) v[i][c] = (m2 >> (i * CT + c)) & 1u ? v[i][c] : 0.f;
    __syncthreads();
    tile_store<H>(sm + S::H2, tm, v);
    __syncthreads();
    // gW2, gb2 (h1 and dh2); dh1 in registers
    {
      float t[CT][CT];
#pragma unroll
      for (int i = 0; i < CT; ++i)
#pragma unroll
        for (int j = 0; j < CT; ++j) t[i][j] = 0.f;
      const float* x = sm + S::H1 + pg * kLd;
      const float* y = sm + S::H2 + tm.cg * kLd;
#pragma unroll 2
      for (int r = 0; r < kTile; r += 4) {
        float4 xv[CT], yv[CT];
#pragma unroll
        for (int i = 0; i < CT; ++i) xv[i] = *reinterpret_cast<const float4*>(x + 16 * i * kLd + r);
#pragma unroll
        for (int j = 0; j < CT; ++j) yv[j] = *reinterpret_cast<const float4*>(y + 16 * j * kLd + r);
#pragma unroll
        for (int i = 0; i < CT; ++i)
#pragma unroll
          for (int j = 0; j < CT; ++j) {
            t[i][j] = fmaf(xv[i].x, yv[j].x, t[i][j]);
            t[i][j] = fmaf(xv[i].y, yv[j].y, t[i][j]);
            t[i][j] = fmaf(xv[i].z, yv[j].z, t[i][j]);
            t[i][j] = fmaf(xv[i].w, yv[j].w, t[i][j]);
          }
      }
#pragma unroll
      for (int i = 0; i < CT; ++i)
#pragma unroll
        for (int j = 0; j < CT; ++j) a2[i][j] += t[i][j];
    }
    if (tid < H) ab[1] += sum(sm + S::H2 + tid * kLd);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < CT; ++c) v[i][c] = 0.f;
    tile_gemm<H, H>(sm + S::H2, w2t, tm, v);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < CT; ++c) v[i][c] = (m1 >> (i * CT + c)) & 1u ? v[i][c] : 0.f;
    __syncthreads();
    tile_store<H>(sm + S::H2, tm, v);
    __syncthreads();
    // gW1, gb1 (F and dh1)
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      const int e = tid + k * kThr;
      a1[k] += dot(sm + S::F + (e / H) * kLd, sm + S::H2 + (e % H) * kLd);
    }
    if (tid < H) ab[0] += sum(sm + S::H2 + tid * kLd);
  }
  double* out = partial + (int64_t)blockIdx.x * P::COUNT;
#pragma unroll
  for (int k = 0; k < N1; ++k) out[P::W1 + tid + k * kThr] = (double)a1[k];
#pragma unroll
  for (int i = 0; i < CT; ++i)
#pragma unroll
    for (int j = 0; j < CT; ++j) out[P::W2 + (pg + 16 * i) * H + tm.cg + 16 * j] = (double)a2[i][j];
#pragma unroll
  for (int k = 0; k < N3; ++k)
    if (tid + k * kThr < H * B) out[P::W3 + tid + k * kThr] = (double)a3[k];
  if (tid < H) {
    out[P::B1 + tid] = (double)ab[0];
    out[P::B2 + tid] = (double)ab[1];
  }
  if (tid < B) out[P::B3 + tid] = (double)ab[2];
}

// grad[e] = sum over the CTAs' partials: 64 entries per block, four threads each taking every
// fourth CTA in order, then a fixed sum of the four.
__global__ void __launch_bounds__(256) grad_reduce_kernel(const double* __restrict__ partial, int nctas, int count,
                                                          float* __restrict__ grad) {
  __shared__ double red[4][64];
  const int e = blockIdx.x * 64 + (threadIdx.x & 63), part = threadIdx.x >> 6;
  double s = 0.0;
  if (e < count) {
#pragma unroll 8
    for (int c = part; c < nctas; c += 4) s += partial[(int64_t)c * count + e];
  }
  red[part][threadIdx.x & 63] = s;
  __syncthreads();
  if (part == 0 && e < count)
    grad[e] = (float)((red[0][threadIdx.x] + red[1][threadIdx.x]) + (red[2][threadIdx.x] + red[3][threadIdx.x]));
}

// tot[e] = sum over c < nctas of partial[c * np + e], e < np: one warp per output, lane l adding
// partials l, l + 32, .. in order, then a fixed tree.  All threads call it; ends with a barrier.
__device__ void sum_partials(const double* __restrict__ partial, int nctas, int np, double* tot) {
  const int lane = threadIdx.x & 31;
  for (int e = threadIdx.x >> 5; e < np; e += blockDim.x >> 5) {
    double s = 0.0;
#pragma unroll 4
    for (int c = lane; c < nctas; c += 32) s += partial[(int64_t)c * np + e];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) tot[e] = s;
  }
  __syncthreads();
}

// From the per-CTA partials: T = 0 (column form) coef = [-2 s_j/q_j (B), 2 s_j^2/q_j^2 (B)],
// L = sum_j (1 - s_j^2/q_j); T > 0 (subspace form) coef = [-2 S_tj/q_j (T x B), 2 P_j/q_j^2 (B)]
// with P_j = sum_t S_tj^2, L = sum_j (1 - P_j/q_j).  One CTA, a thread per column.
constexpr int kCoefThreads = 512;
__global__ void __launch_bounds__(kCoefThreads) loss_coef_kernel(const double* __restrict__ partial, int nctas, int B,
                                                                 int T, double* __restrict__ coef,
                                                                 double* __restrict__ loss) {
  __shared__ double tot[256], Lj[16];
  const int ns = T == 0 ? B : T * B, np = ns + B, rows = T == 0 ? 1 : T;
  sum_partials(partial, nctas, np, tot);
  const int j = threadIdx.x;
  if (j < B) {
    const double q = tot[ns + j];
    double P = 0.0;
    for (int t = 0; t < rows; ++t) {
      const double st = tot[t * B + j];
      P += st * st;
      coef[t * B + j] = q > 0.0 ? -2.0 * st / q : 0.0;
    }
    coef[ns + j] = q > 0.0 ? 2.0 * P / (q * q) : 0.0;
    Lj[j] = q > 0.0 ? 1.0 - P / q : 1.0;
  }
  __syncthreads();
  if (j == 0) {
    double L = 0.0;
    for (int k = 0; k < B; ++k) L += Lj[k];
    *loss = L;
  }
}

// Span form: from partials [S (T x B), M (B x B)]: N = S^T S, Mi = M^{-1} (Gauss-Jordan with
// partial pivoting, B <= 8), coef = [A = -2 S Mi (T x B), C = 2 Mi N Mi (B x B)],
// loss = B - tr(Mi N).  One CTA, a thread per matrix entry; the sums of the partials and the
// B elimination steps are its time (B = 4, T = 8: 649 us with one thread for all of it, 18 us now).
__global__ void __launch_bounds__(kCoefThreads) span_coef_kernel(const double* __restrict__ partial, int nctas, int B,
                                                                 int T, double* __restrict__ coef,
                                                                 double* __restrict__ loss) {
  __shared__ double tot[256], A[8][16], N[8 * 8], X[8 * 8];   // A = [M | I] -> [I | Mi]
  __shared__ int piv, ok;
  const int ns = T * B, np = ns + B * B, tid = threadIdx.x;
  sum_partials(partial, nctas, np, tot);
  const double* S = tot;
  const int i = tid / 16, k = tid % 16;   // entry of A (128 threads)
  const bool on = tid < 128 && i < B && k < 2 * B;
  if (on) A[i][k] = k < B ? tot[ns + i * B + k] : (k - B == i ? 1.0 : 0.0);
  if (tid < B * B) {                      // N = S^T S
    double v = 0.0;
    for (int t = 0; t < T; ++t) v = fma(S[t * B + tid / B], S[t * B + tid % B], v);
    N[tid] = v;
  }
  if (tid == 0) ok = 1;
  __syncthreads();
  for (int c = 0; c < B; ++c) {
    if (tid == 0) {
      int p = c;
      for (int r = c + 1; r < B; ++r)
        if (fabs(A[r][c]) > fabs(A[p][c])) p = r;
      piv = p;
      if (!(fabs(A[p][c]) > 0.0)) ok = 0;
    }
    __syncthreads();
    if (!ok) break;
    const int p = piv;
    // row i after the exchange of rows c and p, minus its multiple of the scaled pivot row
    double v = 0.0;
    if (on) {
      const double pr = A[p][k] / A[p][c];
      const int src = i == p ? c : i;
      v = i == c ? pr : A[src][k] - A[src][c] * pr;
    }
    __syncthreads();
    if (on) A[i][k] = v;
    __syncthreads();
  }
  if (!ok) {
    for (int e = tid; e < np; e += blockDim.x) coef[e] = 0.0;
    if (tid == 0) *loss = (double)B;
    return;
  }
  if (tid < B * B) {                      // X = Mi N
    double v = 0.0;
    for (int l = 0; l < B; ++l) v = fma(A[tid / B][B + l], N[l * B + tid % B], v);
    X[tid] = v;
  }
  __syncthreads();
  if (tid < T * B) {                      // A = -2 S Mi
    double v = 0.0;
    for (int l = 0; l < B; ++l) v = fma(S[(tid / B) * B + l], A[l][B + tid % B], v);
    coef[tid] = -2.0 * v;
  }
  if (tid < B * B) {                      // C = 2 (Mi N) Mi
    double v = 0.0;
    for (int l = 0; l < B; ++l) v = fma(X[(tid / B) * B + l], A[l][B + tid % B], v);
    coef[ns + tid] = 2.0 * v;
  }
  if (tid == 0) {
    double tr = 0.0;
    for (int l = 0; l < B; ++l) tr += X[l * B + l];
    *loss = (double)B - tr;
  }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t count, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.0f - b1) * gg;
    const float vv = b2 * v[e] + (1.0f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    p[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  }
}

// ---------------------------------------------------------------- dispatch
// One CTA per tile up to the resident CTAs (two per SM where shared memory allows).
template <int H, int B>
static int forward_hb(const float* F, int64_t n, const float* params, float* Z, cudaStream_t s) {
  const size_t smem = sizeof(float) * FwdSmem<H, B>::END;
  static KernelSetup ks;
  const void* fn = reinterpret_cast<const void*>(mlp_forward_kernel<H, B>);
  FE_TRY(kernel_configure(ks, fn, (int)smem));
  int per_sm = 0;
  FE_TRY(kernel_occupancy(ks, fn, kThr, smem, 0, &per_sm));
  const int ctas = (int)std::min<int64_t>(ceil_div(n, kTile), (int64_t)per_sm * num_sms());
  mlp_forward_kernel<H, B><<<std::max(ctas, 1), kThr, smem, s>>>(F, n, params, Z);
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

template <int H, int B, int TT = 0, bool SPAN = false>
static int loss_grad_hb(const float* F, int64_t n, const float* params, const float* U,
                        float* grad, double* loss_host, cudaStream_t s) {
  using P = MlpParams<H, B>;
  using SS = StatsShape<TT, B, SPAN>;
  const size_t ssmem = StatsSmem<H, B, TT, SPAN>::BYTES;
  const size_t gsmem = sizeof(float) * GradSmem<H, B, TT, SPAN>::TOTAL;
  static KernelSetup kst, kgr;
  const void* fs = reinterpret_cast<const void*>(mlp_stats_kernel<H, B, TT, SPAN>);
  const void* fg = reinterpret_cast<const void*>(mlp_grad_kernel<H, B, TT, SPAN>);
  FE_TRY(kernel_configure(kst, fs, (int)ssmem));
  FE_TRY(kernel_configure(kgr, fg, (int)gsmem));
  int sper = 0, gper = 0;
  FE_TRY(kernel_occupancy(kst, fs, kThr, ssmem, 0, &sper));
  FE_TRY(kernel_occupancy(kgr, fg, kThr, gsmem, 0, &gper));
  const int64_t tiles = std::max<int64_t>(1, ceil_div(n, kTile));
  const int sctas = (int)std::min<int64_t>(tiles, (int64_t)sper * num_sms());
  const int gctas = (int)std::min<int64_t>(tiles, (int64_t)gper * num_sms());
  double* part = small_scratch(15, (size_t)sctas * SS::NP + SS::NP + 1);
  double* gpart = small_scratch(16, (size_t)gctas * P::COUNT);
  if (!part || !gpart) return FE_ERR_OOM;
  double* coef = part + (size_t)sctas * SS::NP;
  double* dloss = coef + SS::NP;
  mlp_stats_kernel<H, B, TT, SPAN><<<sctas, kThr, ssmem, s>>>(F, n, params, U, part);
  count_launch();
  if (SPAN) span_coef_kernel<<<1, kCoefThreads, 0, s>>>(part, sctas, B, TT, coef, dloss);
  else loss_coef_kernel<<<1, kCoefThreads, 0, s>>>(part, sctas, B, TT, coef, dloss);
  count_launch();
  mlp_grad_kernel<H, B, TT, SPAN><<<gctas, kThr, gsmem, s>>>(F, n, params, U, coef, gpart);
  count_launch();
  grad_reduce_kernel<<<(unsigned)ceil_div(P::COUNT, 64), 256, 0, s>>>(gpart, gctas, P::COUNT, grad);
  count_launch();
  FE_CUDA(cudaGetLastError());
  if (loss_host) {
    FE_CUDA(cudaMemcpyAsync(loss_host, dloss, sizeof(double), cudaMemcpyDeviceToHost, s));
    FE_CUDA(cudaStreamSynchronize(s));
  }
  return FE_OK;
}

#define FE_MLP_DISPATCH(H, EXPR_B)                                   \
  switch (b) {                                                       \
    case 1: return EXPR_B(H, 1);                                     \
    case 2: return EXPR_B(H, 2);                                     \
    case 4: return EXPR_B(H, 4);                                     \
    case 8: return EXPR_B(H, 8);                                     \
    case 16: return EXPR_B(H, 16);                                   \
  }

int mlp_forward(const float* F, int64_t n, const float* params, int hidden, int b, float* Z,
                cudaStream_t s) {
#define FWD(H, B) forward_hb<H, B>(F, n, params, Z, s)
  if (hidden == 64) { FE_MLP_DISPATCH(64, FWD) }
  if (hidden == 32) { FE_MLP_DISPATCH(32, FWD) }
#undef FWD
  return set_error(FE_ERR_INVALID, "mlp: hidden must be 32 or 64 and b in {1,2,4,8,16} (got %d, %d)", hidden, b);
}

int mlp_loss_grad(const float* F, int64_t n, const float* params, int hidden, int b,
                  const float* U, float* grad, double* loss, cudaStream_t s) {
#define LG(H, B) loss_grad_hb<H, B>(F, n, params, U, grad, loss, s)
  if (hidden == 64) { FE_MLP_DISPATCH(64, LG) }
  if (hidden == 32) { FE_MLP_DISPATCH(32, LG) }
#undef LG
  return set_error(FE_ERR_INVALID, "mlp: hidden must be 32 or 64 and b in {1,2,4,8,16} (got %d, %d)", hidden, b);
}

int mlp_subspace_loss_grad(const float* F, int64_t n, const float* params, int hidden, int b,
                           const float* U, int t, float* grad, double* loss, cudaStream_t s) {
#define SLG(TT, B) loss_grad_hb<64, B, TT>(F, n, params, U, grad, loss, s)
  if (hidden == 64 && (b == 4 || b == 8) && (t == 4 || t == 8 || t == 16)) {
    if (b == 4) {
      if (t == 4) return SLG(4, 4);
      if (t == 8) return SLG(8, 4);
      return SLG(16, 4);
    }
    if (t == 4) return SLG(4, 8);
    if (t == 8) return SLG(8, 8);
    return SLG(16, 8);
  }
#undef SLG
  return set_error(FE_ERR_INVALID, "mlp subspace loss: needs hidden 64, b in {4, 8}, t in {4, 8, 16} (got %d, %d, %d)", hidden, b, t);
}

int mlp_span_loss_grad(const float* F, int64_t n, const float* params, int hidden, int b,
                       const float* U, int t, float* grad, double* loss, cudaStream_t s) {
#define PLG(TT, B) loss_grad_hb<64, B, TT, true>(F, n, params, U, grad, loss, s)
  if (hidden == 64 && b == 4 && t == 4) return PLG(4, 4);
  if (hidden == 64 && b == 4 && t == 8) return PLG(8, 4);
  if (hidden == 64 && b == 8 && t == 8) return PLG(8, 8);
#undef PLG
  return set_error(FE_ERR_INVALID, "mlp span loss: needs hidden 64 and (b, t) in {(4,4), (4,8), (8,8)} (got %d, %d, %d)", hidden, b, t);
}

// Start block for fe_eigs: features -> MLP -> FP64 row-major n x b (the solver orthonormalises).
int mlp_start_block(fe_csr h, const float* weights, int hidden, int b, uint64_t seed,
                    double* out, cudaStream_t s) {
  const int64_t n = h->n;
  DevBuf fbuf, zbuf;
  FE_TRY(fbuf.alloc(sizeof(float) * (size_t)n * kNFeat));
  FE_TRY(zbuf.alloc(sizeof(float) * (size_t)n * b));
  FE_TRY(vertex_features(h, seed, fbuf.as<float>(), s));
  FE_TRY(mlp_forward(fbuf.as<float>(), n, weights, hidden, b, zbuf.as<float>(), s));
  FE_TRY(convert_block(zbuf.p, FE_F32, b, out, FE_F64, b, n, b, s));
  FE_CUDA(cudaStreamSynchronize(s));
  return FE_OK;
}

}  // namespace fe

using namespace fe;

extern "C" {

int64_t fe_mlp_param_count(int hidden, int b) {
  if ((hidden != 32 && hidden != 64) || !is_pow2_le16(b)) return -1;
  return mlp_param_count(hidden, b);
}

int fe_vertex_features(fe_csr h, uint64_t seed, float* F) {
  FE_ARG(h && F, "fe_vertex_features: NULL argument");
  return vertex_features(h, seed, F, cur_stream());
}

int fe_mlp_forward(const float* F, int64_t n, const float* params, int hidden, int b, float* Z) {
  FE_ARG(F && params && Z && n >= 1, "fe_mlp_forward: bad argument");
  return mlp_forward(F, n, params, hidden, b, Z, cur_stream());
}

int fe_mlp_loss_grad(const float* F, int64_t n, const float* params, int hidden, int b,
                     const float* U, float* grad, double* loss) {
  FE_ARG(F && params && U && grad && n >= 1, "fe_mlp_loss_grad: bad argument");
  return mlp_loss_grad(F, n, params, hidden, b, U, grad, loss, cur_stream());
}

int fe_mlp_subspace_loss_grad(const float* F, int64_t n, const float* params, int hidden, int b,
                              const float* U, int t, float* grad, double* loss) {
  FE_ARG(F && params && U && grad && n >= 1, "fe_mlp_subspace_loss_grad: bad argument");
  return mlp_subspace_loss_grad(F, n, params, hidden, b, U, t, grad, loss, cur_stream());
}

int fe_mlp_span_loss_grad(const float* F, int64_t n, const float* params, int hidden, int b,
                          const float* U, int t, float* grad, double* loss) {
  FE_ARG(F && params && U && grad && n >= 1, "fe_mlp_span_loss_grad: bad argument");
  return mlp_span_loss_grad(F, n, params, hidden, b, U, t, grad, loss, cur_stream());
}

int fe_mlp_adam(float* params, const float* grad, float* m, float* v, int64_t count, double lr,
                double beta1, double beta2, double eps, int step) {
  FE_ARG(params && grad && m && v && count >= 1 && step >= 1, "fe_mlp_adam: bad argument");
  const float c1 = 1.0f - (float)pow(beta1, step), c2 = 1.0f - (float)pow(beta2, step);
  const int ctas = (int)std::min<int64_t>(ceil_div(count, 256), 4 * num_sms());
  adam_kernel<<<std::max(ctas, 1), 256, 0, cur_stream()>>>(params, grad, m, v, count, (float)lr,
                                                          (float)beta1, (float)beta2, (float)eps, c1, c2);
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

}  // extern "C"
