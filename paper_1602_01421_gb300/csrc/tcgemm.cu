// FP64 tall-skinny products on the FP16 tensor cores by exact digit splitting ("split
// products"; the Ozaki scheme, Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012), for
// the restart / Ritz-vector product of the Block Krylov-Schur solver (Table 1 "op1" shape,
// V_out = V Y with V n x K, Y K x N, K <= 64 and N <= 32):
//
//   * every V row is scaled by its largest binary exponent and its 53-bit aligned significands
//     are cut into seven 8-bit digits (sign-magnitude, so every digit is an integer in
//     [-255, 255]; as an operand it is d 2^-24, a subnormal FP16 number, exact): V[r][c] = 2^(Er - 1075) sum_i d_i[r][c] 2^(45 - 8 i);
//   * every Y column likewise by its largest exponent: Y[c][q] = 2^(Fq - 1075) sum_j e_j 2^(45-8j);
//   * the digit products are exact in the tensor core's FP32 accumulator as long as each
//     accumulator sums at most 2^24 / 255^2 = 258 of them: one accumulator per digit-weight
//     class g = i + j (g <= 6) and per 32-wide slice of K holds at most 7 * 32 products;
//   * V Y = 2^(Er + Fq - 2108) * T with T = sum_g D_g 2^(8 (6 - g)), assembled in 64-bit
//     integer arithmetic from the accumulators (T / 2^12, rounded) and rounded once to FP64.
//
// Error: the digit products dropped (i + j >= 7), the truncation of each entry below its
// row's (column's) leading bit and the 12 dropped bits of T bound |error| <=
// 2^-49 (K + 1) max_c |V[r][c]| max_c |Y[c][q]| + 2^-52 |result|.  The FP64 pipe (1/64 of the FP32
// rate on this part) only converts: one 64-bit integer per result.
//
// What bounds these kernels is the integer work of the split and of the assembly, on an ALU that takes
// a warp's instruction every other clock, and the latencies between the phases of a tile.  So a value
// is cut with as few instructions as possible (digits8: 11 for the 14 digits of two values), a result
// assembled with 32-bit multiply-adds before 64-bit ones (sum7) and converted by one instruction
// (scale_int), and each splitting thread takes one unit of eight values, with registers capped at 64
// so that 28-30 warps fit (without spills: beside the staging buffers L1 has no room for them).
//
// Kernels: for K <= 32 a warp-specialised pipeline (tc_combine_pipe_kernel: TMA producer,
// digit splitters, one MMA-issuing thread, result assemblers over double-buffered tiles; see its
// comment); for 32 < K <= 64 tc_combine_kernel, one 128-row tile per loop trip and two
// persistent CTAs of 256 threads per SM: two threads share a row of the V tile, each splits half
// of its K values into the digit tiles, thread 0 issues one MMA per digit and K-step and commits
// to an mbarrier, then the two threads assemble half of the row's N results each.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "fe_internal.cuh"
#include "tc.cuh"
#include "vec.cuh"

namespace fe {

namespace {

constexpr int kDigits = 7;           // 8-bit digits per 53-bit significand (7 * 8 >= 53)
constexpr int kClasses = 7;          // digit-weight classes g = i + j kept (g <= 6)
constexpr int kTileRows = 128;       // MMA M
constexpr int kKChunk = 32;          // K columns per accumulator set (exactness bound)
constexpr int kMaxK = 64;
constexpr int kMaxN = 32;
constexpr int kThreads = 256;
// Sleeping waits: at most 2^16 polls of up to 32 us each (about 2 s in all).
constexpr uint32_t kPipePolls = 1u << 16;
constexpr uint32_t kPipeSleepNs = 32768;
constexpr int kCoreBytes = 128;      // 8 rows x 16 bytes
// A (V digits): per (K chunk, digit) a 128 x 32 FP16 tile = 8 KB; SBO = 4 core matrices
constexpr int kATileBytes = kTileRows * kKChunk * 2;
constexpr uint32_t kLBO = kCoreBytes;               // next core matrix along K
constexpr uint32_t kSBO = (kKChunk / 8) * kCoreBytes;  // next 8-row group

// Byte offset of element (row, k) of a [rows x 32] 16-bit K-major tile (k < 32).
__host__ __device__ inline uint32_t tile_off(int row, int k) {
  return (uint32_t)((row >> 3) * kSBO + (k >> 3) * kLBO + (row & 7) * 16 + (k & 7) * 2);
}

// Biased exponent field of a double (0 for zero and subnormals, which are read as zero).
__device__ __forceinline__ int exp_field(double x) {
  return (int)((__double_as_longlong(x) >> 52) & 0x7FF);
}

// Significand of x aligned to the binary exponent field emax (>= x's): a non-negative integer
// below 2^53 with x = +-M * 2^(emax - 1075) up to the bits shifted out.
__device__ __forceinline__ uint64_t aligned_sig(double x, int emax) {
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7FF);
  const int sh = emax - e;
  if (e == 0 || sh > 52) return 0;
  return ((u & 0xFFFFFFFFFFFFFull) | (1ull << 52)) >> sh;
}

// Digit i of an aligned significand: bits [45 - 8 i, 52 - 8 i] for i < 6, the low 5 bits
// shifted up by 3 for i = 6 (weight 2^(45 - 8 i) in both cases).
__device__ __forceinline__ uint32_t digit(uint64_t m, int i) {
  return i < 6 ? (uint32_t)(m >> (45 - 8 * i)) & 0xFFu : ((uint32_t)m & 0x1Fu) << 3;
}

// FP16 x2 fused multiply-add on packed halves (round to nearest).
__device__ __forceinline__ uint32_t hfma2_u32(uint32_t x, uint32_t y, uint32_t z) {
  uint32_t d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(x), "r"(y), "r"(z));
  return d;
}

// Eight FP64 values prepared for the cut into digits: their significands aligned to a common exponent
// and shifted up by 3 bits (56 bits: digit i is byte 6 - i), and the signs of neighbouring values in
// bits 15 and 31.
struct Sig8 {
  uint32_t lo[8], hi[8], s2[4];
};

// Largest exponent of the eight values, in its place in the high word (0: all zero or subnormal).
__device__ __forceinline__ uint32_t top_exp8(const double (&x)[8]) {
  uint32_t e = 0;
#pragma unroll
  for (int t = 0; t < 8; ++t) e = max(e, (uint32_t)__double2hiint(x[t]) & 0x7FF00000u);
  return e;
}

// emax: exponent in its place in the high word, at least every value's.  A zero gives zero, and so
// does a value below 2^-56 of 2^emax.  (Subnormals only count beside the smallest normal numbers,
// and then as half their value.)
__device__ __forceinline__ void align8(const double* x, uint32_t emax, Sig8& s) {
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const uint32_t hi = (uint32_t)__double2hiint(x[t]), ev = hi & 0x7FF00000u;
    const uint32_t h = (hi & 0xFFFFFu) | min(ev, 0x100000u);   // with the leading one
    uint64_t m = (((uint64_t)h << 32) | (uint32_t)__double2loint(x[t])) << 3;
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"((emax - ev) >> 20));
    s.lo[t] = (uint32_t)m;
    s.hi[t] = (uint32_t)(m >> 32);
  }
#pragma unroll
  for (int t = 0; t < 4; ++t)
    s.s2[t] = __byte_perm((uint32_t)__double2hiint(x[2 * t]), (uint32_t)__double2hiint(x[2 * t + 1]), 0x7632) & 0x80008000u;
}

// Digits of the eight values with their signs; put(i, w) takes digit i of all eight, as FP16 numbers
// +-d 2^-24: a byte d with zeros above it is the subnormal FP16 number d 2^-24, which the tensor cores
// multiply exactly.  Per pair of values a byte permute takes two neighbouring digit bytes of both and
// one more per digit puts their bytes under the signs: 11 instructions for the 14 digits.
constexpr float kDigitUnit = 16777216.0f;   // 2^24
template <class Put>
__device__ __forceinline__ void digits8(const Sig8& s, Put put) {
#pragma unroll
  for (int g = 0; g < 4; ++g) {   // bytes (6, 5), 4, (3, 2), (1, 0) of the significands
    const int k = g == 0 ? 6 : g == 1 ? 4 : g == 2 ? 3 : 1;
    const uint32_t b1 = k & 3, b0 = g == 1 ? b1 : b1 - 1;
    uint32_t w0[4], w1[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const uint32_t pa = g < 2 ? s.hi[2 * t] : s.lo[2 * t], pb = g < 2 ? s.hi[2 * t + 1] : s.lo[2 * t + 1];
      const uint32_t q = __byte_perm(pa, pb, b1 | (b0 << 4) | ((4 + b1) << 8) | ((4 + b0) << 12));
      w0[t] = __byte_perm(q, s.s2[t], 0x7250);
      w1[t] = __byte_perm(q, s.s2[t], 0x7351);
    }
    put(6 - k, make_uint4(w0[0], w0[1], w0[2], w0[3]));
    if (g != 1) put(7 - k, make_uint4(w1[0], w1[1], w1[2], w1[3]));
  }
}

// The FP16 bits of s d for a digit d in [0, 255] and a sign bit (the same exact FMA).
__device__ __forceinline__ uint16_t digit_f16(uint32_t d, uint32_t sign) {
  const uint32_t s2 = 0x3C00u | (sign << 15);
  return (uint16_t)(hfma2_u32(0x6400u | d, s2, s2 ^ 0xD800u) & 0xFFFFu);
}

// Exact integer value of an FP32 accumulator holding an integer of magnitude below 2^24 in units of
// 1 / unit (a power of two).
__device__ __forceinline__ int32_t acc_int(uint32_t bits, float unit) {
  return __float2int_rn(__uint_as_float(bits) * unit);
}

// Seven accumulators d_g of weights 2^(8 (6 - g)) form T = sum_g d_g 2^(8 (6 - g)); it is taken as
// T / 2^12 rounded to an integer of at most 60 bits: the 12 dropped bits are below the digit
// truncation already made (2^-50 of max|V_r| max|Y_q|).
constexpr int kAsmShift = 12;

// floor((T + 256 rnd) / 2^12): rnd = 8 rounds to the nearest; 16 j more adds j to the result.  d_0 and
// d_2 are below 2^31 / 257 (the sums of up to 128 rows of a Gram tile, 128 * 255^2, and the first three
// classes of a 32-column product), so pairs of them go through 32-bit multiply-adds.
__device__ __forceinline__ int64_t sum7(const uint32_t (&d)[7], float unit, int rnd) {
  const int a01 = acc_int(d[0], unit) * 256 + acc_int(d[1], unit);
  const int a23 = acc_int(d[2], unit) * 256 + acc_int(d[3], unit);
  const int a6 = __float2int_rd(__uint_as_float(d[6]) * (unit * 0.00390625f));   // floor(d_6 / 2^8)
  const int a456 = acc_int(d[4], unit) * 16 + ((acc_int(d[5], unit) + a6 + rnd) >> 4);
  return (int64_t)a01 * (1 << 28) + ((int64_t)a23 * 4096 + a456);
}

// 2^s * t rounded to FP64; zero below the normal range, infinity above it.
__device__ __forceinline__ double scale_int(int64_t t, int s) {
  const double d = __ll2double_rn((long long)t);
  const uint32_t h = (uint32_t)__double2hiint(d);
  const int ef = (int)((h >> 20) & 0x7FFu) + s;
  uint32_t rh = h + ((uint32_t)s << 20), rl = (uint32_t)__double2loint(d);
  if (h == 0 || (uint32_t)(ef - 1) >= 2046u) {
    rh = (h & 0x80000000u) | (h != 0 && ef >= 2047 ? 0x7FF00000u : 0u);
    rl = 0;
  }
  return __hiloint2double((int)rh, (int)rl);
}

// Bounded wait that sleeps until the phase completes: waiting threads take no issue slots from
// the other CTA on the SM.  True when the phase completed.
__device__ __forceinline__ bool wait_sleep(uint64_t* bar, uint32_t parity) {
  return tc::mbar_wait(bar, parity, 1) || tc::mbar_wait_sleep(bar, parity, kPipePolls, kPipeSleepNs);
}

struct TcArgs {
  const double* vblk[kMaxK];   // K / BV blocks of n x BV (ld BV)
  double* oblk[kMaxN];         // N / BV output blocks of n x BV (ld BV); fewer when BV < 4
  int64_t n;
  int K, N, NP;                // NP: N padded to the MMA's N (16 or 32)
  int nkc;                     // K chunks of 32
  const uint16_t* bdig;        // global: [nkc][7][NP x 32] canonical tiles
  const int* fexp;             // global: N column exponent fields of Y
  double beta;                 // Out = beta Out + (alpha V Y); beta = 0: Out is not read
  int bulk;                    // 1: every V block is 16-byte aligned (TMA bulk copies allowed)
  int ovec;                    // 1: every output block is 16-byte aligned (vector stores allowed)
};

}  // namespace

// Y (K x N FP64, row-major, ld ldy) -> per-column exponent fields and the seven digit tiles of
// every 32-row K chunk in the MMA's B layout (row q of B = column q of Y; rows N..NP-1 and
// K beyond K zero).  One CTA, bound by the latency of its few dependent steps: the exponents are
// shared-memory maxima over all of Y (K = 32, N = 4: 2.5 us, 3.5 with a column per thread of 256).
constexpr int kPrepThreads = 512;
__global__ void tc_prep_y_kernel(const double* __restrict__ Y, int ldy, double alpha, int K, int N, int NP,
                                 int nkc, uint16_t* __restrict__ bdig, int* __restrict__ fexp) {
  __shared__ int sf[kMaxN];
  for (int q = threadIdx.x; q < N; q += blockDim.x) sf[q] = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < K * N; e += blockDim.x) {
    const int c = e / N, q = e - c * N;
    atomicMax(sf + q, exp_field(alpha * Y[c * ldy + q]));
  }
  __syncthreads();
  for (int q = threadIdx.x; q < N; q += blockDim.x) fexp[q] = sf[q];
  const int per_tile = NP * kKChunk;  // elements of one [NP x 32] tile
  const int total = nkc * per_tile;
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int kc = e / per_tile, r = e % per_tile;
    const int q = r / kKChunk, k = r % kKChunk;
    const int c = kc * kKChunk + k;
    uint64_t m = 0;
    uint32_t sgn = 0;
    if (q < N && c < K) {
      const double y = alpha * Y[c * ldy + q];
      m = aligned_sig(y, sf[q]);
      sgn = (uint32_t)((uint64_t)__double_as_longlong(y) >> 63);
    }
    for (int j = 0; j < kDigits; ++j) {
      const uint16_t bits = digit_f16(digit(m, j), sgn);
      char* tile = reinterpret_cast<char*>(bdig) + (size_t)(kc * kDigits + j) * per_tile * 2;
      *reinterpret_cast<uint16_t*>(tile + tile_off(q, k)) = bits;
    }
  }
}

// Row r of a 128-row tile is handled by two threads (warps w and w + 4 address the same TMEM
// lane quarter): each loads and splits half of the row's K values, and each assembles half of
// the row's N results.
// 32 < K <= 64 (fewer columns take the pipeline below); 256 TMEM columns up to N = 16, else 512.
template <int BV>
__global__ void __launch_bounds__(kThreads, 1) tc_combine_kernel(const TcArgs a) {
  constexpr int KMAX = kMaxK, KH = KMAX / 2;  // V values per thread
  extern __shared__ __align__(1024) unsigned char smem[];
  const int nkc = a.nkc, NP = a.NP;
  unsigned char* sA = smem;                                        // [nkc][7] x 8 KB
  unsigned char* sB = sA + (size_t)nkc * kDigits * kATileBytes;    // [nkc][7] x NP*64
  const size_t btile = (size_t)NP * kKChunk * 2;
  double* sV = reinterpret_cast<double*>(sB + (size_t)nkc * kDigits * btile);  // [K/BV][128][BV]
  uint64_t* bar = reinterpret_cast<uint64_t*>(sV + (size_t)kTileRows * KMAX);
  uint64_t* lbar = bar + 1;                      // V tile copies
  uint64_t* sDesc = bar + 2;                     // [nkc][7][2] A and B descriptors (K-step 0)
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sDesc + 2 * kDigits * (KMAX / kKChunk) * 2);
  int* sF = reinterpret_cast<int*>(tslot + 1);   // N column exponents of Y
  int* sE = sF + kMaxN;                          // [2][128] partial row exponents
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int half = warp >> 2;
  const int row = (warp & 3) * 32 + lane;        // row of the tile = TMEM lane
  const uint32_t ncols = (uint32_t)nkc * kClasses * NP <= 256 ? 256u : 512u;

  // B digits and column exponents (once per CTA)
  {
    const int4* src = reinterpret_cast<const int4*>(a.bdig);
    int4* dst = reinterpret_cast<int4*>(sB);
    const int n16 = (int)((size_t)nkc * kDigits * btile / 16);
    for (int e = tid; e < n16; e += kThreads) dst[e] = src[e];
    for (int q = tid; q < a.N; q += kThreads) sF[q] = a.fexp[q];
  }
  if (warp == 0) {
    tc::tmem_alloc(tslot, ncols);
    tc::tmem_relinquish();
  }
  const int nblk = a.K / BV;
  const bool add_out = a.beta != 0.0;   // decided once: an FP64 compare per result would
                                        // occupy the FP64 pipe
  const int64_t ntiles = (a.n + kTileRows - 1) / kTileRows;
  // a tile's V rows come in by TMA bulk copies (one per block) when their byte count is a
  // multiple of 16 (every full tile); otherwise (a ragged last tile) by plain loads
  auto bulk_ok = [&](int64_t t) {
    return a.bulk && ((uint64_t)min((int64_t)kTileRows, a.n - t * kTileRows) * BV * 8) % 16 == 0;
  };
  auto issue = [&](int64_t t) {
    const int64_t r0 = t * kTileRows;
    const uint32_t bytes = (uint32_t)(min((int64_t)kTileRows, a.n - r0) * BV * 8);
    tc::mbar_arrive_expect_tx(lbar, bytes * (uint32_t)nblk);
    for (int j = 0; j < nblk; ++j) tc::bulk_g2s(sV + (size_t)j * kTileRows * BV, a.vblk[j] + r0 * BV, bytes, lbar);
  };
  if (tid == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(lbar, 1);
    tc::mbar_fence_init();
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (tid == 0 && (int64_t)blockIdx.x < ntiles && bulk_ok(blockIdx.x)) issue(blockIdx.x);
  const uint32_t tbase = *tslot;
  const uint32_t sa0 = tc::smem_addr(sA), sb0 = tc::smem_addr(sB);
  if (tid == 0)
    for (int kc = 0; kc < nkc; ++kc)
      for (int i = 0; i < kDigits; ++i) {
        sDesc[(kc * kDigits + i) * 2] = tc::smem_desc(sa0 + (uint32_t)((kc * kDigits + i) * kATileBytes), kLBO, kSBO);
        sDesc[(kc * kDigits + i) * 2 + 1] = tc::smem_desc(sb0 + (uint32_t)((kc * kDigits + i) * btile), kLBO, kSBO);
      }
  const int cbeg = half * KH;                    // this thread's first V column
  const int kc_mine = cbeg / kKChunk, k_mine = cbeg % kKChunk;
  uint32_t phase = 0, lphase = 0;

  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t r = tile * kTileRows + row;
    const bool live = r < a.n;
    const bool bulk = bulk_ok(tile);
    bool ok = true;
    if (bulk) {
      ok = wait_sleep(lbar, lphase);
      if (!ok) {
        wait_sleep(lbar, lphase);  // no copy left in flight
      }
      lphase ^= 1;
    }
    // ---- this thread's half of row r and its largest exponent
    double v[KH];
    int emax = 0;
#pragma unroll
    for (int c0 = 0; c0 < KH; c0 += BV) {
      if (live && cbeg + c0 < a.K) {
        if (bulk) {
          const double* src = sV + ((size_t)((cbeg + c0) / BV) * kTileRows + row) * BV;
#pragma unroll
          for (int p = 0; p < BV; ++p) v[c0 + p] = src[p];
        } else {
          const double* src = a.vblk[(cbeg + c0) / BV] + r * BV;   // scalar loads: any alignment
#pragma unroll
          for (int p = 0; p < BV; ++p) v[c0 + p] = src[p];
        }
      } else {
#pragma unroll
        for (int p = 0; p < BV; ++p) v[c0 + p] = 0.0;
      }
    }
#pragma unroll
    for (int c = 0; c < KH; ++c) emax = max(emax, exp_field(v[c]));
    sE[half * kTileRows + row] = emax;
    __syncthreads();  // every thread has its V values: the staging buffer takes the next tile
    if (tid == 0) {
      const int64_t nt = tile + gridDim.x;
      if (nt < ntiles && bulk_ok(nt)) issue(nt);
    }
    emax = max(sE[row], sE[kTileRows + row]);
    // ---- split into seven digits and write them to the A tiles
#pragma unroll
    for (int k8 = 0; k8 < KH; k8 += 8) {
      Sig8 s8;
      align8(v + k8, (uint32_t)emax << 20, s8);
      const int kk = k_mine + k8;   // column within the chunk
      const int kc = kc_mine + kk / kKChunk;
      unsigned char* dst = sA + (size_t)kc * kDigits * kATileBytes + tile_off(row, kk % kKChunk);
      digits8(s8, [&](int i, uint4 w) { *reinterpret_cast<uint4*>(dst + i * kATileBytes) = w; });
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    // ---- one thread issues the digit products: class g = i + j accumulates A_i B_j
    if (tid == 0) {
      tc::fence_after_sync();
      // descriptor of K-step ks = that of K-step 0 with the start address advanced by 2 core
      // matrices (256 bytes, 16 in the descriptor's address field)
      // digit i of A against the B digit tiles 0..6-i of the chunk stacked as one operand of
      // (7-i) NP rows: column block j of the product accumulates into class i + j
      for (int kc = 0; kc < nkc; ++kc)
#pragma unroll
        for (int i = 0; i < kDigits; ++i) {
          const uint64_t ad = sDesc[(kc * kDigits + i) * 2];
          const uint64_t bd = sDesc[(kc * kDigits) * 2 + 1];
          const uint32_t dt = tbase + (uint32_t)((kc * kClasses + i) * NP);
          const uint32_t id = tc::idesc_f16_f32(kTileRows, (kDigits - i) * NP);
#pragma unroll
          for (int ks = 0; ks < kKChunk / 16; ++ks)
            tc::mma_f16(dt, ad + (uint64_t)(ks * 2 * kLBO >> 4), bd + (uint64_t)(ks * 2 * kLBO >> 4), id,
                         (i > 0 || ks > 0) ? 1u : 0u);
        }
      tc::mma_commit(bar);
    }
    // ---- wait for the products (bounded), then read row `row`'s accumulators
    if (!wait_sleep(bar, phase)) {
      ok = false;
      wait_sleep(bar, phase);  // let the MMAs in flight finish before TMEM is reused
    }
    phase ^= 1;
    tc::fence_after_sync();
    const uint32_t lane_addr = tbase + ((uint32_t)((warp & 3) * 32) << 16);
    const int ebase = emax - 2108 + kAsmShift;
    for (int q0 = 4 * half; q0 < a.N; q0 += 8) {   // groups of 4 results, alternating halves
      uint32_t acc[KMAX / kKChunk][kClasses][4];
#pragma unroll
      for (int kc = 0; kc < KMAX / kKChunk; ++kc)
        if (kc < nkc)
#pragma unroll
          for (int g = 0; g < kClasses; ++g)
            tc::tmem_ld4(lane_addr + (uint32_t)((kc * kClasses + g) * NP + q0), acc[kc][g]);
      tc::tmem_ld_wait();
#pragma unroll
      for (int kc = 0; kc < KMAX / kKChunk; ++kc)
        if (kc < nkc)
#pragma unroll
          for (int g = 0; g < kClasses; ++g) tc::reg_after_wait(acc[kc][g]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = q0 + u;
        int64_t hi = 0, lo = 0;
#pragma unroll
        for (int kc = 0; kc < KMAX / kKChunk; ++kc)
          if (kc < nkc) {
            // 32 x 32 -> 64-bit multiply-adds by powers of two
            hi += (int64_t)acc_int(acc[kc][0][u], kDigitUnit) * 65536 + (int64_t)acc_int(acc[kc][1][u], kDigitUnit) * 256 +
                  (int64_t)acc_int(acc[kc][2][u], kDigitUnit);
            lo += (int64_t)acc_int(acc[kc][3][u], kDigitUnit) * 16777216 + (int64_t)acc_int(acc[kc][4][u], kDigitUnit) * 65536 +
                  (int64_t)acc_int(acc[kc][5][u], kDigitUnit) * 256 + (int64_t)acc_int(acc[kc][6][u], kDigitUnit);
          }
        if (live && q < a.N) {
          double y = 0.0;
          if (!ok) y = __longlong_as_double(0x7FF8000000000000ll);
          else if (emax > 0)
            y = scale_int((hi << (32 - kAsmShift)) + ((lo + (1 << (kAsmShift - 1))) >> kAsmShift), ebase + sF[q]);
          double* dst = a.oblk[q / BV] + r * BV + q % BV;
          if (add_out) y = fma(a.beta, *dst, y);
          *dst = y;
        }
      }
    }
    tc::fence_before_sync();
    __syncthreads();  // TMEM read, A tiles and row exponents free for the next tile
  }
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tbase, ncols);
}

// Shared-memory bytes of tc_combine_kernel for nkc K chunks and padded N.
static size_t tc_smem_bytes(int nkc, int NP) {
  const int kmax = nkc == 1 ? 32 : 64;
  return (size_t)nkc * kDigits * kATileBytes + (size_t)nkc * kDigits * NP * kKChunk * 2 +
         (size_t)kTileRows * kmax * 8 + 16 + 8 * 2 * kDigits * (kmax / kKChunk) * 2 + 8 + 4 * kMaxN +
         4 * 2 * kTileRows + 64;
}

// ---------------------------------------------------------------- pipelined form (K <= 32)
// The same product with the phases of consecutive tiles overlapped.  One persistent CTA per SM
// with four warp roles (numbers for K > 16; up to there warps 0-7, 24, 25 and 8-23, PipeRoles):
//   warps 0-15  split V rows into digits: a unit is 8 columns of one row, thread t takes unit
//               t = row + 128 cb (cb < ceil(K / 8)); units write the digit tiles of buffer t % 2;
//   warp 28     (one thread) issues the TMA copies of tile t's V rows into staging buffer t % 2;
//   warp 29     (one thread) issues tile t's MMAs into TMEM buffer t % 2 and owns the TMEM
//               allocation;
//   warps 16-27 read tile t's accumulators (TMEM lane quarter = warp % 4, three threads per row,
//               every third pair of results each), assemble and store them; with beta != 0 a
//               thread with at most two pairs (N <= 12: all of them) loads its rows of Out for
//               the next tiles while tile t is assembled.
// V staging, digit tiles and accumulators are double-buffered, so tile t + 1 is split while tile
// t's products run and its results are assembled.  Five mbarrier pairs hand each buffer on:
// vfull (TMA -> splitters), vempty (splitters -> TMA), afull (splitters -> MMA and
// epilogue: digits and row exponents written), mdone (tcgen05.commit -> splitters and
// epilogue: products complete, digit tiles free), tempty (epilogue -> MMA and splitters: TMEM
// and row exponents read).  The k-th use of a buffer waits for phase parity k & 1; a
// barrier cannot run two phases ahead of a waiter because every phase of it needs a phase the
// waiter itself completes first.  The splitters meet once per tile at a named barrier that
// also ORs their wait failures, so they leave the loop together.  Every wait is bounded; a
// wait that runs out marks the CTA aborted, the other roles stop at their next wait, the
// epilogue writes NaN to the rows of the tiles it has not finished, and the TMA copies and MMAs
// in flight are waited for (again bounded) before TMEM is freed.
// 2^20 rows, K = 32, N = 20 (436 MB): a call takes 182 us (194 with 8 splitting and 8 assembling warps,
// truncating 64-bit assembly and two barriers per tile).  The kernel alone: 173 us; 137 without the
// assembly, 97 without the split as well; 186 with 8 assembling warps, 187 with every other result
// normalised in integers instead of converted.
namespace {
// Warp roles: 16 splitting and 12 assembling warps, three threads per row of results.  Up to 16 columns of V
// (FEW) half of the splitting warps would have no unit and only meet at the barriers, and the results
// bind: 8 and 16 there, four threads per row (4.2 million rows, 8 columns into 8 340 -> 269 us, 16 into 8
// 356 -> 307, 16 into 32 902 -> 650 against 8 and 8 warps; 357, 380 and 801 with 16 and 12).
template <bool FEW>
struct PipeRoles {
  static constexpr int kSplitWarps = FEW ? 8 : 16, kEpiWarps = FEW ? 16 : 12;
  static constexpr int kEpiParts = kEpiWarps / 4;                 // epilogue threads per row
  static constexpr int kSplitThreads = kSplitWarps * 32;
  static constexpr int kProdWarp = kSplitWarps + kEpiWarps, kMmaWarp = kProdWarp + 1;
  static constexpr int kPipeThreads = (kMmaWarp + 1) * 32;
};

struct PipeBars {
  uint64_t vfull[2], vempty[2], afull[2], mdone[2], tempty[2];
};

// Shared-memory bytes of tc_combine_pipe_kernel for padded N.
constexpr size_t pipe_smem_bytes(int NP) {
  return (size_t)2 * kDigits * kATileBytes + (size_t)kDigits * NP * kKChunk * 2 +
         (size_t)2 * kTileRows * kKChunk * 8 + sizeof(PipeBars) + 8 + 4 * kMaxN + 4 * 10 * kTileRows + 64;
}
}  // namespace

// Bounded wait for one phase of a pipeline barrier, sleeping between polls; false when the CTA
// has aborted or the polls ran out, which also marks it aborted.  The warp form gives every
// lane the same answer.
__device__ __forceinline__ bool pipe_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  bool ok = tc::mbar_wait(bar, parity, 1);   // a completed phase returns at once
  for (uint32_t r = 0; r < kPipePolls && !ok; ++r) {
    ok = tc::mbar_wait_sleep(bar, parity, 1, kPipeSleepNs);
    if (!ok && *abort_flag) break;
  }
  if (!ok) *abort_flag = 1;
  return ok;
}
__device__ __forceinline__ bool pipe_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return __all_sync(0xffffffffu, pipe_wait(bar, parity, abort_flag));
}

// Named barrier `id` over `nthreads` threads that returns the OR of every thread's `p`.
__device__ __forceinline__ bool bar_or(int id, int nthreads, bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)p), "r"(id), "r"(nthreads)
      : "memory");
  return r != 0;
}

template <int BV, int NP, bool FEW>
__global__ void __launch_bounds__(PipeRoles<FEW>::kPipeThreads, 1) tc_combine_pipe_kernel(const TcArgs a) {
  using PR = PipeRoles<FEW>;
  constexpr int kSplitWarps = PR::kSplitWarps, kEpiWarps = PR::kEpiWarps, kEpiParts = PR::kEpiParts,
                kSplitThreads = PR::kSplitThreads, kProdWarp = PR::kProdWarp, kMmaWarp = PR::kMmaWarp,
                kPipeThreads = PR::kPipeThreads;
  constexpr uint32_t kBufCols = NP == 32 ? 256u : 128u;  // TMEM columns per buffer (7 NP used)
  constexpr size_t kBTile = (size_t)NP * kKChunk * 2;
  constexpr int kVBuf = kTileRows * kKChunk;              // doubles per V staging buffer
  constexpr int W = BV < 8 ? BV : 8;                      // columns of one block read per step
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sA = smem;                                        // [2][7] x 8 KB
  unsigned char* sB = sA + 2 * kDigits * kATileBytes;              // [7] x NP*64
  double* sV = reinterpret_cast<double*>(sB + kDigits * kBTile);   // [2][32 / BV][128][BV]
  PipeBars* bars = reinterpret_cast<PipeBars*>(sV + 2 * kVBuf);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  int* sF = reinterpret_cast<int*>(tslot + 2);                     // N column exponents of Y
  int* sE = sF + kMaxN;                                            // [2][128] row exponents
  int* sEp = sE + 2 * kTileRows;                                   // [2][4][128] unit exponents
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  {
    const int4* src = reinterpret_cast<const int4*>(a.bdig);
    int4* dst = reinterpret_cast<int4*>(sB);
    for (int e = tid; e < (int)(kDigits * kBTile / 16); e += kPipeThreads) dst[e] = src[e];
    for (int q = tid; q < a.N; q += kPipeThreads) sF[q] = a.fexp[q];
    // digit columns at or beyond K stay zero in both buffers
    int4* z = reinterpret_cast<int4*>(sA);
    for (int e = tid; e < 2 * kDigits * kATileBytes / 16; e += kPipeThreads) z[e] = make_int4(0, 0, 0, 0);
  }
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&bars->vfull[b], 1);
      tc::mbar_init(&bars->vempty[b], kSplitWarps);
      tc::mbar_init(&bars->afull[b], kSplitWarps);
      tc::mbar_init(&bars->mdone[b], 1);
      tc::mbar_init(&bars->tempty[b], kEpiWarps);
    }
    *abort_flag = 0;
    tc::mbar_fence_init();
  }
  if (warp == kMmaWarp) {
    tc::tmem_alloc(tslot, 2 * kBufCols);
    tc::tmem_relinquish();
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = *tslot;
  const int64_t ntiles = (a.n + kTileRows - 1) / kTileRows;
  const int64_t cnt = (int64_t)blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  auto tile_of = [&](int64_t it) { return (int64_t)blockIdx.x + it * gridDim.x; };
  // every tile but a ragged last one is a multiple of 16 bytes
  const int64_t nbulk = !a.bulk ? 0 : ((a.n - (ntiles - 1) * kTileRows) * BV * 8) % 16 == 0 ? ntiles : ntiles - 1;
  auto bulk_ok = [&](int64_t t) { return t < nbulk; };

  if (warp == kProdWarp) {
    // ---- TMA: V rows of tile `it` into staging buffer it % 2
    int64_t issued = 0;
    if (lane == 0) {
      const int nblk = a.K / BV;
      for (int64_t it = 0; it < cnt; ++it) {
        const int b = (int)(it & 1);
        const uint32_t k = (uint32_t)(it >> 1);
        if (k > 0 && !pipe_wait(&bars->vempty[b], (k - 1) & 1, abort_flag)) break;
        const int64_t r0 = tile_of(it) * kTileRows;
        if (bulk_ok(tile_of(it))) {
          const uint32_t bytes = (uint32_t)(min((int64_t)kTileRows, a.n - r0) * BV * 8);
          tc::mbar_arrive_expect_tx(&bars->vfull[b], bytes * (uint32_t)nblk);
          for (int j = 0; j < nblk; ++j)
            tc::bulk_g2s(sV + (size_t)b * kVBuf + (size_t)j * kTileRows * BV, a.vblk[j] + r0 * BV, bytes,
                         &bars->vfull[b]);
        } else {
          tc::mbar_arrive(&bars->vfull[b]);   // ragged or unaligned tile: splitters load V directly
        }
        issued = it + 1;
      }
      // copies in flight complete before the CTA exits (immediate unless the CTA aborted)
      for (int b = 0; b < 2; ++b) {
        const int64_t uses = (issued + 1 - b) / 2;
        if (uses > 0) wait_sleep(&bars->vfull[b], (uint32_t)((uses - 1) & 1));
      }
    }
  } else if (warp == kMmaWarp) {
    // ---- MMA issue: digit i of A against the B digit tiles 0..6-i stacked as one (7-i) NP-row
    // operand; the product's column block j lands on class i + j's accumulator (TMEM column
    // (i + j) NP of buffer it % 2)
    int64_t committed = 0;
    if (lane == 0) {
      const int ksteps = a.K <= 16 ? 1 : 2;   // K-steps of 16 holding non-zero digits
      const uint32_t sa0 = tc::smem_addr(sA), sb0 = tc::smem_addr(sB);
      const uint64_t bd = tc::smem_desc(sb0, kLBO, kSBO);
      for (int64_t it = 0; it < cnt; ++it) {
        const int b = (int)(it & 1);
        const uint32_t k = (uint32_t)(it >> 1);
        if (!pipe_wait(&bars->afull[b], k & 1, abort_flag)) break;
        if (k > 0 && !pipe_wait(&bars->tempty[b], (k - 1) & 1, abort_flag)) break;
        tc::fence_after_sync();
        const uint32_t dbase = tbase + (uint32_t)b * kBufCols;
#pragma unroll
        for (int i = 0; i < kDigits; ++i) {
          const uint64_t ad = tc::smem_desc(sa0 + (uint32_t)((b * kDigits + i) * kATileBytes), kLBO, kSBO);
          const uint32_t idesc = tc::idesc_f16_f32(kTileRows, (kDigits - i) * NP);
          for (int ks = 0; ks < ksteps; ++ks)
            tc::mma_f16(dbase + (uint32_t)(i * NP), ad + (uint64_t)(ks * 2 * kLBO >> 4),
                        bd + (uint64_t)(ks * 2 * kLBO >> 4), idesc, (i > 0 || ks > 0) ? 1u : 0u);
        }
        tc::mma_commit(&bars->mdone[b]);
        committed = it + 1;
      }
      for (int b = 0; b < 2; ++b) {
        const int64_t uses = (committed + 1 - b) / 2;
        if (uses > 0) wait_sleep(&bars->mdone[b], (uint32_t)((uses - 1) & 1));
      }
    }
  } else if (warp < kSplitWarps) {
    // ---- split: units of 8 columns of one row
    const int ncb = (a.K + 7) >> 3, row = tid & (kTileRows - 1), cb = tid >> 7;
    const bool unit = cb < ncb;
    const uint32_t doff = (uint32_t)tile_off(row, cb * 8);
    const double* sVu = sV + ((size_t)(cb * 8 / BV) * kTileRows + row) * BV + cb * 8 % BV;
    bool bad = false;
    for (int64_t it = 0; it < cnt; ++it) {
      const int b = (int)(it & 1);
      const uint32_t k = (uint32_t)(it >> 1);
      const int64_t tile = tile_of(it);
      int* sEb = sEp + b * 4 * kTileRows + row;
      const bool ok = pipe_wait_warp(&bars->vfull[b], k & 1, abort_flag);
      double v[8];
      if (unit) {
        const bool live = tile * kTileRows + row < a.n;
        const double* sv = sVu + b * kVBuf;
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = 0.0;
        if (live && bulk_ok(tile)) {
#pragma unroll
          for (int c0 = 0; c0 < 8; c0 += W)
            if (W == 8 || cb * 8 + c0 < a.K) {
              if constexpr (W % 2 == 0) {
#pragma unroll
                for (int p = 0; p < W; p += 2) {
                  const double2 x = *reinterpret_cast<const double2*>(sv + (c0 / BV) * kTileRows * BV + p);
                  v[c0 + p] = x.x;
                  v[c0 + p + 1] = x.y;
                }
              } else {
                v[c0] = sv[c0 * kTileRows];
              }
            }
        } else if (live) {
#pragma unroll
          for (int c0 = 0; c0 < 8; c0 += W) {
            const int c = cb * 8 + c0;
            if (c < a.K) {
              const double* src = a.vblk[c / BV] + (tile * kTileRows + row) * BV + c % BV;
#pragma unroll
              for (int p = 0; p < W; ++p) v[c0 + p] = __ldg(src + p);
            }
          }
        }
        sEb[cb * kTileRows] = (int)top_exp8(v);
      }
      if (bar_or(1, kSplitThreads, !ok || bad)) break;   // V read, unit exponents written
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->vempty[b]);
      int emax = 0;
      for (int c = 0; c < ncb; ++c) emax = max(emax, sEb[c * kTileRows]);
      // digit tiles and row exponents of this buffer are free once tile it - 2's products and
      // results are done
      if (k > 0) bad = !pipe_wait_warp(&bars->mdone[b], (k - 1) & 1, abort_flag) ||
                       !pipe_wait_warp(&bars->tempty[b], (k - 1) & 1, abort_flag);
      if (bad) continue;   // the splitters leave together at the next tile's barrier
      if (unit) {
        if (cb == 0) sE[b * kTileRows + row] = emax >> 20;
        Sig8 s8;
        align8(v, (uint32_t)emax, s8);
        unsigned char* dst = sA + (size_t)b * kDigits * kATileBytes + doff;
        digits8(s8, [&](int i, uint4 w) { *reinterpret_cast<uint4*>(dst + i * kATileBytes) = w; });
      }
      tc::fence_async_smem();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->afull[b]);
    }
  } else {
    // ---- epilogue: TMEM lane quarter warp % 4; the warps of a quarter take turns at groups of two
    // results (q0 = 2 part + kStep jj)
    const int quarter = warp & 3, part = (warp - kSplitWarps) >> 2;
    const int row = quarter * 32 + lane;
    const bool add_out = a.beta != 0.0;
    constexpr int kStep = 2 * kEpiParts;
    const int ngroups = a.N > 2 * part ? (a.N - 2 * part + kStep - 1) / kStep : 0;        // this thread's groups of two results
    // rows of Out loaded ahead of their tile: by a thread with one group (three threads a row: N <= 6) two
    // tiles ahead into slot it % 2, with two groups (N <= 12) one tile ahead into slot = group
    const int pf = !add_out ? 0 : ngroups <= 1 ? 2 : ngroups == 2 ? 1 : 0;
    double opf[2][2];
    auto load_grp = [&](int64_t it, int jj, int slot) {
      const int64_t r = tile_of(it) * kTileRows + row;
      const int q0 = 2 * part + kStep * jj;
      if (r >= a.n || q0 >= a.N) return;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int q = q0 + u;
        const double x = q < a.N ? a.oblk[q / BV][r * BV + q % BV] : 0.0;
        if (slot == 0) opf[0][u] = x;
        else opf[1][u] = x;
      }
    };
    if (pf == 2) {
      if (cnt > 0) load_grp(0, 0, 0);
      if (cnt > 1) load_grp(1, 0, 1);
    } else if (pf == 1 && cnt > 0) {
      load_grp(0, 0, 0);
      load_grp(0, 1, 1);
    }
    int64_t it = 0;
    for (; it < cnt; ++it) {
      const int b = (int)(it & 1);
      const uint32_t k = (uint32_t)(it >> 1);
      if (!pipe_wait_warp(&bars->afull[b], k & 1, abort_flag)) break;
      if (!pipe_wait_warp(&bars->mdone[b], k & 1, abort_flag)) break;
      tc::fence_after_sync();
      const int64_t r = tile_of(it) * kTileRows + row;
      const bool live = r < a.n;
      const int emax = sE[b * kTileRows + row];
      const int ebase = emax - 2108 + kAsmShift;
      const uint32_t lane_addr = tbase + ((uint32_t)(quarter * 32) << 16) + (uint32_t)b * kBufCols;
      // the accumulators of group jj + 1 are loaded while group jj is assembled
      uint32_t nxt[kClasses][2];
      if (ngroups > 0) {
#pragma unroll
        for (int g = 0; g < kClasses; ++g) tc::tmem_ld2(lane_addr + (uint32_t)(g * NP + 2 * part), nxt[g]);
      }
      for (int jj = 0; jj < ngroups; ++jj) {
        const int q0 = 2 * part + kStep * jj;
        tc::tmem_ld_wait();
        uint32_t acc[kClasses][2];
#pragma unroll
        for (int g = 0; g < kClasses; ++g) {
          tc::reg_after_wait(nxt[g]);
          acc[g][0] = nxt[g][0];
          acc[g][1] = nxt[g][1];
        }
        if (jj + 1 < ngroups) {
#pragma unroll
          for (int g = 0; g < kClasses; ++g) tc::tmem_ld2(lane_addr + (uint32_t)(g * NP + q0 + kStep), nxt[g]);
        }
        if (jj == ngroups - 1) {
          // TMEM buffer and row exponent read: the buffer goes back to the MMA issuer
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&bars->tempty[b]);
        }
        double y[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t d[kClasses] = {acc[0][u], acc[1][u], acc[2][u], acc[3][u], acc[4][u], acc[5][u], acc[6][u]};
          const double x = scale_int(sum7(d, kDigitUnit, 8), ebase + sF[min(q0 + u, kMaxN - 1)]);
          y[u] = emax > 0 ? x : 0.0;
        }
        if (live) {
          if (add_out) {
            if (pf != 0) {
              const bool s1 = pf == 2 ? (it & 1) != 0 : jj != 0;
#pragma unroll
              for (int u = 0; u < 2; ++u) y[u] = fma(a.beta, s1 ? opf[1][u] : opf[0][u], y[u]);
            } else {
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int q = q0 + u;
                if (q < a.N) y[u] = fma(a.beta, a.oblk[q / BV][r * BV + q % BV], y[u]);
              }
            }
          }
          if (BV >= 2 && q0 + 2 <= a.N && a.ovec) {
            *reinterpret_cast<double2*>(a.oblk[q0 / BV] + r * BV + q0 % BV) = make_double2(y[0], y[1]);
          } else {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int q = q0 + u;
              if (q < a.N) a.oblk[q / BV][r * BV + q % BV] = y[u];
            }
          }
        }
      }
      if (ngroups == 0) {
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bars->tempty[b]);
      }
      if (pf == 2 && it + 2 < cnt) load_grp(it + 2, 0, (int)(it & 1));
      if (pf == 1 && it + 1 < cnt) {
        load_grp(it + 1, 0, 0);
        load_grp(it + 1, 1, 1);
      }
    }
    // after an abort: the rows of every tile not finished read NaN
    for (; it < cnt; ++it) {
      const int64_t r = tile_of(it) * kTileRows + row;
      if (r < a.n)
        for (int jj = 0; jj < ngroups; ++jj)
          for (int q = 2 * part + kStep * jj; q < min(a.N, 2 * part + kStep * jj + 2); ++q)
            a.oblk[q / BV][r * BV + q % BV] = __longlong_as_double(0x7FF8000000000000ll);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == kMmaWarp) tc::tmem_dealloc(tbase, 2 * kBufCols);
}

template <int BV, int NP, bool FEW>
static int launch_tc_combine_pipe_np(const TcArgs& a, cudaStream_t s) {
  static KernelSetup ks;
  const void* fn = reinterpret_cast<const void*>(tc_combine_pipe_kernel<BV, NP, FEW>);
  constexpr size_t smem = pipe_smem_bytes(NP);
  FE_TRY(kernel_configure(ks, fn, (int)smem));
  const int64_t ntiles = ceil_div(a.n, kTileRows);
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)num_sms()));
  tc_combine_pipe_kernel<BV, NP, FEW><<<(unsigned)grid, PipeRoles<FEW>::kPipeThreads, smem, s>>>(a);
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

template <int BV>
static int launch_tc_combine_pipe(const TcArgs& a, cudaStream_t s) {
  if (a.K <= 16) {
    if (a.NP == 16) return launch_tc_combine_pipe_np<BV, 16, true>(a, s);
    return launch_tc_combine_pipe_np<BV, 32, true>(a, s);
  }
  if (a.NP == 16) return launch_tc_combine_pipe_np<BV, 16, false>(a, s);
  return launch_tc_combine_pipe_np<BV, 32, false>(a, s);
}

bool tc_combine_supported(const BlockSet& V, const BlockSet& Out, fe_dtype dt) {
  const int K = V.nv * V.bv, N = Out.nv * Out.bv;
  return dt == FE_F64 && V.bv == Out.bv && V.ld == V.bv && Out.ld == Out.bv && K >= 1 && K <= kMaxK &&
         N >= 1 && N <= kMaxN && V.bv >= 1 && V.bv <= 16;
}

template <int BV>
static int launch_tc_combine(const TcArgs& a, size_t smem, bool two_per_sm, cudaStream_t s) {
  static KernelSetup ks;
  const void* fn = reinterpret_cast<const void*>(tc_combine_kernel<BV>);
  FE_TRY(kernel_configure(ks, fn, 227 * 1024));
  const int64_t ntiles = ceil_div(a.n, kTileRows);
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)(two_per_sm ? 2 : 1) * num_sms()));
  tc_combine_kernel<BV><<<(unsigned)grid, kThreads, smem, s>>>(a);
  count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// Out = V Y on the tensor cores (FP64 blocks; see tc_combine_supported for the shapes).
int tc_combine(const BlockSet& V, int64_t n, const double* Y, int ldy, const BlockSet& Out,
               cudaStream_t s, double alpha, double beta) {
  FE_ARG(tc_combine_supported(V, Out, FE_F64), "tc_combine: unsupported shape");
  TcArgs a;
  memset(&a, 0, sizeof(a));
  const int BV = V.bv;
  a.n = n;
  a.K = V.nv * BV;
  a.N = Out.nv * BV;
  a.NP = a.N <= 16 ? 16 : 32;
  a.nkc = (int)ceil_div(a.K, kKChunk);
  a.beta = beta;
  a.bulk = 1;
  for (int j = 0; j < V.nv; ++j) {
    a.vblk[j] = static_cast<const double*>(V.blk[j]);
    if (reinterpret_cast<uintptr_t>(V.blk[j]) % 16) a.bulk = 0;
  }
  a.ovec = 1;
  for (int o = 0; o < Out.nv; ++o) {
    a.oblk[o] = const_cast<double*>(static_cast<const double*>(Out.blk[o]));
    if (reinterpret_cast<uintptr_t>(Out.blk[o]) % 16) a.ovec = 0;
  }
  // scratch: B digit tiles, column exponents
  const size_t bbytes = (size_t)a.nkc * kDigits * a.NP * kKChunk * 2;
  double* scr = small_scratch(17, bbytes / 8 + kMaxN);
  if (!scr) return FE_ERR_OOM;
  a.bdig = reinterpret_cast<const uint16_t*>(scr);
  a.fexp = reinterpret_cast<const int*>(scr + bbytes / 8);
  tc_prep_y_kernel<<<1, kPrepThreads, 0, s>>>(Y, ldy, alpha, a.K, a.N, a.NP, a.nkc, const_cast<uint16_t*>(a.bdig),
                                     const_cast<int*>(a.fexp));
  count_launch();
  FE_CUDA(cudaGetLastError());
  if (a.nkc == 1) {
    switch (BV) {
      case 1: return launch_tc_combine_pipe<1>(a, s);
      case 2: return launch_tc_combine_pipe<2>(a, s);
      case 4: return launch_tc_combine_pipe<4>(a, s);
      case 8: return launch_tc_combine_pipe<8>(a, s);
      case 16: return launch_tc_combine_pipe<16>(a, s);
    }
  }
  // two CTAs per SM when their TMEM (256 columns each) fits; the shared-memory request keeps a
  // third CTA off the SM, so no CTA waits in tcgen05.alloc
  const bool two = a.nkc * kClasses * a.NP <= 256;
  const size_t smem = std::max(tc_smem_bytes(a.nkc, a.NP), two ? (size_t)100 * 1024 : (size_t)120 * 1024);
  switch (BV) {
    case 1: return launch_tc_combine<1>(a, smem, two, s);
    case 2: return launch_tc_combine<2>(a, smem, two, s);
    case 4: return launch_tc_combine<4>(a, smem, two, s);
    case 8: return launch_tc_combine<8>(a, smem, two, s);
    case 16: return launch_tc_combine<16>(a, smem, two, s);
  }
  return set_error(FE_ERR_INVALID, "tc_combine: block width %d", BV);
}


// ---------------------------------------------------------------- Gram V^T W (op3)
// G = alpha V^T W for FP64 blocks on the tensor cores (Table 1 "op3", MvTransMv), the same
// digit splitting as above with the roles of rows and columns exchanged: the contraction runs
// over the rows, so every column of V and of W is scaled by its largest exponent within each
// 112-row tile.  Per tile the MMA multiplies ALL digit slices at once: A holds the digit rows
// (i, c) of V^T (7 * KV <= 252 rows, two 128-row M tiles), B the digit rows (j, q) of W^T
// (7 * bw rows), K = the tile's 112 rows; every accumulator D[(i, c)][(j, q)] sums 112
// products below 2^16 and is exact.  TMEM lane (i, c) then forms T_i = sum_j D 2^(8 (6 - j))
// for each q in 64-bit integers (T_i / 2^12, rounded); the seven slices i of each output are added as
// sum_i T_i 2^(-8 i), rounded at each step to T_0's unit, and the sum, scaled by the tile's column
// exponents, is rounded once to FP64 and added to the CTA's accumulator of G; the CTAs' partial Gram
// matrices are added in a fixed order.
// Error per tile: 2^-50 * 112 * max|V[., c]| * max|W[., q]| over the tile's rows, plus the FP64
// roundings of the sums over tiles and CTAs.
namespace {
constexpr int kGramMaxKV = 36;                       // 7 * 36 = 252 digit rows of V^T
constexpr int kGramMaxBW = 8;                        // 7 * 8 = 56 digit rows of W^T
// Rows per tile (MMA K = 7 x 16): two digit buffers of 112 rows leave room for two staging buffers at
// 36 + 4 columns.  3000017 x (36 + 4), the kernel alone: 303 us (404 with 12 splitting and 4 epilogue
// warps, 128-bit sums and 128 rows); 128 rows (one staging buffer, whose load latency shows)
// 330, 96 rows (three) 309, 80 rows 343; one digit buffer and three staging buffers of 128 rows 426.
constexpr int kGramRows = 112;
constexpr uint32_t kGSBO = (kGramRows / 8) * kCoreBytes;  // between 8-row groups
constexpr int kGATile = 128 * kGramRows * 2;         // one 128-row M tile of V^T digits: 28 KB

struct TcGramArgs {
  const double* vblk[kMaxBlocks];
  int bv, KV;            // V: KV / bv blocks of n x bv (ld bv)
  const double* W;
  int bw, NP;            // W: n x bw (ld bw); NP = 7 bw padded to the MMA's N
  int nmt;               // M tiles of V^T digits (1 or 2)
  int64_t n;
  double* partial;       // [gridDim.x][KV * bw]
  int bulk;              // 1: V blocks and W 16-byte aligned (TMA bulk copies allowed)
  int nxb;               // staging buffers of the pipelined kernel (1 or 2)
};
}  // namespace

// ---------------------------------------------------------------- pipelined Gram
// The same Gram with its phases overlapped, in the warp roles of the pipelined block product:
//   warps 0-19  split: a unit is 8 rows (group g) of column c of [V W], thread t takes unit
//               t = g (KV + bw) + c; the column exponents are shared-memory maxima over the groups;
//               digits go to the A / B tiles of buffer t % 2;
//   warp 28     (one thread) TMA copies of the tile's rows into one of up to four staging buffers;
//   warp 29     (one thread) the nmt x 7 MMAs of a tile into TMEM buffer t % 2;
//   warps 20-27 (TMEM lane quarter = warp % 4, two warps each) for every lane (i, c) and column q:
//               T_i into shared memory; after a barrier of these warps each output (c, q) adds its
//               seven slices and adds the tile's result to the thread's FP64 partial of G.
// Barriers: xfull / xempty (staging), afull / mdone / tempty per buffer, as in the block
// product; the splitters meet twice per tile and the epilogue warps twice, at named barriers
// that OR their wait failures.
namespace {
constexpr int kGSplitWarps = 20, kGEpiWarps = 8;    // 20 x 32 >= (36 + 8) columns x 14 groups
constexpr int kGSplitThreads = kGSplitWarps * 32;
constexpr int kGEpiThreads = kGEpiWarps * 32;
constexpr int kGOuts = 2;            // outputs per epilogue thread
constexpr int kGMaxStages = 4;       // staging buffers
constexpr int kGProdWarp = kGSplitWarps + kGEpiWarps, kGMmaWarp = kGProdWarp + 1;
constexpr int kGPipeThreads = (kGMmaWarp + 1) * 32;

struct GramBars {
  uint64_t xfull[kGMaxStages], xempty[kGMaxStages], afull[2], mdone[2], tempty[2];
};
constexpr int kGramMaxCols = kGramMaxKV + kGramMaxBW;

struct GramPipeLayout {
  size_t a, b, x, xbuf, t, e, bars, total;
  int nxb;   // staging buffers: as many as fit, at most kGMaxStages
};
__host__ __device__ inline GramPipeLayout gram_pipe_layout(int nmt, int NP, int nvb, int bv, int bw, int KV,
                                                          int nxb) {
  GramPipeLayout L;
  L.nxb = nxb;
  L.a = 0;
  L.b = L.a + (size_t)2 * nmt * kGATile;
  L.x = L.b + (size_t)2 * NP * kGramRows * 2;
  const size_t xd = (size_t)nvb * (kGramRows * bv + 4) + (size_t)kGramRows * bw + 4;
  L.xbuf = (xd * 8 + 15) & ~(size_t)15;
  L.t = L.x + (size_t)nxb * L.xbuf;
  L.e = L.t + (size_t)7 * KV * bw * 8;
  L.bars = (L.e + (size_t)4 * kGramMaxCols * 4 + 15) & ~(size_t)15;
  L.total = L.bars + sizeof(GramBars) + 16;
  return L;
}
}  // namespace

template <int BW>
__global__ void __launch_bounds__(kGPipeThreads, 1) tc_gram_pipe_kernel(const TcGramArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr int bw = BW;
  constexpr int NP = (7 * BW + 15) / 16 * 16;
  const int KV = a.KV, nmt = a.nmt, bv = a.bv;
  const int ncol = KV + bw;
  const int nvb = KV / bv;
  const int XS = kGramRows * bv + 4;           // doubles per staged V block (padded)
  const GramPipeLayout L = gram_pipe_layout(nmt, NP, nvb, bv, bw, KV, a.nxb);
  const int nxb = a.nxb;
  unsigned char* sA = smem + L.a;              // [2][nmt] x 28 KB
  unsigned char* sB = smem + L.b;              // [2] x NP x 112 FP16
  double* sX = reinterpret_cast<double*>(smem + L.x);
  int64_t* sT = reinterpret_cast<int64_t*>(smem + L.t);   // [bw][7][KV] slice integers
  int* sEx = reinterpret_cast<int*>(smem + L.e);          // [2][ncol] column exponents by buffer
  int* sExw = sEx + 2 * kGramMaxCols;                      // [2][ncol] maxima being formed
  GramBars* bars = reinterpret_cast<GramBars*>(smem + L.bars);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bufcols = nmt * NP <= 64 ? 64u : 128u;

  {
    int4* z = reinterpret_cast<int4*>(smem);
    for (int e = tid; e < (int)(L.x / 16); e += kGPipeThreads) z[e] = make_int4(0, 0, 0, 0);
  }
  if (tid == 0) {
    for (int b = 0; b < nxb; ++b) {
      tc::mbar_init(&bars->xfull[b], 1);
      tc::mbar_init(&bars->xempty[b], kGSplitWarps);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&bars->afull[b], kGSplitWarps);
      tc::mbar_init(&bars->mdone[b], 1);
      tc::mbar_init(&bars->tempty[b], kGEpiWarps);
    }
    *abort_flag = 0;
    tc::mbar_fence_init();
  }
  if (warp == kGMmaWarp) {
    tc::tmem_alloc(tslot, 2 * bufcols);
    tc::tmem_relinquish();
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = *tslot;
  const int64_t ntiles = (a.n + kGramRows - 1) / kGramRows;
  const int cnt = (int64_t)blockIdx.x < ntiles ? (int)((ntiles - 1 - blockIdx.x) / gridDim.x + 1) : 0;
  auto tile_of = [&](int it) { return (int64_t)blockIdx.x + (int64_t)it * gridDim.x; };
  // this CTA's last tile is the matrix's last one: its rows past the end read zero, and it is loaded
  // without TMA unless its bytes are a multiple of 16
  const bool own_last = cnt > 0 && tile_of(cnt - 1) == ntiles - 1;
  const int last = (int)(a.n - (ntiles - 1) * kGramRows);
  const int nbulk = !a.bulk ? 0 : own_last && ((last * bv) % 2 != 0 || (last * bw) % 2 != 0) ? cnt - 1 : cnt;

  if (warp == kGProdWarp) {
    int issued = 0;
    if (lane == 0) {
      int xb = 0;
      uint32_t xk = 0;   // uses of each buffer so far
      for (int it = 0; it < cnt; ++it) {
        if (xk > 0 && !pipe_wait(&bars->xempty[xb], (xk - 1) & 1, abort_flag)) break;
        const int64_t t = tile_of(it), r0 = t * kGramRows;
        double* sXb = sX + (size_t)xb * (L.xbuf / 8);
        if (it < nbulk) {
          const int64_t rows = min((int64_t)kGramRows, a.n - r0);
          const uint32_t vb = (uint32_t)(rows * bv * 8), wb = (uint32_t)(rows * bw * 8);
          tc::mbar_arrive_expect_tx(&bars->xfull[xb], vb * (uint32_t)nvb + wb);
          for (int j = 0; j < nvb; ++j) tc::bulk_g2s(sXb + (size_t)j * XS, a.vblk[j] + r0 * bv, vb, &bars->xfull[xb]);
          tc::bulk_g2s(sXb + (size_t)nvb * XS, a.W + r0 * bw, wb, &bars->xfull[xb]);
        } else {
          tc::mbar_arrive(&bars->xfull[xb]);   // ragged or unaligned tile: splitters load directly
        }
        issued = it + 1;
        if (++xb == nxb) {
          xb = 0;
          ++xk;
        }
      }
      for (xb = 0; xb < nxb; ++xb) {
        const int uses = (issued + nxb - 1 - xb) / nxb;
        if (uses > 0) wait_sleep(&bars->xfull[xb], (uint32_t)((uses - 1) & 1));
      }
    }
  } else if (warp == kGMmaWarp) {
    int committed = 0;
    if (lane == 0) {
      const uint32_t idesc = tc::idesc_f16_f32(128, NP);
      const uint32_t sa0 = tc::smem_addr(sA), sb0 = tc::smem_addr(sB);
      for (int it = 0; it < cnt; ++it) {
        const int b = (int)(it & 1);
        const uint32_t k = (uint32_t)(it >> 1);
        if (!pipe_wait(&bars->afull[b], k & 1, abort_flag)) break;
        if (k > 0 && !pipe_wait(&bars->tempty[b], (k - 1) & 1, abort_flag)) break;
        tc::fence_after_sync();
        for (int mt = 0; mt < nmt; ++mt)
#pragma unroll
          for (int ks = 0; ks < kGramRows / 16; ++ks) {
            const uint64_t ad = tc::smem_desc(sa0 + (uint32_t)((b * nmt + mt) * kGATile + ks * 2 * kCoreBytes),
                                              kCoreBytes, kGSBO);
            const uint64_t bd = tc::smem_desc(sb0 + (uint32_t)(b * NP * kGramRows * 2 + ks * 2 * kCoreBytes),
                                              kCoreBytes, kGSBO);
            tc::mma_f16(tbase + (uint32_t)b * bufcols + (uint32_t)(mt * NP), ad, bd, idesc, ks > 0 ? 1u : 0u);
          }
        tc::mma_commit(&bars->mdone[b]);
        committed = it + 1;
      }
      for (int b = 0; b < 2; ++b) {
        const int uses = (committed + 1 - b) / 2;
        if (uses > 0) wait_sleep(&bars->mdone[b], (uint32_t)((uses - 1) & 1));
      }
    }
  } else if (warp < kGSplitWarps) {
    // ---- split: unit (column c, 8-row group g) of thread u = g ncol + c, so that a warp's lanes read
    // and write neighbouring columns (no shared-memory bank conflicts); the column exponents
    // are maxima over the groups through shared-memory atomics (double-buffered by tile)
    const bool unit = tid < ncol * (kGramRows / 8);
    const int c = unit ? tid % ncol : 0, g = unit ? tid / ncol : 0;
    const bool isv = c < KV;
    const int str = isv ? bv : bw;
    const int soff = (isv ? (c / bv) * XS + c % bv : nvb * XS + (c - KV)) + g * 8 * str;
    uint32_t doff[kDigits];   // where the unit's digits go
#pragma unroll
    for (int i = 0; i < kDigits; ++i) {
      const int m = isv ? i * KV + c : i * bw + (c - KV);
      doff[i] = (uint32_t)((isv ? L.a + (size_t)(m >> 7) * kGATile + ((m & 127) >> 3) * kGSBO
                                : L.b + (size_t)(m >> 3) * kGSBO) + g * kCoreBytes + (m & 7) * 16);
    }
    const uint32_t dbuf = isv ? (uint32_t)(nmt * kGATile) : (uint32_t)(NP * kGramRows * 2);
    for (int e = tid; e < 2 * kGramMaxCols; e += kGSplitThreads) sExw[e] = 0;
    bar_or(1, kGSplitThreads, false);
    int xb = 0;               // staging buffer
    uint32_t xph = 0;
    for (int it = 0; it < cnt; ++it) {
      const int b = (int)(it & 1);
      const uint32_t k = (uint32_t)(it >> 1);
      int* exw = sExw + b * kGramMaxCols;
      const bool ok = pipe_wait_warp(&bars->xfull[xb], xph, abort_flag);
      double x[8];
      if (unit) {
        if (it < nbulk) {
          const double* scol = sX + xb * (int)(L.xbuf / 8) + soff;   // in the staging buffer in any case
#pragma unroll
          for (int tt = 0; tt < 8; ++tt) x[tt] = scol[tt * str];
        } else {
          const int64_t r = tile_of(it) * kGramRows + g * 8;
          const double* src = (isv ? a.vblk[c / bv] + c % bv : a.W + (c - KV)) + r * str;
#pragma unroll
          for (int tt = 0; tt < 8; ++tt) x[tt] = r + tt < a.n ? __ldg(src + tt * str) : 0.0;
        }
        if (own_last && it == cnt - 1) {
#pragma unroll
          for (int tt = 0; tt < 8; ++tt) x[tt] = g * 8 + tt < last ? x[tt] : 0.0;
        }
        const uint32_t e = top_exp8(x);
        if (e > 0) atomicMax(exw + c, (int)e);
      }
      if (bar_or(1, kGSplitThreads, !ok)) break;   // staging buffer read, exponent maxima formed
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->xempty[xb]);
      if (++xb == nxb) {
        xb = 0;
        xph ^= 1u;
      }
      const uint32_t emax = (uint32_t)exw[c];
      // the other buffer of maxima (read by everyone before the previous tile's second barrier)
      // starts the next tile at zero
      if (tid < ncol) sExw[(b ^ 1) * kGramMaxCols + tid] = 0;
      bool ok2 = true;
      if (k > 0) ok2 = pipe_wait_warp(&bars->mdone[b], (k - 1) & 1, abort_flag) &&
                       pipe_wait_warp(&bars->tempty[b], (k - 1) & 1, abort_flag);
      if (bar_or(1, kGSplitThreads, !ok2)) break;  // digit tiles and exponents of buffer b free
      if (unit) {
        if (g == 0) sEx[b * kGramMaxCols + c] = (int)(emax >> 20);
        Sig8 s8;
        align8(x, emax, s8);
        unsigned char* dst = smem + (uint32_t)b * dbuf;
        digits8(s8, [&](int i, uint4 w) { *reinterpret_cast<uint4*>(dst + doff[i]) = w; });
      }
      tc::fence_async_smem();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->afull[b]);
    }
  } else if (warp < kGSplitWarps + kGEpiWarps) {
    // ---- epilogue: TMEM lane quarter warp % 4 of each M tile
    const int quarter = warp & 3, half = (warp - kGSplitWarps) >> 2, et = tid - kGSplitThreads;
    const int nout = KV * bw;
    double acc[kGOuts] = {};   // outputs et, et + 256 (nout <= 288)
    for (int it = 0; it < cnt; ++it) {
      const int b = (int)(it & 1);
      const uint32_t k = (uint32_t)(it >> 1);
      const bool ok = pipe_wait_warp(&bars->afull[b], k & 1, abort_flag) &&
                      pipe_wait_warp(&bars->mdone[b], k & 1, abort_flag);
      if (bar_or(2, kGEpiThreads, !ok)) break;
      tc::fence_after_sync();
      // this thread's output scales, read before the buffer's exponents are handed back
      const int* ex = sEx + b * kGramMaxCols;
      int scl[kGOuts];
#pragma unroll
      for (int kk = 0; kk < kGOuts; ++kk) {
        const int o = et + kGEpiThreads * kk;
        scl[kk] = 0;
        if (o < nout) {
          const int ec = ex[o / bw], fq = ex[KV + o % bw];
          scl[kk] = ec > 0 && fq > 0 ? ec + fq : 0;
        }
      }
      for (int mt = 0; mt < nmt; ++mt) {
        const int m = mt * 128 + quarter * 32 + lane;
        const uint32_t laddr = tbase + ((uint32_t)(quarter * 32) << 16) + (uint32_t)b * bufcols + (uint32_t)(mt * NP);
#pragma unroll
        for (int q = 0; q < bw; ++q) {
          if (((mt * bw + q) & 1) != half) continue;
          uint32_t d[kDigits];
#pragma unroll
          for (int jd = 0; jd < kDigits; ++jd) d[jd] = tc::tmem_ld1(laddr + (uint32_t)(jd * bw + q));
          tc::tmem_ld_wait();
#pragma unroll
          for (int jd = 0; jd < kDigits; ++jd) tc::reg_after_wait(d[jd]);
          if (m < 7 * KV) {
            // T_i / 2^12 of slice i = m / KV, column c = m % KV; slices i > 0 hold 128 more, the
            // rounding of their division by 2^8
            sT[q * 7 * KV + m] = sum7(d, kDigitUnit * kDigitUnit, m < KV ? 8 : 8 + 16 * 128);
          }
        }
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->tempty[b]);
      bar_or(2, kGEpiThreads, false);   // slice integers written
#pragma unroll
      for (int kk = 0; kk < kGOuts; ++kk) {
        const int o = et + kGEpiThreads * kk;
        if (o < nout) {
          const int c = o / bw, q = o % bw;
          // sum_i T_i 2^(-8 i), rounded at each division
          const int64_t* tq = sT + q * 7 * KV + c;
          int64_t sum = tq[6 * KV];
#pragma unroll
          for (int i = kDigits - 2; i >= 0; --i) sum = tq[i * KV] + (sum >> 8);
          if (scl[kk] > 0) acc[kk] += scale_int(sum, scl[kk] - 2108 + kAsmShift);
        }
      }
      bar_or(2, kGEpiThreads, false);   // slice integers read: the next tile may overwrite them
    }
#pragma unroll
    for (int kk = 0; kk < kGOuts; ++kk) {
      const int o = et + kGEpiThreads * kk;
      if (o < nout) a.partial[(int64_t)blockIdx.x * nout + o] = *abort_flag ? __longlong_as_double(0x7FF8000000000000ll) : acc[kk];
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == kGMmaWarp) tc::tmem_dealloc(tbase, 2 * bufcols);
}

bool tc_gram_supported(const BlockSet& V, int bw, int ldw, fe_dtype dt) {
  const int KV = V.nv * V.bv;
  return dt == FE_F64 && V.ld == V.bv && ldw == bw && KV >= 1 && KV <= kGramMaxKV &&
         (bw == 1 || bw == 2 || bw == 4 || bw == 8) && V.bv >= 1;
}

int tc_gram(const BlockSet& V, int64_t n, const double* W, int bw, double alpha, double* G,
            cudaStream_t s) {
  FE_ARG(tc_gram_supported(V, bw, bw, FE_F64), "tc_gram: unsupported shape");
  TcGramArgs a;
  memset(&a, 0, sizeof(a));
  a.bv = V.bv;
  a.KV = V.nv * V.bv;
  for (int j = 0; j < V.nv; ++j) a.vblk[j] = static_cast<const double*>(V.blk[j]);
  a.W = W;
  a.bw = bw;
  a.bulk = reinterpret_cast<uintptr_t>(W) % 16 == 0;
  for (int j = 0; j < V.nv; ++j)
    if (reinterpret_cast<uintptr_t>(V.blk[j]) % 16) a.bulk = 0;
  a.NP = (int)ceil_div(7 * bw, 16) * 16;
  a.nmt = (int)ceil_div(7 * a.KV, 128);
  a.n = n;
  GramPipeLayout L;
  for (int nxb = kGMaxStages; nxb > 0; --nxb) {
    L = gram_pipe_layout(a.nmt, a.NP, a.KV / a.bv, a.bv, bw, a.KV, nxb);
    if (L.total <= 227 * 1024) break;
  }
  a.nxb = L.nxb;
  FE_ARG(L.total <= 227 * 1024 && a.KV * bw <= kGOuts * kGEpiThreads, "tc_gram: shape too large");
  static KernelSetup kp[4];
  const int bj = bw == 1 ? 0 : bw == 2 ? 1 : bw == 4 ? 2 : 3;
  const void* fp = bw == 1 ? reinterpret_cast<const void*>(tc_gram_pipe_kernel<1>)
                 : bw == 2 ? reinterpret_cast<const void*>(tc_gram_pipe_kernel<2>)
                 : bw == 4 ? reinterpret_cast<const void*>(tc_gram_pipe_kernel<4>)
                           : reinterpret_cast<const void*>(tc_gram_pipe_kernel<8>);
  FE_TRY(kernel_configure(kp[bj], fp, 227 * 1024));
  const int64_t nt = ceil_div(n, kGramRows);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(nt, (int64_t)num_sms()));
  const int nout = a.KV * bw;
  double* scr = small_scratch(18, (size_t)grid * nout);
  if (!scr) return FE_ERR_OOM;
  a.partial = scr;
  switch (bw) {
    case 1: tc_gram_pipe_kernel<1><<<grid, kGPipeThreads, L.total, s>>>(a); break;
    case 2: tc_gram_pipe_kernel<2><<<grid, kGPipeThreads, L.total, s>>>(a); break;
    case 4: tc_gram_pipe_kernel<4><<<grid, kGPipeThreads, L.total, s>>>(a); break;
    default: tc_gram_pipe_kernel<8><<<grid, kGPipeThreads, L.total, s>>>(a); break;
  }
  count_launch();
  FE_CUDA(cudaGetLastError());
  return gram_reduce(a.partial, grid, nout, alpha, G, s);
}

}  // namespace fe
