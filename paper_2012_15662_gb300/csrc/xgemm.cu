// FP64 matrix products on the BF16 tensor cores.
//
// This part issues FP64 at two lanes a clock per SM (1.25 TFLOP/s), 1/1500 of its BF16
// tensor rate, so a product that has to be as good as an FP64 one is taken from digit
// planes: every row of A and every column of B as a power-of-two exponent and seven
// balanced base-512 digits of a 62-bit integer,
//   x = 2^(e - 62) X,  X = d0 2^54 + d1 2^45 + ... + d6,  |X| < 2^61,
//   d0 in [-128, 128], d1..d6 in [-256, 255],
// each digit exact in BF16 (eight significant bits and a sign hold every integer to 256).  The
// 34 digit-pair products with t + u <= 7 go to eight FP32 accumulators g = t + u, which are read
// out after every K chunk of 128 elements and added in two int64 per output.  A K element adds at
// most 2^14, 2^16, 2^17, 3 2^16, 2^18 to groups 0..4, so a chunk's sums of groups 0..2 are
// integers of at most 2^24 and exact.  A sum of a later group is exact too unless it passes 2^24,
// for which the digits of both rows have to stay at two thirds (group 3) or half (group 4) of
// their maxima, in size and with one sign, over the whole chunk without being equal (16 equal
// products are a multiple of 16); random digits reach 2^20, in a row times itself 2^22.  (Chunks of 64 hold groups 0..4
// exactly whatever the digits are; an iteration by FP64 products at C10H20 took 5.11 ms with
// them, 4.49 with 128 and 4.45 with 256, at C6H12 1.08 / 1.00 / 0.97: the read-out of a chunk is
// longer than the products of 64 elements.)  Groups g >= 8 are dropped (2^-72 of the leading
// pair per digit pair).
//
// Error.  An element is off by at most 2^-61 of its row's (column's) largest one, so an output by
// 2^-61 (max|a| sum|b| + max|b| sum|a|), and by its one rounding, where an FP64 chain rounds every
// partial sum.  The bound is one on the norm: where small elements of a row meet the large ones of
// a column all along K, sum |a||b| is far below it, and so is the error of FP64 FMAs.  Rms error
// relative to sum |a||b| at K = 144, rows and columns graded against one another over a factor of
// 1 / 2^10 / 2^20 / 2^40: 6e-18 / 2e-17 / 8e-15 / 7e-9, FP64 FMAs 4e-17 to 7e-17.  (Base 256, 55
// bits: 1e-17 / 2e-15 / 1e-12 / 9e-7.)  b_half at C10H20, of its largest element, for orbitals
// spread over the ring / of RHF / nearest to the basis functions: 4e-17 / 3e-17 / 3e-16, FP64 FMAs
// 2e-16 / 1e-16 / 7e-16 (base 256: 7e-16 / 1e-15 / 5e-14).
//
// Time: 34 products at the tensor rate are 45 times faster than FP64.  With both operands'
// digitisation, against the FP64 kernel: 720 x 720 x 720 51 us (725), 32 of 400 x 400 x 400
// 225 us (4424), 96 x 96 x 96 21 us (29).  A CTA takes 70 KB of operands per 1088 tensor
// cycles, about what an SM draws from L2, and writes FP64 outputs; short products are
// bound by their three launches.
#include "common.cuh"
#include "tcgen05.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <limits.h>

namespace donof {

constexpr int X_PLANES = 7, X_NG = 8;
constexpr int X_BM = 128, X_BN = 32, X_BK = 32;
constexpr int X_CHUNK_KB = 4;  // K blocks whose sums one accumulator set holds (128 elements)
constexpr int X_STAGES = 3;
constexpr int X_SETS = 2;      // accumulator sets: 2 x 8 groups x 32 columns, all of TMEM
constexpr int X_NWG = 4, X_WN = X_BN / X_NWG;  // epilogue warpgroups, columns of each
constexpr int X_THREADS = 128 + 128 * X_NWG;
constexpr uint32_t X_A_BYTES = X_PLANES * X_BM * X_BK * 2, X_B_BYTES = X_PLANES * X_BN * X_BK * 2;
constexpr uint32_t X_STAGE_BYTES = X_A_BYTES + X_B_BYTES;
constexpr size_t X_SMEM = X_STAGES * (size_t)X_STAGE_BYTES + 256;
static_assert(X_SMEM <= 227 * 1024, "shared memory of a CTA");

// A product C[b] = alpha A[b] B[b] + beta C[b], tile by tile.
struct XParams {
  CUtensorMap a, b;       // (k, row, batch entry, digit)
  const int *ea, *eb;     // [entry][M], [entry][N]
  int M, N, K, batch;
  int a_batched, b_batched;
  int mt, nt;             // tiles
  int a_tri, b_tri;       // A's rows / B's columns end at their own index (lower triangular)
  int c_tri;              // 1: only tiles that reach the diagonal or lie below it; 2: or above it
  double* C;
  long long sCb, sCm, sCn;
  int fm, fn;             // rows / columns of one batch entry where they are folded into M / N (else 0)
  double alpha, beta;
  int* status;
};

// The seven digits of |X| < 2^61 as BF16 patterns: the 9-bit fields of X + 256 (2^45 + 2^36 + ...
// + 1) are d1 + 256, ..., d6 + 256 (each read as a float under the exponent of 2^23), and what is
// above them is d0 with its sign.
constexpr int X_BITS = 62, X_RADIX = 9;
__device__ __forceinline__ void x_digits(long long X, __nv_bfloat16 d[X_PLANES]) {
  const long long U = X + 256ll * ((1ll << 45) + (1ll << 36) + (1ll << 27) + (1ll << 18) + (1ll << 9) + 1ll);
  const unsigned int lo = (unsigned int)U, hi = (unsigned int)((unsigned long long)U >> 32);
  d[0] = __float2bfloat16((float)((int)hi >> 22));
#pragma unroll
  for (int t = 1; t < X_PLANES; ++t) {
    const int sh = X_RADIX * (X_PLANES - 1 - t);  // 45, 36, ..., 0
    const unsigned int f = sh >= 32 ? hi >> (sh - 32) : __funnelshift_r(lo, hi, sh);
    const float x = __uint_as_float((f & 511u) | 0x4B000000u) - 8388864.0f;  // 2^23 + 256
    d[t] = __ushort_as_bfloat16((unsigned short)(__float_as_uint(x) >> 16));
  }
}

// The exponent of a row that holds an infinity or a NaN: every product with it is NaN.
constexpr int X_NONFINITE = 1 << 28;

// |x| as an integer that orders like it (the FP64 pipe stays free; NaN is above everything)
__device__ __forceinline__ unsigned long long x_mag(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// Exponent e with |x| < 2^(e-1) for |x| up to the magnitude; 0 for zero.
__device__ __forceinline__ int x_expo(unsigned long long mag) {
  const int f = (int)(mag >> 52);
  return mag == 0 ? 0 : f == 2047 ? X_NONFINITE : (f ? f : 1) - 1021;
}

// x 2^(62 - e) rounded to the nearest integer (ties away from zero), |x| < 2^(e-1), by integer
// instructions: this part's FP64 pipe converts and multiplies two lanes a clock, and a
// digitisation of a 504 x 144 x 144 tensor took 126 us with it (90 along rows), 48 (59) without.
__device__ __forceinline__ long long x_fixed(double x, int e) {
  const unsigned long long mag = x_mag(x);
  const int f = (int)(mag >> 52);
  const unsigned long long m = ((mag & 0xFFFFFFFFFFFFFull) | (f ? 1ull << 52 : 0ull)) << 8;
  const int sh = e - (f ? f : 1) + 1021;  // x = m 2^(f - 1083), X = m 2^-sh; sh >= 0
  const unsigned long long r = sh > 62 ? 0ull : (m + ((1ull << sh) >> 1)) >> sh;
  return x < 0.0 ? -(long long)r : (long long)r;
}

// (H + L 2^-32) 2^k rounded to FP64 (to nearest, up to 2^-11 of a half unit), by integer
// instructions: with FP64 conversions and scalings the epilogue took longer than the tensor
// products of K <= 256.
__device__ __forceinline__ double x_value(long long H, long long L, int k) {
  long long h = H + (L >> 32);
  unsigned int l = (unsigned int)L;  // H 2^32 + L = h 2^32 + l, 0 <= l < 2^32
  const bool neg = h < 0;
  if (neg) {
    l = 0u - l;
    h = ~h + (l == 0);
  }
  unsigned long long M = (unsigned long long)h;
  if (M == 0) {
    M = l;
    l = 0;
    k -= 32;
    if (M == 0) return 0.0;
  }
  const int lz = __clzll((long long)M);
  M <<= lz;
  M |= lz <= 32 ? ((unsigned long long)l << lz) >> 32 : (unsigned long long)l << (lz - 32);
  const unsigned long long mant = (M >> 11) + ((M >> 10) & 1);  // in [2^52, 2^53]
  const int field = k - lz + 1086;
  unsigned long long bits = ((unsigned long long)(unsigned int)(field - 1) << 52) + mant;
  if (field < 1 || field > 2045) bits = (unsigned long long)__double_as_longlong(ldexp((double)mant, field - 1075));
  return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}

// Digit rows of a matrix whose elements (r, k) lie at X[r rs + k]: a warp per row, neighbouring
// pairs of k per lane.
__global__ void __launch_bounds__(256) x_digits_rows_kernel(const double* __restrict__ X, int rows, int K, long long rs,
                                                            long long sb, __nv_bfloat16* __restrict__ out, int Kp,
                                                            int* __restrict__ exps) {
  pdl_entry();
  const int lane = threadIdx.x % 32, r = blockIdx.x * 8 + threadIdx.x / 32;
  if (r >= rows) return;
  const double* x = X + blockIdx.y * sb + (long long)r * rs;
  unsigned long long mx = 0;
#pragma unroll 4
  for (int k = lane; k < K; k += 32) mx = max(mx, x_mag(x[k]));
  // the largest exponent field decides (a zero row: no bits at all)
  const unsigned int hi = __reduce_max_sync(0xffffffffu, (unsigned int)(mx >> 32) | ((unsigned int)mx != 0));
  const int e = x_expo((unsigned long long)hi << 32);
  const size_t row = (size_t)blockIdx.y * rows + r;
  if (lane == 0) exps[row] = e;
  __nv_bfloat16* o = out + row * X_PLANES * Kp;
#pragma unroll 2
  for (int k = 2 * lane; k < K; k += 64) {  // Kp is even: the pair may end in the padding
    __nv_bfloat16 d0[X_PLANES], d1[X_PLANES];
    x_digits(x_fixed(x[k], e), d0);
    x_digits(k + 1 < K ? x_fixed(x[k + 1], e) : 0, d1);
#pragma unroll
    for (int t = 0; t < X_PLANES; ++t) *(__nv_bfloat162*)(o + (size_t)t * Kp + k) = __halves2bfloat162(d0[t], d1[t]);
  }
}

// The same for elements at X[r + k ks], in two passes over blocks of 32 rows and 64 k (a block
// that walks all of K leaves most SMs idle at a few hundred rows): the largest exponent of
// each block, then the digits under the largest of the row's blocks, turned around in shared
// memory so that both the reads (along r) and the digits (along k) are contiguous.
constexpr int X_CK = 64;

__global__ void __launch_bounds__(256) x_maxexp_cols_kernel(const double* __restrict__ X, int rows, int K, long long ks,
                                                            long long sb, int* __restrict__ part) {
  pdl_entry();
  __shared__ unsigned long long red[8][32];
  const int tx = threadIdx.x, ty = threadIdx.y, r = blockIdx.x * 32 + tx, k0 = blockIdx.y * X_CK;
  const double* x = X + blockIdx.z * sb + r;
  unsigned long long mx = 0;
  if (r < rows) {
#pragma unroll
    for (int i = 0; i < X_CK / 8; ++i) {
      const int k = k0 + ty + 8 * i;
      if (k < K) mx = max(mx, x_mag(x[(long long)k * ks]));
    }
  }
  red[ty][tx] = mx;
  __syncthreads();
  if (ty == 0 && r < rows) {
#pragma unroll
    for (int y = 1; y < 8; ++y) mx = max(mx, red[y][tx]);
    part[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * rows + r] = mx ? x_expo(mx) : INT_MIN;
  }
}

__global__ void __launch_bounds__(256) x_digits_cols_kernel(const double* __restrict__ X, int rows, int K, long long ks,
                                                            long long sb, const int* __restrict__ part,
                                                            __nv_bfloat16* __restrict__ out, int Kp,
                                                            int* __restrict__ exps) {
  pdl_entry();
  __shared__ long long tile[X_CK][33];
  __shared__ int es[32];
  const int tx = threadIdx.x, ty = threadIdx.y, r0 = blockIdx.x * 32, r = r0 + tx, k0 = blockIdx.y * X_CK;
  const double* x = X + blockIdx.z * sb + r;
  const size_t row0 = (size_t)blockIdx.z * rows;
  double v[X_CK / 8];
#pragma unroll
  for (int i = 0; i < X_CK / 8; ++i) {
    const int k = k0 + ty + 8 * i;
    v[i] = r < rows && k < K ? x[(long long)k * ks] : 0.0;
  }
  if (ty == 0) {
    int e = INT_MIN;
    if (r < rows)
      for (int c = 0; c < (int)gridDim.y; ++c) e = max(e, part[((size_t)blockIdx.z * gridDim.y + c) * rows + r]);
    if (e == INT_MIN) e = 0;
    es[tx] = e;
    if (blockIdx.y == 0 && r < rows) exps[row0 + r] = e;
  }
  __syncthreads();
  const int e = es[tx];
#pragma unroll
  for (int i = 0; i < X_CK / 8; ++i) tile[ty + 8 * i][tx] = x_fixed(v[i], e);
  __syncthreads();
  // Kp is even and past K there are zeros in the tile: pairs of k may end in the padding
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int rr = ty + 8 * i, k = k0 + 2 * tx;
    if (r0 + rr < rows && k < K) {
      __nv_bfloat16 d0[X_PLANES], d1[X_PLANES];
      x_digits(tile[2 * tx][rr], d0);
      x_digits(tile[2 * tx + 1][rr], d1);
      __nv_bfloat16* o = out + (row0 + r0 + rr) * X_PLANES * Kp + k;
#pragma unroll
      for (int t = 0; t < X_PLANES; ++t) *(__nv_bfloat162*)(o + (size_t)t * Kp) = __halves2bfloat162(d0[t], d1[t]);
    }
  }
}

// K blocks of a tile: all of K, or up to the last row / column of a triangular operand.
__device__ __forceinline__ int x_kblocks(const XParams& p, int m0, int n0) {
  int k = p.K;
  if (p.a_tri) k = min(k, m0 + X_BM);
  if (p.b_tri) k = min(k, n0 + X_BN);
  return (k + X_BK - 1) / X_BK;
}

__device__ __forceinline__ bool x_skip(const XParams& p, int m0, int n0) {
  return p.c_tri && (p.c_tri == 1 ? n0 >= m0 + X_BM : m0 >= n0 + X_BN);
}

// The t-th tile of this CTA: batch entry and origin; false past the end.
__device__ __forceinline__ bool x_tile(const XParams& p, long long t, int& b, int& m0, int& n0) {
  const long long per = (long long)p.mt * p.nt;
  if (t >= per * p.batch) return false;
  b = (int)(t / per);
  const int r = (int)(t - b * per);
  m0 = r / p.nt * X_BM;
  n0 = r % p.nt * X_BN;
  return true;
}

template <bool FIRST>
__device__ __forceinline__ void x_mma_block(uint32_t d, uint64_t a0, uint64_t b0) {
  // B's planes lie one above the other: one MMA of N = 32 U multiplies digit plane t of A by
  // planes 0..U-1 of B into groups t..t+U-1 (see s4_mma_block); windows t = 0..6 take U = 7,
  // 7, 6, 5, 4, 3, 2.  The first K step writes every group before any MMA adds to it.
  constexpr uint64_t PA = (X_BM * X_BK * 2) >> 4, PB = (X_BN * X_BK * 2) >> 4;
#pragma unroll
  for (int ks = 0; ks < X_BK / 16; ++ks) {
    const uint64_t a = a0 + (uint64_t)(2 * ks), b = b0 + (uint64_t)(2 * ks);
    if (FIRST && ks == 0) {
      mma_bf16(d + X_BN, a + PA, b, idesc_bf16(7 * X_BN), 0u);
      mma_bf16(d, a, b, idesc_bf16(X_BN), 0u);
      mma_bf16(d + X_BN, a, b + PB, idesc_bf16(6 * X_BN), 1u);
    } else {
      mma_bf16(d, a, b, idesc_bf16(7 * X_BN), 1u);
      mma_bf16(d + X_BN, a + PA, b, idesc_bf16(7 * X_BN), 1u);
    }
#pragma unroll
    for (int t = 2; t < X_PLANES; ++t) mma_bf16(d + t * X_BN, a + t * PA, b, idesc_bf16((X_NG - t) * X_BN), 1u);
  }
}

__global__ void __launch_bounds__(X_THREADS, 1) x_gemm_kernel(const __grid_constant__ XParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* full = (uint64_t*)(smem + (size_t)X_STAGES * X_STAGE_BYTES);
  uint64_t* empty = full + X_STAGES;
  uint64_t* accf = empty + X_STAGES;
  uint64_t* acce = accf + X_SETS;
  uint64_t* drain = acce + X_SETS;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < X_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < X_SETS; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], 128 * X_NWG);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_entry();

  if (warp == 0) {
    if (lane == 0) {
      int it = 0, s = 0;
      uint32_t ph = 1;
      bool ok = true;
      int b, m0, n0;
      for (long long t = blockIdx.x; ok && x_tile(p, t, b, m0, n0); t += gridDim.x) {
        if (x_skip(p, m0, n0)) continue;
        const int nkb = x_kblocks(p, m0, n0);
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(&empty[s], ph, abort_flag, p.status)) { ok = false; break; }
          mbar_expect_tx(&full[s], X_STAGE_BYTES);
          uint8_t* st = smem + (size_t)s * X_STAGE_BYTES;
          tma_load_4d(st, &p.a, &full[s], kb * X_BK, m0, p.a_batched ? b : 0, 0);
          tma_load_4d(st + X_A_BYTES, &p.b, &full[s], kb * X_BK, n0, p.b_batched ? b : 0, 0);
          ++it;
          if (++s == X_STAGES) { s = 0; ph ^= 1; }
        }
      }
      for (int j = max(0, it - X_STAGES); j < it; ++j)
        mbar_wait(&full[j % X_STAGES], (uint32_t)((j / X_STAGES) & 1), nullptr, p.status);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint64_t STAGE = X_STAGE_BYTES >> 4, AB = X_A_BYTES >> 4;
      const uint64_t a_desc = sdesc_sw64(smem_u32(smem));
      int s = 0, c = 0;
      uint32_t ph = 0;
      bool ok = true;
      int b, m0, n0;
      for (long long t = blockIdx.x; ok && x_tile(p, t, b, m0, n0); t += gridDim.x) {
        if (x_skip(p, m0, n0)) continue;
        const int nkb = x_kblocks(p, m0, n0);
        for (int k0 = 0; k0 < nkb && ok; k0 += X_CHUNK_KB, ++c) {
          const int set = c & 1;
          if (!mbar_wait(&acce[set], (uint32_t)(((c >> 1) & 1) ^ 1), abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d = tmem_base + (uint32_t)(set * X_NG * X_BN);
          const int n = min(X_CHUNK_KB, nkb - k0);
          for (int j = 0; j < n; ++j) {
            if (!mbar_wait(&full[s], ph, abort_flag, p.status)) { ok = false; break; }
            tc_fence_after();
            const uint64_t st = a_desc + (uint64_t)s * STAGE;
            if (j == 0) x_mma_block<true>(d, st, st + AB);
            else x_mma_block<false>(d, st, st + AB);
            mma_commit(&empty[s]);
            if (++s == X_STAGES) { s = 0; ph ^= 1; }
          }
          if (ok) mma_commit(&accf[set]);
        }
      }
      mma_commit(drain);
      mbar_wait(drain, 0, nullptr, p.status);
    }
  } else if (warp >= 4) {
    const int ew = warp - 4, q = warp & 3, row = q * 32 + lane, col = (ew / 4) * X_WN;
    const uint32_t tb = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)col;
    int c = 0;
    bool ok = true;
    int b, m0, n0;
    for (long long t = blockIdx.x; ok && x_tile(p, t, b, m0, n0); t += gridDim.x) {
      if (x_skip(p, m0, n0)) continue;
      const int nkb = x_kblocks(p, m0, n0), m = m0 + row;
      const int ea = m < p.M ? __ldg(p.ea + (p.a_batched ? (size_t)b * p.M : 0) + m) : 0;
      long long H[X_WN], L[X_WN];  // exact sums of groups 0..3 (units 2^-31) and 4..7 (2^-63)
#pragma unroll
      for (int j = 0; j < X_WN; ++j) H[j] = L[j] = 0;
      for (int k0 = 0; k0 < nkb; k0 += X_CHUNK_KB, ++c) {
        const int set = c & 1;
        if (!mbar_wait(&accf[set], (uint32_t)((c >> 1) & 1), abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t ts = tb + (uint32_t)(set * X_NG * X_BN);
#pragma unroll
        for (int j0 = 0; j0 < X_WN; j0 += 4) {
          uint32_t g[X_NG][4];
          __syncwarp();
#pragma unroll
          for (int i = 0; i < X_NG; ++i) tmem_ld_issue<4>(ts + (uint32_t)(i * X_BN + j0), g[i]);
#pragma unroll
          for (int i = 0; i < X_NG; ++i) tmem_wait<4>(g[i]);
          if (j0 + 4 == X_WN) {
            tc_fence_before();
            mbar_arrive(&acce[set]);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              H[j0 + j] += (long long)__float2int_rn(__uint_as_float(g[i][j])) << (31 - X_RADIX * i);
              L[j0 + j] += (long long)__float2int_rn(__uint_as_float(g[i + 4][j])) << (27 - X_RADIX * i);
            }
          }
        }
      }
      if (!ok || m >= p.M) continue;
      double* crow = p.C + (p.fm ? (long long)(m / p.fm) * p.sCb + (long long)(m % p.fm) * p.sCm
                                 : (long long)b * p.sCb + (long long)m * p.sCm);
      // C's old values in one go: a load after a store to C would wait for it
      double old[X_WN];
      if (p.beta != 0.0) {
#pragma unroll
        for (int j = 0; j < X_WN; ++j) {
          const int n = n0 + col + j;
          if (n < p.N)
            old[j] = crow[p.fn ? (long long)(n / p.fn) * p.sCb + (long long)(n % p.fn) * p.sCn : (long long)n * p.sCn];
        }
      }
#pragma unroll
      for (int j = 0; j < X_WN; ++j) {
        const int n = n0 + col + j;
        if (n < p.N) {
          const int eb = __ldg(p.eb + (p.b_batched ? (size_t)b * p.N : 0) + n);
          // value 2^(ea + eb - 16) sum_g G_g 2^(-9g), sum_g = H 2^-31 + L 2^-63
          double* dst = crow + (p.fn ? (long long)(n / p.fn) * p.sCb + (long long)(n % p.fn) * p.sCn : (long long)n * p.sCn);
          const int k = ea + eb - 47;
          double v;
          if (p.beta != 0.0) {  // the leading part first: what cancels against C does so exactly
            v = fma(p.alpha, x_value(H[j], 0, k), p.beta == 1.0 ? old[j] : p.beta * old[j]);
            v = fma(p.alpha, x_value(L[j], 0, k - 32), v);
          } else {
            v = x_value(H[j], L[j], k);
            if (p.alpha != 1.0) v *= p.alpha;
          }
          if (max(ea, eb) == X_NONFINITE) v = __longlong_as_double(0x7ff8000000000000ll);
          *dst = v;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// Upper triangles from the lower ones, 32 x 32 tiles turned around in shared memory.
__global__ void __launch_bounds__(256) mirror_lower_kernel(double* X, int n) {
  __shared__ double s[32][33];
  if (blockIdx.x > blockIdx.y) return;
  double* M = X + (size_t)blockIdx.z * n * n;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += 8)
    if (r0 + i < n && c0 + threadIdx.x < n) s[i][threadIdx.x] = M[(size_t)(r0 + i) * n + c0 + threadIdx.x];
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = c0 + i, c = r0 + threadIdx.x;
    if (c < n && r < c) M[(size_t)r * n + c] = s[threadIdx.x][i];
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
static int x_ld(int K) { return (K + 15) / 16 * 16; }
static int x_chunks(int K) { return (K + X_CK - 1) / X_CK; }

size_t xgemm_operand_bytes(int rows, int K, int batch) {
  return ((size_t)batch * rows * X_PLANES * x_ld(K) * 2 + 255) / 256 * 256 +
         ((size_t)batch * rows * 4 * (1 + x_chunks(K)) + 255) / 256 * 256;
}

static int x_map(PFN_cuTensorMapEncodeTiled_v12000 encode, CUtensorMap* map, const void* base, int K, int rows, int batch,
                 int brow) {
  const cuuint64_t ld = (cuuint64_t)x_ld(K);
  const cuuint64_t d[4] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batch, X_PLANES};
  const cuuint64_t s[3] = {ld * X_PLANES * 2, ld * X_PLANES * 2 * rows, ld * 2};
  const cuuint32_t box[4] = {X_BK, (cuuint32_t)brow, 1, X_PLANES}, es[4] = {1, 1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)base, d, s, box, es,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? DONOF_RI_OK : DONOF_RI_E_CUDA;
}

// Digits of `rows` rows of K elements (element (r, k) of entry b at X[b sb + r rs + k ks], one
// stride 1) into ws.
static int x_digitise(donof_ri_ctx* ctx, const double* X, int rows, int K, long long rs, long long ks, long long sb,
                      int batch, void* ws, __nv_bfloat16** dig, int** exps) {
  const int Kp = x_ld(K);
  *dig = (__nv_bfloat16*)ws;
  *exps = (int*)((char*)ws + ((size_t)batch * rows * X_PLANES * Kp * 2 + 255) / 256 * 256);
  if (ks == 1)
    launch_pdl(x_digits_rows_kernel, dim3((rows + 7) / 8, batch), dim3(256), 0, ctx->stream, X, rows, K, rs, sb, *dig, Kp, *exps);
  else {
    int* part = *exps + (size_t)batch * rows;
    const dim3 grid((rows + 31) / 32, x_chunks(K), batch);
    launch_pdl(x_maxexp_cols_kernel, grid, dim3(32, 8), 0, ctx->stream, X, rows, K, ks, sb, part);
    DONOF_LAUNCH_CHECK(ctx);
    launch_pdl(x_digits_cols_kernel, grid, dim3(32, 8), 0, ctx->stream, X, rows, K, ks, sb, (const int*)part, *dig, Kp,
               *exps);
  }
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

// Device memory of `bytes`, or of half, a quarter, ... of it down to `least` where there is not
// that much room (launch_gemm64 then works in smaller pieces, with the same bits).  Which
// arithmetic a product takes never depends on the free memory: below `least` there is E_OOM.
int xgemm_alloc(size_t bytes, size_t least, void** p, size_t* got) {
  for (size_t n = bytes;; n = n / 2 > least ? n / 2 : least) {
    if (cudaMalloc(p, n) == cudaSuccess) {
      *got = n;
      return DONOF_RI_OK;
    }
    cudaGetLastError();
    *p = nullptr;
    *got = 0;
    if (n <= least) return DONOF_RI_E_OOM;
  }
}

// The context's workspace (xws_bytes long): `bytes` if there is room, at least `least`; it grows
// on demand and stays until it is released or the context goes.
int xgemm_workspace(donof_ri_ctx* ctx, size_t bytes, size_t least, void** ws) {
  if (ctx->xws_bytes < bytes) {
    if (ctx->d_xws) cudaFree(ctx->d_xws);  // waits for the work that uses it
    const int rc = xgemm_alloc(bytes, least, &ctx->d_xws, &ctx->xws_bytes);
    if (rc) return rc;
  }
  *ws = ctx->d_xws;
  return DONOF_RI_OK;
}

void xgemm_release(donof_ri_ctx* ctx) {
  if (ctx->d_xws) cudaFree(ctx->d_xws);
  ctx->d_xws = nullptr;
  ctx->xws_bytes = 0;
}

// True when launch_xgemm takes this product: unit strides along one dimension of each
// operand, and enough work for the tensor cores to pay (96 x 96 x 96: 21 us against the FP64
// kernel's 29; 64 x 64 x 64: 19 against 21, and one operand is padded to 128 rows).
bool xgemm_takes(const Gemm64& g) {
  const int lo = g.M < g.N ? g.M : g.N, hi = g.M < g.N ? g.N : g.M;
  return (g.sAk == 1 || g.sAm == 1) && (g.sBk == 1 || g.sBn == 1) && lo >= 32 && hi >= 96 && g.K >= 64 &&
         (double)g.M * g.N * g.K * g.batch >= 96.0 * 96 * 96 && g.batch <= 65535 && g.K <= (1 << 16);
}

// True when both operands are the rows of one matrix (X X^T): one set of digits serves both.
static bool x_same(const Gemm64& g) {
  return g.A == g.B && g.M == g.N && g.sAm == g.sBn && g.sAk == g.sBk && g.sAb == g.sBb;
}

// ws: at least xgemm_operand_bytes of A's rows and of B's columns together.  tri: XG_A_LOWER,
// XG_B_LOWER (element (k, n) of B is zero for k > n), XG_C_LOWER (C's tiles wholly above the
// diagonal are left alone).
int launch_xgemm(donof_ri_ctx* ctx, const Gemm64& g, void* ws, int tri) {
  static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return (PFN_cuTensorMapEncodeTiled_v12000)f;
  }();
  if (!encode) return DONOF_RI_E_UNSUPPORTED;
  // The accumulator's rows are the lanes of a warp: they run along C's unit stride (C^T = B^T A^T
  // where that is n), so that a warp's store is 256 contiguous bytes.
  const bool sw = g.sCn == 1 && g.sCm != 1;
  struct Side {
    const double* X;
    int rows, batch;
    long long rs, ks, sb;
  } sd[2] = {{g.A, g.M, g.sAb != 0 && g.batch > 1 ? g.batch : 1, g.sAm, g.sAk, g.sAb},
             {g.B, g.N, g.sBb != 0 && g.batch > 1 ? g.batch : 1, g.sBn, g.sBk, g.sBb}};
  Side &a = sd[sw], &b = sd[!sw];
  XParams p{};
  p.batch = g.batch;
  // one operand shared by the batch and the other's entries one below the other: a single
  // product over all their rows (an entry's rows would be padded to 128 or 32)
  const bool c_lower = tri & XG_C_LOWER;
  if (g.batch > 1 && !c_lower && (a.batch > 1) != (b.batch > 1)) {
    Side& f = a.batch > 1 ? a : b;
    const int f_tri = &f == &sd[0] ? XG_A_LOWER : XG_B_LOWER;
    if (f.sb == f.rows * f.rs && !(tri & f_tri) && (long long)f.rows * g.batch < (1LL << 30)) {
      (&f == &a ? p.fm : p.fn) = f.rows;
      f.rows *= g.batch;
      f.batch = 1;
      p.batch = 1;
    }
  }
  __nv_bfloat16 *da, *db;
  int *ea, *eb, rc;
  char* w = (char*)ws;
  if ((rc = x_digitise(ctx, a.X, a.rows, g.K, a.rs, a.ks, a.sb, a.batch, w, &da, &ea))) return rc;
  w += xgemm_operand_bytes(a.rows, g.K, a.batch);
  if (x_same(g)) {
    db = da;
    eb = ea;
  } else if ((rc = x_digitise(ctx, b.X, b.rows, g.K, b.rs, b.ks, b.sb, b.batch, w, &db, &eb))) {
    return rc;
  }
  if ((rc = x_map(encode, &p.a, da, g.K, a.rows, a.batch, X_BM)) || (rc = x_map(encode, &p.b, db, g.K, b.rows, b.batch, X_BN)))
    return rc;
  p.ea = ea; p.eb = eb;
  p.a_batched = a.batch > 1;
  p.b_batched = b.batch > 1;
  p.M = a.rows; p.N = b.rows; p.K = g.K;
  p.mt = (p.M + X_BM - 1) / X_BM;
  p.nt = (p.N + X_BN - 1) / X_BN;
  p.a_tri = tri & (sw ? XG_B_LOWER : XG_A_LOWER) ? 1 : 0;
  p.b_tri = tri & (sw ? XG_A_LOWER : XG_B_LOWER) ? 1 : 0;
  p.c_tri = c_lower ? 1 + sw : 0;
  p.C = g.C; p.sCb = g.sCb;
  p.sCm = sw ? g.sCn : g.sCm;
  p.sCn = sw ? g.sCm : g.sCn;
  p.alpha = g.alpha; p.beta = g.beta;
  p.status = ctx->d_status;
  const long long tiles = (long long)p.mt * p.nt * p.batch;
  DONOF_CUDA_TRY(cudaFuncSetAttribute(x_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)X_SMEM));
  launch_pdl(x_gemm_kernel, dim3((unsigned)(tiles < 152 ? tiles : 152)), dim3(X_THREADS), X_SMEM, ctx->stream, p);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

int launch_mirror_lower(donof_ri_ctx* ctx, double* X, int n, int batch) {
  const unsigned int nt = (n + 31) / 32;
  for (int b = 0; b < batch; b += 65535) {
    mirror_lower_kernel<<<dim3(nt, nt, batch - b < 65535 ? batch - b : 65535), dim3(32, 8), 0, ctx->stream>>>(
        X + (size_t)b * n * n, n);
    DONOF_LAUNCH_CHECK(ctx);
  }
  return DONOF_RI_OK;
}

// The product by launch_xgemm, in as many pieces as its digits need to fit `bytes` of ws
// (batch entries, or 128-row multiples of the longer side); by the FP64 kernel where the caller
// has no ws or xgemm_takes refuses the product.  K sums are exact, so the pieces do not change a
// bit.  E_OOM if ws holds not even one piece.
int launch_gemm64(donof_ri_ctx* ctx, const Gemm64& g, void* ws, size_t bytes, int tri) {
  if (!ws || !xgemm_takes(g)) return launch_dgemm(ctx, g);
  Gemm64 h = g;
  int rc;
  if (g.batch > 1) {
    const size_t a = xgemm_operand_bytes(g.M, g.K, 1), b = xgemm_operand_bytes(g.N, g.K, 1);
    const size_t fixed = (g.sAb ? 0 : a) + (g.sBb ? 0 : b), per = (g.sAb ? a : 0) + (g.sBb && !x_same(g) ? b : 0);
    if (per == 0) return launch_dgemm(ctx, g);
    if (fixed + per > bytes) return DONOF_RI_E_OOM;
    const size_t fit = (bytes - fixed) / per;
    const int step = fit < (size_t)g.batch ? (int)fit : g.batch;
    for (int i = 0; i < g.batch; i += step) {
      h.batch = g.batch - i < step ? g.batch - i : step;
      h.A = g.A + (long long)i * g.sAb;
      h.B = g.B + (long long)i * g.sBb;
      h.C = g.C + (long long)i * g.sCb;
      if ((rc = launch_xgemm(ctx, h, ws, tri))) return rc;
    }
    return DONOF_RI_OK;
  }
  const bool n_long = g.N >= g.M;
  const int rows = n_long ? g.N : g.M;
  const size_t other = xgemm_operand_bytes(n_long ? g.M : g.N, g.K, 1);
  int step = rows;
  while (step > 128 && other + xgemm_operand_bytes(step, g.K, 1) > bytes) step = ((step + 1) / 2 + 127) / 128 * 128;
  if (other + xgemm_operand_bytes(step, g.K, 1) > bytes || (step < rows && (tri || x_same(g)))) return DONOF_RI_E_OOM;
  for (int i = 0; i < rows; i += step) {
    const int n = rows - i < step ? rows - i : step;
    (n_long ? h.N : h.M) = n;
    if (n_long) h.B = g.B + (long long)i * g.sBn;
    else h.A = g.A + (long long)i * g.sAm;
    h.C = g.C + (long long)i * (n_long ? g.sCn : g.sCm);
    if ((rc = launch_xgemm(ctx, h, ws, tri))) return rc;
  }
  return DONOF_RI_OK;
}

}  // namespace donof
