// Exact-accumulation BF16 digit-plane path (DONOF_RI_SLICE4) for sm_103a.
//
// Every GEMM operand row r is stored as a power-of-two exponent e_r and four
// balanced base-256 digits: X_rk = 2^(e_r - 31) Xint_rk with
//   Xint = d0 2^24 + d1 2^16 + d2 2^8 + d3,  |Xint| < 2^30,
//   d0 in [-64, 64], d1..d3 in [-128, 127],
// so the digits are small integers, exact in BF16, and the int32 Xint turns into
// digits with one addition (Xint + 0x808080: the top byte is d0, the others are
// d_t + 128).  The four digits of a row are stored interleaved per row:
// element (r, t, k) at [(r*4 + t)*ld + k], one TMA coordinate selecting t.
//
// A product of operand rows i and j is
//   sum_k A_ik B_jk = 2^(ea_i + eb_j - 62) sum_{t,u} 256^(6-t-u) sum_k dA_t dB_u,
// and the digit-pair products with t + u <= 4 (13 of the 16) are issued as
// tcgen05.mma kind::f16 into five FP32 TMEM accumulators, one per g = t + u.  The
// g = 4 group lies 2^-32 below the leading pair but is kept: for a row multiplied
// by itself (J_pp, K^(p)_{mu mu}) its (2,2) product is a sum of squares whose bias
// grows with K.  With |d0| <= 64 and |d1..d3| <= 128 one K element adds at most
// 2^12, 2^14, 2^15, 3 2^14, 3 2^14 to groups 0..4, so over a 512-wide K chunk
// every partial sum of groups 0..2 is an integer of magnitude <= 2^24 and their
// FP32 accumulation is exact; groups 3 and 4 may round once they pass 2^24, an
// error below 2^-38 of the leading group's scale.  After every chunk the
// epilogue combines the five sums: J_pq and the multi-chunk J^(q), K^(q) and full
// transform fold them into one int64 per output (v = sum_g G_g 2^(32 - 8g); the
// value is 2^(ea + eb - 46) v), so the reduction over K is exact in its leading
// 38 bits and independent of order; single-chunk units convert them straight to
// a double-float pair (groups_to_df); the half transform rounds each group term
// to an integer at its output scale (half_fold) and adds the chunks' integers.
// The other errors are the 31-bit digit representation of the operands and the
// dropped pair products (g >= 5).
// Outputs feeding another GEMM are re-digitised in integer arithmetic, with
// bound-based exponents (b_half) or exact row maxima (d, J^(q), K^(q)).
//
// Rows of the hot path as in tc.cu (HALF, FULLSQ, JMO, JAO, KAO, FOCK); the paper's
// equations: Sec. 2, Tables 2 and 3, Eq. (PNOF).
#include "common.cuh"
#include "numeric.cuh"
#include "tcgen05.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <stdlib.h>

#include <algorithm>
#include <new>
#include <vector>

namespace donof {

// S_JKAO: J^(q) and K^(q) of one orbital iteration in one persistent launch (the
// J^(q) tiles, then the K^(q) (tile, orbital) units).
// S_CTR: the contracted Lagrangian's F^(p) C_p without J^(q), K^(q): one GEMM over
// K = (q, P), sum_q sum_P X^P_qp b^P_{q mu}, one batch per orbital q (rows mu of the
// b_half digits in the K^(q) layout, columns p of the X digits, both over P) whose
// chunks are converted to double-float and summed across the unit's orbitals.
enum S4Kind {
  S_HALF = 0, S_FULLSQ = 1, S_JMO = 2, S_JAO = 3, S_KAO = 4, S_FOCK = 5, S_JKAO = 6, S_CTR = 7,
  S_NKINDS = 8
};

static_assert(DONOF_RI_GEMM_FOCK - DONOF_RI_GEMM_HALF == S_FOCK, "GEMM profile rows follow the kind order");

constexpr int S4_BM = 128;      // rows per tile
constexpr int S4_BK = 32;       // BF16 elements per K block (one 64-byte swizzle row)
constexpr int S4_KS = S4_BK / 16;  // MMA K steps per K block
constexpr int S4_CHUNK_KB = 16; // K blocks per chunk (512 elements; groups 0..2 exact)
// The kinds that contract over the orbital basis (K = nbf: the half and full
// transforms and F^(p) C_p) take chunks of up to 23 blocks (736 elements), so that
// a basis of up to 736 functions needs one epilogue drain per unit.  Past 512
// elements group 2's FP32 sum may round once it exceeds 2^24, which needs most of
// the chunk's top-digit products near their maximum; each rounding is at most one
// unit of the group, and the 3 K/16 accumulations into it add at most
// 3 K/16 2^(32-16) to the 2^(32 + 24.5)-scale sums: below 2^-30 of the largest
// value the chunk can hold (the operands' 31-bit digits already cost 2^-31).
constexpr int S4_CHUNK_KB_NB = 23;
// K blocks per epilogue chunk of a kind
__host__ __device__ constexpr int s4_chunk_kb(int kind) {
  return (kind == S_HALF || kind == S_FULLSQ || kind == S_FOCK) ? S4_CHUNK_KB_NB : S4_CHUNK_KB;
}
constexpr int S4_PLANES = 4;
constexpr int S4_NG = 5;        // digit-pair groups g = t + u = 0..4
constexpr int S4_SHIFT = 46;    // value = 2^(ea + eb - 46) v

// Tile of a CTA: 128 rows x two halves of 48 columns.  Each half has its own
// accumulator set (five groups x 48 TMEM columns, 480 of 512 together), its own
// MMA-issuing warp and its own two epilogue warpgroups; a stage holds one K block of the
// four A planes and of the four B planes of both halves, so the A digits are fetched once
// for 96 columns.
//
// Why this shape.  The MMAs of a 32-wide K block and one half take 624 cycles (measured
// alone: 4095 multiply-adds a cycle per SM, the tensor pipe's rate), so at 128 x 48 the
// operands need 72 bytes a cycle per SM from L2, above what it delivers; 128 x 96 needs
// 46.  One window over 96 columns would need N = 384 per MMA, hence two halves.
// Measured (us, C20H40: nbf 720, naux 2520, 400 orbitals; with a 128 x 48 tile, one issuer
// and one epilogue warpgroup per accumulator set -> now): half transform 11110 -> 8430,
// full transform 9090 -> 5410, J^(q) 7690 -> 5200, K^(q) 6680 -> 4720, F^(p) C_p 5800 -> 3020;
// the half transform executes 1.61 PFLOP/s of BF16 products, and the card is at its
// power limit (1.3-1.4 kW) there.
constexpr int S4_BN = 48;
constexpr int S4_NHALF = 2;
// Two epilogue warpgroups per half, 24 columns each: four warps per scheduler hide one
// another's arithmetic latency (a batch's conversion and sums are chains of dependent
// FP32 operations), and a half is drained in half the time.
constexpr int S4_NWG = 2 * S4_NHALF;
constexpr int S4_WN = S4_BN / 2;  // columns of an epilogue warpgroup
constexpr int S4_THREADS = 128 + 128 * S4_NWG;
constexpr int S4_TMEM_COLS = 512;
constexpr uint32_t S4_A_BYTES = S4_PLANES * S4_BM * S4_BK * 2;
constexpr uint32_t S4_B_BYTES = S4_PLANES * S4_BN * S4_BK * 2;
constexpr uint32_t S4_STAGE_BYTES = S4_A_BYTES + S4_NHALF * S4_B_BYTES;
// Each half has an MMA-issuing warp of its own.  One thread's waits and address
// arithmetic between the blocks are not hidden by the MMAs it has queued (a wait, a
// commit and the next block's descriptors cost up to 1000 cycles per K block of both
// halves here), two threads hide one another's (measured alone: 1251 cycles per K block
// of both halves against 1248 of MMA time); and the halves drift apart by up to the
// depth of the pipeline, so that one half's MMAs run while the other half is drained.
// K blocks by which the producer's L2 prefetch runs ahead of its loads.  A's tiles come
// from HBM, and the stages in flight (57 to 114 KB) do not cover that latency.
constexpr int S4_AHEAD = 6;
// Shared memory: the stages, the barriers (256 bytes) and per epilogue warp the exponents
// of its 24 columns; everything else a batch needs per column comes by shuffles from the
// lanes that hold it, so that four stages fit.
constexpr int S4_MAX_STAGES = 4;
constexpr size_t S4_FIXED_SMEM = 256 + 4 * S4_NWG * (size_t)(S4_WN * 4);
static_assert(S4_FIXED_SMEM + S4_MAX_STAGES * (size_t)S4_STAGE_BYTES <= 227 * 1024, "shared memory of a CTA");
constexpr int S4_SMS = 152;

// One operand pair of a kind.  A's rows are (batch entry, row): a tile holds `rows per
// group` R consecutive rows of 128 / R consecutive batch entries (R = 128: one
// entry), so that a row count that fills 128-row tiles badly (400 orbitals: 78 %)
// takes the group that fills them best.
struct S4Operands {
  CUtensorMap a, b;  // (k, row, batch entry, digit) and (k, column, batch entry or 0, digit)
  const int* ea;     // exponents of A's rows [entry][nrows]
  const int* eb;     // of B's columns [ncols], or [entry][ncols] when batched
  int rshift;        // log2 R
  int nrows, ncols, nent;
  int batched;       // B's columns belong to the batch entry
};

// Partials per output of a kind whose units are summed afterwards: `pair` for columns
// below `split` (units of two halves), `single` from there on.
struct S4Slots {
  int pair, single, split;
};

struct S4Params {
  S4Operands op[2];   // [1]: the K^(q) units of the merged J^(q) + K^(q) launch
  const int4* units;  // {first batch, batches | halves << 28 | operand pair << 30 | first of its row tile << 31, row tile, column tile | slot << 16}
  int nunits;
  int stages;
  int nkb;            // K blocks of a batch (all of K, or the kind's K chunk)
  int nkb_all;        // K blocks of the whole contraction
  int nc;             // K chunks a batch entry is split into (F^(p) C_p, J_pq; 1 otherwise)
  int nb, nx, m, nbp;
  const int* e3m;     // HALF: output exponents less C's and 17, e3[P][p] - eC[p] - 17, e6[p][nu] - eC[p] - 17
  const short* e6m;   // [nu][p], row stride e6ld: a thread's 24 columns are three 16-byte loads
  int e6ld;
  int* x6;            // ... and the b_half integers [nx][m][nbp] at scale min(e3, e6)
  float* ohi;         // J^(q), K^(q) as double-float [2m][nb][ldo]
  float* olo;
  int ldo;
  void* partial;      // sums of a unit: [slot x groups][prow][pcol]
  int prow, pcol;
  const float2* w;    // FOCK weights as double-float pairs [2m][m]
  int* status;
  const int* tri;     // J^(q): packed row r of the upper triangle -> mu << 16 | nu
  double* bfull;      // FULLSQ: when set, b^P_qp is also stored, [P][p][q] (FP64)
};

// ---------------------------------------------------------------------------
// integer / double-float helpers
// ---------------------------------------------------------------------------
// Four balanced digits of |X| < 2^30 as BF16 values.  U = X + 0x80808080 holds
// digit + 128 in each byte (the top digit lies in [-64, 64]).  A byte b placed
// under the exponent of 2^23 reads as the float 2^23 + b, and subtracting
// 2^23 + 128 leaves the digit exactly; an integer of at most 8 significant bits
// is exact in BF16, so its BF16 pattern is the top half of the FP32 pattern.
__device__ __forceinline__ void digits_bf16(int X, __nv_bfloat16 d[4]) {
  const unsigned int U = (unsigned int)X + 0x80808080u;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const float x = __uint_as_float(__byte_perm(U, 0x4B000000u, 0x7440u | (unsigned int)(3 - t))) - 8388736.0f;
    d[t] = __ushort_as_bfloat16((unsigned short)(__float_as_uint(x) >> 16));
  }
}

// The digits of two integers at once, as BF16 pairs (d[t].x from X0, d[t].y from X1):
// the same exact digit values, each pair rounded to BF16 by one packed conversion
// (exact: every digit has at most 8 significant bits).
__device__ __forceinline__ void digits_bf16x2(int X0, int X1, __nv_bfloat162 d[4]) {
  const unsigned int U0 = (unsigned int)X0 + 0x80808080u, U1 = (unsigned int)X1 + 0x80808080u;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const unsigned int sel = 0x7440u | (unsigned int)(3 - t);
    const float x0 = __uint_as_float(__byte_perm(U0, 0x4B000000u, sel)) - 8388736.0f;
    const float x1 = __uint_as_float(__byte_perm(U1, 0x4B000000u, sel)) - 8388736.0f;
    d[t] = __floats2bfloat162_rn(x0, x1);
  }
}

// Exponent e with |x| < 2^(e-1) for every |x| <= amax (amax >= 0); 0 for amax == 0.
__device__ __forceinline__ int expo_of(double amax) {
  if (!(amax > 0.0)) return 0;
  int k;
  frexp(amax, &k);
  return k + 1;
}

// expo_of((double)mx * (1 + 2^-16)) for an FP32 bound mx, in integer arithmetic
// (the product is exact in FP64: 24 x 17 significant bits).  With mx = I0 2^(E-150),
// I0 = 2^23 + mantissa, the product is I0 (2^16 + 1) 2^(E-166), whose frexp
// exponent is E - 126, or E - 125 once I0 (2^16 + 1) reaches 2^40.  Zero,
// subnormal and non-finite bounds take the FP64 route.  (FP64 instructions run
// at a small fraction of the FP32 rate; these bounds are taken once per row.)
__device__ __forceinline__ int expo_of_inflated(float mx) {
  const unsigned int b = __float_as_uint(mx);
  const int E = (int)((b >> 23) & 0xFFu);
  if (mx > 0.f && E > 0 && E < 255) {
    const unsigned long long I = (unsigned long long)((b & 0x7FFFFFu) | 0x800000u) * 65537ull;
    return E - 125 + (I >= (1ull << 40) ? 1 : 0);
  }
  return expo_of((double)mx * (1.0 + 1.0 / 65536.0));
}

// x 2^k for FP64 x: one multiplication by an exact power of two while 2^k is a
// normal double (the same correctly rounded result as ldexp), ldexp beyond.
__device__ __forceinline__ double scale_pow2(double x, int k) {
  if (k >= -1022 && k <= 1023) return x * __longlong_as_double((long long)(k + 1023) << 52);
  return ldexp(x, k);
}

// FP64 -> double-float pair (h + l = x to about 2^-48 relative).
__device__ __forceinline__ float2 to_df(double x) {
  const float h = (float)x;
  return make_float2(h, (float)(x - (double)h));
}
__device__ __forceinline__ float2 to_df(float2 x) { return x; }

__device__ __forceinline__ void two_sum_f(float a, float b, float& s, float& e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// (sh, sl) += (ph, pl) in double-float arithmetic.
__device__ __forceinline__ void df_add(float& sh, float& sl, float ph, float pl) {
  float s, e;
  two_sum_f(sh, ph, s, e);
  e += sl + pl;
  sh = s + e;
  sl = e - (sh - s);
}

// 2^k as an FP32 value for k in [-126, 127] (k is clamped to that range).
__device__ __forceinline__ float exp2_int(int k) {
  k = k < -126 ? -126 : (k > 127 ? 127 : k);
  return __int_as_float((k + 127) << 23);
}

// v + x 2^k (0 <= k <= 32)
__device__ __forceinline__ long long mad_wide(int x, int k, long long v) {
  if (k == 32) return v + ((long long)x << 32);
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(v) : "r"(x), "r"(1 << k));
  return v;
}

// (h, l)[j] *= 2^(k[j]) for N column pairs (k: 2N exponents): one multiplication each
// while every 2^k of the warp is a normal float, two beyond (up to 2^(+-252)).  One
// branch for all of them, taken by the whole warp (every lane calls this): a branch per
// value would keep the values' dependent chains from overlapping.
template <int N>
__device__ __forceinline__ void df_scale(f32x2* h, f32x2* l, const int* k) {
  bool wide = false;
#pragma unroll
  for (int j = 0; j < 2 * N; ++j) wide |= (unsigned int)(k[j] + 126) > 253u;
  if (!__any_sync(0xffffffffu, wide)) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const f32x2 sc = pack2(__int_as_float((k[2 * j] + 127) << 23), __int_as_float((k[2 * j + 1] + 127) << 23));
      h[j] = mul2(h[j], sc);
      l[j] = mul2(l[j], sc);
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int ka = min(max(k[2 * j], -126), 127), kb = min(max(k[2 * j + 1], -126), 127);
      const f32x2 s1 = pack2(exp2_int(ka), exp2_int(kb)), s2 = pack2(exp2_int(k[2 * j] - ka), exp2_int(k[2 * j + 1] - kb));
      h[j] = mul2(mul2(h[j], s1), s2);
      l[j] = mul2(mul2(l[j], s1), s2);
    }
  }
}

// int64 as a double-float pair, built from 32-bit pieces only (|v| < 2^55):
// v = a 2^32 + b1 2^16 + b0 with every piece exact in FP32, summed with TwoSum.
__device__ __forceinline__ void ll_to_df(long long v, float& h, float& l) {
  const int a = (int)(v >> 32);
  const unsigned int lo = (unsigned int)v;
  const float fa = (float)a * 4294967296.f, f1 = (float)(lo >> 16) * 65536.f, f0 = (float)(lo & 0xFFFFu);
  float s, e;
  two_sum_f(fa, f1, s, e);
  float s2, e2;
  two_sum_f(s, f0, s2, e2);
  const float t = e + e2;
  h = s2 + t;
  l = t - (h - s2);
}

// Double-float values of one chunk's five group sums, sum_g G_g 2^(-8g), for a pair of
// columns, without the int64 fold.  Every term G_g 2^(-8g) is exact in FP32 and the sums
// are multiples of a common power of two, so each addition and its rounding error are
// three operations, s = fma(G, c, s0), e = fma(G, c, s0 - s) (a TwoSum of the scaled
// term takes seven); the errors and the last group are collected beside the sum.
// Error about 2^-48 of the largest sum, as the int64 fold and its conversion.
__device__ __forceinline__ void groups_to_df(const f32x2* G, f32x2& h, f32x2& l) {
  f32x2 s = G[0], e = 0;
#pragma unroll
  for (int g = 1; g < S4_NG - 1; ++g) {
    const f32x2 c = both2(exp2_int(-8 * g));
    const f32x2 t = fma2(G[g], c, s);
    const f32x2 r = fma2(G[g], c, sub2(s, t));
    e = g == 1 ? r : add2(e, r);
    s = t;
  }
  e = fma2(G[S4_NG - 1], both2(exp2_int(-8 * (S4_NG - 1))), e);
  h = add2(s, e);
  l = sub2(e, sub2(h, s));
}

// Output integer of the half transform from one chunk's group sums:
// X = sum_g rint(T_g), clamped to [-2^30, 2^30], with T_g = G_g 2^(sigma - 8 g) (exact).  Each term is rounded on its own, so X differs
// from round(v 2^(sigma - 32)) by at most 2.5; the row exponents guarantee
// |X| < 2^30 (the leading term is X to within a few per cent), so no term
// reaches the int32 range.
__device__ __forceinline__ int half_fold(const float T[S4_NG]) {
  int X = 0;
#pragma unroll
  for (int g = 0; g < S4_NG; ++g) X += __float2int_rn(T[g]);
  X = X > (1 << 30) ? (1 << 30) : X;
  X = X < -(1 << 30) ? -(1 << 30) : X;
  return X;
}

// round(X 2^-d) for d >= 0 (halves rounded up), without overflow.
__device__ __forceinline__ int rshift_round(int X, int d) {
  if (d <= 0) return X;
  const int sh = d - 1 > 31 ? 31 : d - 1;
  return ((X >> sh) + 1) >> 1;
}

// ---------------------------------------------------------------------------
// The digit-plane GEMM kernel
// ---------------------------------------------------------------------------
// A unit of work: one 128-row tile, one or two 48-column halves and a range of batches
// whose results are summed (FULLSQ, FOCK, CTR, JMO) or are one batch.  The units of a
// launch have equal cost (a unit with one half takes twice the batches); CTA c takes
// unit w G + (c + w) mod G in its w-th turn (G CTAs), so that a period of the list
// (the last column tile of every row tile has one half) does not fall on the same CTA.
// Walks the batches of the units of this CTA that have more than `h` halves; the next
// unit's descriptor is read while the current unit is worked on.
struct S4Cursor {
  int4 un, next;
  int b, w;
  bool valid, next_valid;

  __device__ __forceinline__ int nbat() const { return un.y & 0x0FFFFFFF; }
  __device__ __forceinline__ int nh() const { return (un.y >> 28) & 3; }
  __device__ __forceinline__ int opi() const { return (un.y >> 30) & 1; }
  __device__ __forceinline__ bool first() const { return un.y < 0; }
  __device__ __forceinline__ int mt() const { return un.z; }
  __device__ __forceinline__ int nt() const { return un.w & 0xFFFF; }
  __device__ __forceinline__ int slot() const { return (int)((unsigned int)un.w >> 16); }
  __device__ __forceinline__ void fetch(const S4Params& p) {
    const int G = (int)gridDim.x;
    int c = (int)blockIdx.x + w % G;
    if (c >= G) c -= G;
    const long long U = (long long)w * G + c;
    next_valid = U < p.nunits;
    if (next_valid) next = __ldg(p.units + U);
    ++w;
  }
  __device__ __forceinline__ void take(const S4Params& p, int h) {
    do {
      valid = next_valid;
      if (!valid) return;
      un = next;
      fetch(p);
    } while (h >= nh());
    b = un.x;
  }
  __device__ __forceinline__ void start(const S4Params& p, int h) {
    w = 0;
    fetch(p);
    take(p, h);
  }
  __device__ __forceinline__ bool last() const { return b + 1 >= un.x + nbat(); }
  __device__ __forceinline__ void step(const S4Params& p, int h) {
    if (last()) take(p, h);
    else ++b;
  }
};

// K blocks of batch b: the first one and their number.
__device__ __forceinline__ void s4_kblocks(const S4Params& p, int b, int& ent, int& kb0, int& nkb) {
  ent = b;
  kb0 = 0;
  nkb = p.nkb;
  if (p.nc > 1) {
    ent = b / p.nc;
    kb0 = (b - ent * p.nc) * p.nkb;
    nkb = min(p.nkb, p.nkb_all - kb0);
  }
}

// The eight MMAs of one K block and one half.  The B planes of a half sit one above the
// other (plane u at rows u*BN), so one MMA of N = 4*BN multiplies digit plane t of A by
// all four B planes and, with the accumulator window shifted by t*BN columns, adds
// product (t,u) to group t+u.  Window t covers groups t..min(t+3,4): four MMAs per K
// step instead of 13.  FIRST: the first block of a chunk, whose first K step writes
// every group once with accumulate = 0 before any MMA adds to it (window 1 initialises
// groups 1..4; group 0 is initialised by (0,0) alone and (0,1..3) then adds).
template <bool FIRST>
__device__ __forceinline__ void s4_mma_block(uint32_t dbase, uint64_t a0, uint64_t b0) {
  constexpr uint32_t BN = S4_BN;
  constexpr uint64_t PA = (S4_BM * S4_BK * 2) >> 4, PB = (BN * S4_BK * 2) >> 4;  // plane strides in descriptor units
  const uint32_t id1 = idesc_bf16(BN), id2 = idesc_bf16(2 * BN), id3 = idesc_bf16(3 * BN), id4 = idesc_bf16(4 * BN);
  // K step ks: +32 bytes inside the 64-byte swizzle row (+2 in the descriptor's address field)
#pragma unroll
  for (int ks = 0; ks < S4_KS; ++ks) {
    const uint64_t a = a0 + (uint64_t)(2 * ks), b = b0 + (uint64_t)(2 * ks);
    if (FIRST && ks == 0) {
      mma_bf16(dbase + BN, a + PA, b, id4, 0u);
      mma_bf16(dbase, a, b, id1, 0u);
      mma_bf16(dbase + BN, a, b + PB, id3, 1u);
    } else {
      mma_bf16(dbase, a, b, id4, 1u);
      mma_bf16(dbase + BN, a + PA, b, id4, 1u);
    }
    mma_bf16(dbase + 2 * BN, a + 2 * PA, b, id3, 1u);
    mma_bf16(dbase + 3 * BN, a + 3 * PA, b, id2, 1u);
  }
}

// STORE (full transform): b^P_qp is also stored, p.bfull.
template <int KIND, int ONE, bool STORE = false>
__global__ void __launch_bounds__(S4_THREADS, 1) s4_gemm_kernel(const __grid_constant__ S4Params p) {
  // ONE: every unit is a single K chunk (K <= 512, and always for F^(p) C_p), so the
  // epilogue converts group sums straight to double-float pairs and carries no int64
  // running sums; chosen at launch from the problem's K extent.
  // Beyond 736 functions the full transform's 24 int64 and 24 double-float sums a thread
  // spill (832 bytes of stores; 640 threads leave 96 registers each).  It is faster than the
  // 128 x 48 tile all the same, which spilled 136: nbf 761, naux 1200, 480 orbitals 6.53 ->
  // 3.61 ms (192 orbitals 1.07 -> 0.64; nbf 864 1.16 -> 0.70), the half transform 8.68 -> 6.23.
  constexpr int BN = S4_BN;
  constexpr int WN = S4_WN;  // columns of an epilogue warpgroup
  constexpr bool SUM_DF = (KIND == S_FULLSQ || KIND == S_FOCK || KIND == S_CTR);
  constexpr bool SUMS = SUM_DF || KIND == S_JMO;
  constexpr int CKB = s4_chunk_kb(KIND);
  // int64 running sums: J_pq and the multi-chunk kinds.  FOCK units are single chunks, CTR
  // converts every chunk on its own, and the half transform keeps its partial sums in its
  // output: none carries them
  constexpr int NACC = (KIND == S_JMO || (!ONE && (KIND == S_FULLSQ || KIND == S_JAO || KIND == S_KAO || KIND == S_JKAO))) ? WN : 1;
  // columns read from TMEM at a time (J^(q) and K^(q) take eight, a full sector of
  // their output rows; the others four, for their registers), blocks of them, and columns per unit action
  constexpr int CW = (SUM_DF || NACC > 1 || KIND == S_HALF) ? 4 : 8, NCB = WN / CW;
  constexpr int CN = NACC > 1 ? (SUM_DF ? 4 : 8) : CW;
  extern __shared__ __align__(1024) uint8_t smem[];  // stages first: swizzle atoms of 512 bytes
  const int S = p.stages;
  uint64_t* full = (uint64_t*)(smem + (size_t)S * S4_STAGE_BYTES);
  uint64_t* empty = full + S;
  uint64_t* accf = empty + S;
  uint64_t* acce = accf + S4_NHALF;
  uint64_t* drain = acce + S4_NHALF;
  uint32_t* tmem_slot = (uint32_t*)(drain + S4_NHALF);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], S4_NHALF);
    }
    for (int h = 0; h < S4_NHALF; ++h) {
      mbar_init(&accf[h], 1);
      mbar_init(&acce[h], 128 * S4_NWG / S4_NHALF);
      mbar_init(&drain[h], 1);
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, S4_TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // barriers and TMEM are set up; global memory only from here on
  pdl_entry();

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      int it = 0, s = 0;
      uint32_t ph = 1;
      bool ok = true;
      S4Cursor cu{}, pf;
      cu.start(p, 0);
      pf = cu;
      int pent = 0, pkb = 0, pend = 0;  // the prefetch's entry, next K block and end of its batch
      auto prefetch_batch = [&]() {
        if (pf.valid) {
          s4_kblocks(p, pf.b, pent, pkb, pend);
          pend += pkb;
        }
      };
      auto prefetch_next = [&]() {
        if (!pf.valid) return;
        const S4Operands& op = p.op[KIND == S_JKAO ? pf.opi() : 0];
        // A's rows once per row tile; the units that share them run at the same time
        if (pf.first()) tma_prefetch_4d(&op.a, pkb * S4_BK, pf.mt() << op.rshift, pent << (7 - op.rshift), 0);
        if (++pkb == pend) {
          pf.step(p, 0);
          prefetch_batch();
        }
      };
      prefetch_batch();
      for (int k = 0; k < S4_AHEAD; ++k) prefetch_next();
      for (; ok && cu.valid; cu.step(p, 0)) {
        const S4Operands& op = p.op[KIND == S_JKAO ? cu.opi() : 0];
        const uint32_t bytes = S4_A_BYTES + (uint32_t)cu.nh() * S4_B_BYTES;
        int ent, kb0, nkb;
        s4_kblocks(p, cu.b, ent, kb0, nkb);
        const int row0 = cu.mt() << op.rshift, n0 = cu.nt() * BN, ea0 = ent << (7 - op.rshift);
        const int eb0 = op.batched ? ent : 0;
        for (int kb = kb0; kb < kb0 + nkb; ++kb) {
          if (!mbar_wait(&empty[s], ph, abort_flag, p.status)) { ok = false; break; }
          mbar_expect_tx(&full[s], bytes);
          uint8_t* st = smem + (size_t)s * S4_STAGE_BYTES;
          tma_load_4d(st, &op.a, &full[s], kb * S4_BK, row0, ea0, 0);
          tma_load_4d(st + S4_A_BYTES, &op.b, &full[s], kb * S4_BK, n0, eb0, 0);
          if (cu.nh() > 1) tma_load_4d(st + S4_A_BYTES + S4_B_BYTES, &op.b, &full[s], kb * S4_BK, n0 + BN, eb0, 0);
          prefetch_next();
          ++it;
          if (++s == S) { s = 0; ph ^= 1; }
        }
      }
      for (int j = max(0, it - S); j < it; ++j) mbar_wait(&full[j % S], (uint32_t)((j / S) & 1), nullptr, p.status);
    }
  } else if (warp <= S4_NHALF) {
    if (lane == 0) {
      // ---------------- MMA issuer of half h ----------------
      const int h = warp - 1;
      const uint32_t dbase = tmem_base + (uint32_t)(h * S4_NG * BN);
      constexpr uint64_t STAGE = S4_STAGE_BYTES >> 4;
      const uint64_t a_desc = sdesc_sw64(smem_u32(smem));
      const uint64_t b_off = (S4_A_BYTES + (uint32_t)h * S4_B_BYTES) >> 4;
      uint64_t st = a_desc;
      int s = 0;
      uint32_t ph = 0, eph = 1;
      bool ok = true;
      auto next_stage = [&]() {
        st += STAGE;
        if (++s == S) {
          s = 0;
          st = a_desc;
          ph ^= 1;
        }
      };
      S4Cursor cu{};
      for (cu.start(p, 0); ok && cu.valid; cu.step(p, 0)) {
        int ent, kb0, nkb;
        s4_kblocks(p, cu.b, ent, kb0, nkb);
        if (h >= cu.nh()) {
          // not this half's unit: release its stages as they come
          for (int j = 0; j < nkb; ++j) {
            if (!mbar_wait(&full[s], ph, abort_flag, p.status)) { ok = false; break; }
            mbar_arrive(&empty[s]);
            next_stage();
          }
          continue;
        }
        for (int ch = 0; ch < nkb && ok; ch += CKB) {
          const int kbs = min(CKB, nkb - ch);
          if (!mbar_wait(&acce[h], eph, abort_flag, p.status)) { ok = false; break; }
          eph ^= 1;
          if (!mbar_wait(&full[s], ph, abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          s4_mma_block<true>(dbase, st, st + b_off);
          mma_commit(&empty[s]);
          next_stage();
          for (int j = 1; j < kbs; ++j) {
            if (!mbar_wait(&full[s], ph, abort_flag, p.status)) { ok = false; break; }
            tc_fence_after();
            s4_mma_block<false>(dbase, st, st + b_off);
            mma_commit(&empty[s]);
            next_stage();
          }
          if (ok) mma_commit(&accf[h]);
        }
      }
      // All MMAs of this thread must complete before TMEM is released.
      mma_commit(&drain[h]);
      mbar_wait(&drain[h], 0, nullptr, p.status);
    }
  } else if (warp >= 4) {
    // ---------------- epilogue (two warpgroups per half) ----------------
    // Each thread owns one output row (its TMEM lane) and 24 columns.  Per block of CW
    // columns the five exact group sums of a chunk are combined; a block is finalised
    // (stored, squared or weighted) as soon as the last chunk of its batch is drained.
    const int ew = warp - 4, h = ew / 8, cpart = ((ew / 4) & 1) * WN;
    const int q = warp & 3;     // TMEM lane quarter this warp may access
    const int row = q * 32 + lane;
    // column exponents, one copy per warp so that staging needs only __syncwarp
    int* es_b = (int*)(smem + (size_t)S * S4_STAGE_BYTES + 256) + ew * WN;
    const uint32_t tb = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * S4_NG * BN + cpart);
    long long acc[NACC];
    f32x2 sh[SUM_DF ? WN / 2 : 1], sl[SUM_DF ? WN / 2 : 1];  // running sums of column pairs
#pragma unroll
    for (int i = 0; i < NACC; ++i) acc[i] = 0;
#pragma unroll
    for (int i = 0; i < (SUM_DF ? WN / 2 : 1); ++i) sh[i] = sl[i] = 0;
    uint32_t fph = 0;
    bool ok = true;
    // Column i of the values that a lane holds for its half-warp's 16 rows (lane l of a
    // half-warp: columns l and 12 + l, l < 12).
    const int l16 = lane & 15, hw = lane & 16;
    S4Cursor cu{};
    for (cu.start(p, h); ok && cu.valid; cu.step(p, h)) {
      const bool kao = KIND == S_KAO || (KIND == S_JKAO && cu.opi());
      const S4Operands& op = p.op[KIND == S_JKAO ? cu.opi() : 0];
      const int rshift = op.rshift;
      const int n0 = (cu.nt() + h) * BN + cpart;  // this thread's first column
      const int ri = (cu.mt() << rshift) + (row & ((1 << rshift) - 1)), sub = row >> rshift;
      int ent, kb0, nkb;
      s4_kblocks(p, cu.b, ent, kb0, nkb);
      const int be = (ent << (7 - rshift)) + sub;  // this row's batch entry
      const bool rvalid = ri < op.nrows && be < op.nent;
      int ea = 0;
      int munu = 0;  // J^(q)
      int c3[2] = {0, 0};
      uint4 e6[3];  // HALF: the 24 columns' e6 as pairs of int16
      float2 cw[2] = {};
      // The exponents and weights of the batch: the loads run while its MMAs do.
      if (KIND != S_JMO) {
        __syncwarp();
        ea = rvalid ? __ldg(op.ea + (size_t)be * op.nrows + ri) : 0;
        if ((KIND == S_JAO || KIND == S_JKAO) && !kao) munu = rvalid ? __ldg(p.tri + ri) : 0;
        if constexpr (KIND != S_HALF) {
          if (lane < WN) {
            es_b[lane] = n0 + lane < op.ncols ? __ldg(op.eb + (op.batched ? (size_t)ent * op.ncols : 0) + n0 + lane) : 0;
          }
        }
        if constexpr (KIND == S_HALF || KIND == S_FOCK) {
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int c = n0 + 12 * k + l16;
            const bool v = l16 < 12 && c < p.m && be < op.nent;
            if constexpr (KIND == S_HALF) c3[k] = v ? __ldg(p.e3m + (size_t)be * p.m + c) : 0;
            else cw[k] = v ? __ldg(p.w + (size_t)be * p.m + c) : make_float2(0.f, 0.f);
          }
        }
        if constexpr (KIND == S_HALF) {
          const uint4* src = (const uint4*)(p.e6m + (size_t)(rvalid ? ri : 0) * p.e6ld + n0);
#pragma unroll
          for (int k = 0; k < 3; ++k) e6[k] = __ldg(src + k);
        }
        __syncwarp();
      }
      // The unit action: CN finished outputs (double-float, in column pairs) from column c of
      // the warpgroup on.  Columns past the last one are zero (the operands' boxes are
      // filled with zeros there), so the sums need no check.
      auto action = [&](const f32x2* hv, const f32x2* lv, int c) {
        if (KIND != S_FOCK && !rvalid) return;  // FOCK: every lane takes part in the shuffles
        const int c0 = n0 + c;
        if constexpr (KIND == S_FULLSQ) {
#pragma unroll
          for (int j = 0; j < CN / 2; ++j) {
            const f32x2 x = hv[j], nx = mul2(x, both2(-1.f));
            const f32x2 np = mul2(nx, x);  // -(x x) rounded
            const f32x2 pl = fma2(add2(x, x), lv[j], fma2(x, x, np));
            df_add2(sh[(c >> 1) + j], sl[(c >> 1) + j], mul2(np, both2(-1.f)), pl);
            if (STORE) {
              float a, b, al, bl;
              unpack2(x, a, b);
              unpack2(lv[j], al, bl);
              // along the rows, which are the lanes: a warp's store is 256 contiguous bytes
              double* dst = p.bfull + ((size_t)be * p.m + c0 + 2 * j) * p.m + ri;
              if (c0 + 2 * j < p.m) dst[0] = (double)a + (double)al;
              if (c0 + 2 * j + 1 < p.m) dst[p.m] = (double)b + (double)bl;
            }
          }
        } else if constexpr (KIND == S_FOCK) {
          // the weight is zero in invalid rows, and so are their sums
#pragma unroll
          for (int j = 0; j < CN / 2; ++j) {
            const int k = (c + 2 * j) / 12, src = hw + (c + 2 * j) % 12;
            const f32x2 wx = pack2(__shfl_sync(0xffffffffu, cw[k].x, src), __shfl_sync(0xffffffffu, cw[k].x, src + 1));
            const f32x2 wy = pack2(__shfl_sync(0xffffffffu, cw[k].y, src), __shfl_sync(0xffffffffu, cw[k].y, src + 1));
            const f32x2 x = hv[j], ph = mul2(x, wx);
            const f32x2 pl = add2(fma2(x, wx, mul2(ph, both2(-1.f))), fma2(x, wy, mul2(lv[j], wx)));
            df_add2(sh[(c >> 1) + j], sl[(c >> 1) + j], ph, pl);
          }
        } else if constexpr (KIND == S_CTR) {
#pragma unroll
          for (int j = 0; j < CN / 2; ++j) df_add2(sh[(c >> 1) + j], sl[(c >> 1) + j], hv[j], lv[j]);
        } else {
          float ho[CN], lo[CN];
#pragma unroll
          for (int j = 0; j < CN / 2; ++j) {
            unpack2(hv[j], ho[2 * j], ho[2 * j + 1]);
            unpack2(lv[j], lo[2 * j], lo[2 * j + 1]);
          }
          if (!kao) {
            // J^(q): packed row (mu, nu), columns q
            const int mu = munu >> 16, nu = munu & 0xFFFF;
#pragma unroll
            for (int j = 0; j < CN; ++j) {
              if (c0 + j < p.m) {
                const size_t o = ((size_t)(c0 + j) * p.nb + mu) * p.ldo + nu;
                p.ohi[o] = ho[j];
                p.olo[o] = lo[j];
              }
            }
          } else {
            // A thread's CN = 8 consecutive columns of one output row are one 32-byte
            // sector of hi and one of lo (ldo is a multiple of 8): two 16-byte vector
            // stores each instead of eight scattered 4-byte ones.
            const size_t o = ((size_t)(p.m + be) * p.nb + ri) * p.ldo + c0;
            if (c0 + CN <= p.nb) {
#pragma unroll
              for (int v = 0; v < CN / 4; ++v) {
                ((float4*)(p.ohi + o))[v] = make_float4(ho[4 * v], ho[4 * v + 1], ho[4 * v + 2], ho[4 * v + 3]);
                ((float4*)(p.olo + o))[v] = make_float4(lo[4 * v], lo[4 * v + 1], lo[4 * v + 2], lo[4 * v + 3]);
              }
            } else {
#pragma unroll
              for (int j = 0; j < CN; ++j) {
                if (c0 + j < p.nb) {
                  p.ohi[o + j] = ho[j];
                  p.olo[o + j] = lo[j];
                }
              }
            }
          }
        }
      };
      for (int ch = 0; ch < nkb; ch += CKB) {
        if (!mbar_wait(&accf[h], fph, abort_flag, p.status)) { ok = false; break; }
        fph ^= 1;
        tc_fence_after();
#pragma unroll
        for (int cb = 0; cb < NCB; ++cb) {
          // group g holds digit pairs with t + u = g; its weight is 2^(32 - 8 g) in units of 2^(ea+eb-46)
          uint32_t gr[S4_NG][CW];
          __syncwarp();
#pragma unroll
          for (int g = 0; g < S4_NG; ++g) tmem_ld_issue<CW>(tb + (uint32_t)(g * BN + cb * CW), gr[g]);
#pragma unroll
          for (int g = 0; g < S4_NG; ++g) tmem_wait<CW>(gr[g]);
          if (cb == NCB - 1) {
            // everything of this chunk is in registers: the half may be overwritten
            tc_fence_before();
            mbar_arrive(&acce[h]);
          }
          if constexpr (KIND == S_HALF) {
            // Half transform: one output integer at the finer of the two output scales
            // (exponents e3, e6), X = sum_g rint(G_g 2^(sigma - 8g)) in int32 per chunk
            // (see half_fold), without an int64 fold.  A unit of several K chunks adds
            // each chunk's integer to the one the same thread stored for the previous
            // chunk of this unit (a read of its own write, held in L2) and clamps the
            // sum, so no running sums occupy registers or local memory; each chunk adds
            // at most 2.5 units of rounding.  xf_to_digits_kernel derives both digit
            // layouts from the final integer.
            int* basef = p.x6 + ((size_t)be * p.m + n0 + cb * CW) * p.nbp + ri;
            int prev[ONE ? 1 : CW];
            if (!ONE && ch > 0) {
#pragma unroll
              for (int j = 0; j < CW; ++j) prev[j] = rvalid && n0 + cb * CW + j < p.m ? basef[(size_t)j * p.nbp] : 0;
            }
#pragma unroll
            for (int j = 0; j < CW; j += 2) {
              float sc[2];
#pragma unroll
              for (int d = 0; d < 2; ++d) {
                const int i = cb * CW + j + d;
                const int e3 = __shfl_sync(0xffffffffu, c3[i / 12], hw + i % 12);
                const uint4 v = e6[i / 8];
                const unsigned int pr = (i % 8) / 2 == 0 ? v.x : (i % 8) / 2 == 1 ? v.y : (i % 8) / 2 == 2 ? v.z : v.w;
                const int e6i = i % 2 ? (int)pr >> 16 : (int)(short)pr;
                sc[d] = exp2_int(ea - min(e3, e6i));
              }
              // T_g = (G_g 2^(-8g)) 2^sigma, both multiplications exact
              float T[2][S4_NG];
              const f32x2 s2 = pack2(sc[0], sc[1]);
#pragma unroll
              for (int g = 0; g < S4_NG; ++g) {
                f32x2 x = pack2(__uint_as_float(gr[g][j]), __uint_as_float(gr[g][j + 1]));
                if (g > 0) x = mul2(x, both2(exp2_int(-8 * g)));
                unpack2(mul2(x, s2), T[0][g], T[1][g]);
              }
#pragma unroll
              for (int d = 0; d < 2; ++d) {
                int X = half_fold(T[d]);
                if (!ONE && ch > 0) {
                  long long v = (long long)prev[j + d] + X;
                  v = v > (1LL << 30) ? (1LL << 30) : (v < -(1LL << 30) ? -(1LL << 30) : v);
                  X = (int)v;
                }
                if (rvalid && n0 + cb * CW + j + d < p.m) basef[(size_t)(j + d) * p.nbp] = X;
              }
            }
          } else if constexpr (NACC > 1) {
            // int64 fold: exact running sums over the K chunks of the batch (J_pq: of the unit)
#pragma unroll
            for (int j = 0; j < CW; ++j) {
              long long v = (KIND == S_JMO || ch > 0) ? acc[cb * CW + j] : 0;
#pragma unroll
              for (int g = 0; g < S4_NG; ++g) v = mad_wide(__float2int_rn(__uint_as_float(gr[g][j])), 32 - 8 * g, v);
              acc[cb * CW + j] = v;
            }
          } else {
            // A single-chunk batch converts its five group sums straight to double-float
            // pairs.  CTR converts every chunk and adds it to the unit's running sums (the
            // exponents are the same for the chunks of a batch, not across batches).
            f32x2 hv[CW / 2], lv[CW / 2];
            int k[CW];
#pragma unroll
            for (int j = 0; j < CW; j += 2) {
              f32x2 G[S4_NG];
#pragma unroll
              for (int g = 0; g < S4_NG; ++g) G[g] = pack2(__uint_as_float(gr[g][j]), __uint_as_float(gr[g][j + 1]));
              groups_to_df(G, hv[j / 2], lv[j / 2]);
            }
#pragma unroll
            for (int j = 0; j < CW; ++j) k[j] = ea + es_b[cb * CW + j] + 32 - S4_SHIFT;
            df_scale<CW / 2>(hv, lv, k);
            action(hv, lv, cb * CW);
          }
        }
      }
      if constexpr (NACC > 1 && KIND != S_JMO) {
        // the exact sums over the chunks are final
        if (ok) {
#pragma unroll
          for (int c = 0; c < WN; c += CN) {
            f32x2 hv[CN / 2], lv[CN / 2];
            int k[CN];
#pragma unroll
            for (int j = 0; j < CN; j += 2) {
              float h0, l0, h1, l1;
              ll_to_df(acc[c + j], h0, l0);
              ll_to_df(acc[c + j + 1], h1, l1);
              hv[j / 2] = pack2(h0, h1);
              lv[j / 2] = pack2(l0, l1);
            }
#pragma unroll
            for (int j = 0; j < CN; ++j) k[j] = ea + es_b[c + j] - S4_SHIFT;
            df_scale<CN / 2>(hv, lv, k);
            action(hv, lv, c);
          }
        }
      }
      // ---- the unit's sums, one partial per (slot, group of rows) ----
      if constexpr (SUMS) {
        if (!cu.last()) continue;
        if (ok && ri < op.nrows) {
          auto sum_of = [&](int i) {
            float a, b, c, d;
            unpack2(sh[SUM_DF ? i / 2 : 0], a, b);
            unpack2(sl[SUM_DF ? i / 2 : 0], c, d);
            return i % 2 ? make_float2(b, d) : make_float2(a, c);
          };
          const size_t sl0 = ((size_t)cu.slot() << (7 - rshift)) + sub;
          if constexpr (KIND == S_JMO) {
            long long* dst = (long long*)p.partial + (sl0 * p.prow + ri) * p.pcol;
#pragma unroll
            for (int i = 0; i < WN; ++i) {
              if (n0 + i < p.pcol) dst[n0 + i] = acc[NACC > 1 ? i : 0];
            }
          } else if constexpr (KIND == S_FULLSQ) {
            float2* dst = (float2*)p.partial + (sl0 * p.prow + ri) * p.pcol;
#pragma unroll
            for (int i = 0; i < WN; ++i) {
              if (n0 + i < p.pcol) dst[n0 + i] = sum_of(i);
            }
          } else {  // rows mu, columns p: partials [p][mu], consecutive mu per warp
            float2* dst = (float2*)p.partial + sl0 * p.prow * p.pcol + ri;
#pragma unroll
            for (int i = 0; i < WN; ++i) {
              if (n0 + i < p.prow) dst[(size_t)(n0 + i) * p.pcol] = sum_of(i);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = 0;
#pragma unroll
        for (int i = 0; i < (SUM_DF ? WN / 2 : 1); ++i) sh[i] = sl[i] = 0;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, S4_TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// digitisation and bound kernels
// ---------------------------------------------------------------------------
// |x| as an integer that orders like it.
__device__ __forceinline__ unsigned long long mag64(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// __double2int_rn(x 2^(31 - e)) for |x| < 2^(e-1), e = expo_of of the row, by integer
// instructions: FP64 multiplies and converts two lanes a clock per SM, which made the one-time
// digitisations of B (387 MB at C10H20) 915 and 343 us; 299 and 182 so, with the maxima that
// two more passes took (387 us).
__device__ __forceinline__ int fixed32(double x, int e) {
  const unsigned long long mag = mag64(x);
  const int f = max((int)(mag >> 52), 1);
  const unsigned long long m = mag >> 52 ? (mag & 0xFFFFFFFFFFFFFull) | 1ull << 52 : mag;
  const int sh = 1044 + e - f;  // x = m 2^(f - 1075); sh >= 23
  if (sh > 60 || sh < 1) return 0;  // below half a unit (or a row that is not finite)
  const unsigned int r = (unsigned int)((m + (1ull << (sh - 1)) - 1 + ((m >> sh) & 1)) >> sh);  // ties to even
  return x < 0.0 ? -(int)r : (int)r;
}

// Rows of an FP64 matrix (element (r, k) at X[r cols + k]) -> interleaved digits
// [(r*4 + t)*ldp + k] with the row's exact exponent, and the row's largest magnitude rounded
// up.  One warp per row, neighbouring pairs of k per lane (ldp is even: a pair may end in the
// padding).
__global__ void __launch_bounds__(256) slice_f64_kernel(const double* __restrict__ X, long long rows, int cols,
                                                        __nv_bfloat16* __restrict__ planes, int ldp,
                                                        int* __restrict__ exps, float* __restrict__ rmax) {
  const long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32;
  const int lane = threadIdx.x % 32;
  if (r >= rows) return;
  const double* x = X + r * cols;
  unsigned long long mx = 0;
#pragma unroll 4
  for (int k = lane; k < cols; k += 32) mx = max(mx, mag64(x[k]));
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const double v = __longlong_as_double((long long)mx);
  const int e = expo_of(v);
  if (lane == 0) {
    exps[r] = e;
    rmax[r] = __double2float_ru(v);
  }
  __nv_bfloat16* out = planes + (size_t)r * 4 * ldp;
#pragma unroll 2
  for (int k = 2 * lane; k < cols; k += 64) {
    __nv_bfloat162 d[4];
    digits_bf16x2(fixed32(x[k], e), k + 1 < cols ? fixed32(x[k + 1], e) : 0, d);
#pragma unroll
    for (int t = 0; t < 4; ++t) *(__nv_bfloat162*)(out + (size_t)t * ldp + k) = d[t];
  }
}

// Digit rows over P of the upper triangle of a symmetric tensor X [P][n][n] (FP64): packed
// row r = (mu, nu), mu <= nu (tri[r] = mu << 16 | nu), -> out[(r*4 + t)*ldp + P] with the
// row's exact exponent.  Consecutive packed rows are consecutive nu, so a block of 32
// reads 256 contiguous bytes per P (and maxB[mu][nu] = max_P |X| rounded up); one pass for the maxima, a second that rounds and
// turns 32 x 32 (P, r) blocks around in shared memory, so that the digit rows are written
// along P (a warp per row reads 8 bytes of every sector instead).
__global__ void __launch_bounds__(256) slice_tri_kernel(const double* __restrict__ X, const int* __restrict__ tri,
                                                        int rows, int n, int nx, __nv_bfloat16* __restrict__ planes,
                                                        int ldp, int* __restrict__ exps, float* __restrict__ maxB) {
  __shared__ unsigned long long red[8][32];
  __shared__ int tile[32][33];
  __shared__ int es[32];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int r0 = blockIdx.x * 32, r = r0 + tx;
  const bool rv = r < rows;
  const int mn = rv ? tri[r] : 0;
  const long long n2 = (long long)n * n;
  const double* x = X + (long long)(mn >> 16) * n + (mn & 0xFFFF);
  unsigned long long mx = 0;
  if (rv) {
#pragma unroll 8
    for (int P = ty; P < nx; P += 8) mx = max(mx, mag64(x[P * n2]));
  }
  red[ty][tx] = mx;
  __syncthreads();
  if (ty == 0) {
#pragma unroll
    for (int y = 1; y < 8; ++y) mx = max(mx, red[y][tx]);
    const double v = __longlong_as_double((long long)mx);
    const int e = expo_of(v);
    es[tx] = e;
    if (rv) {
      exps[r] = e;
      const float f = __double2float_ru(v);
      maxB[(size_t)(mn >> 16) * n + (mn & 0xFFFF)] = f;
      maxB[(size_t)(mn & 0xFFFF) * n + (mn >> 16)] = f;
    }
  }
  __syncthreads();
  const int e = es[tx];
  for (int P0 = 0; P0 < nx; P0 += 32) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int P = P0 + ty + 8 * k;
      tile[ty + 8 * k][tx] = rv && P < nx ? fixed32(x[P * n2], e) : 0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int rr = ty + 8 * k, P = P0 + tx;
      if (r0 + rr < rows && P < nx) {
        __nv_bfloat16 d[4];
        digits_bf16(tile[tx][rr], d);
        __nv_bfloat16* o = planes + (size_t)(r0 + rr) * 4 * ldp + P;
#pragma unroll
        for (int t = 0; t < 4; ++t) o[(size_t)t * ldp] = d[t];
      }
    }
    __syncthreads();
  }
}

// The per-iteration form of slice_f64_kernel (unit column stride): one block per
// row, so that a row's loads are spread over many threads and its FP64 work over
// the SMs.  Rows r in [rows, rows_df) only write their double-float copy.
constexpr int SLICE_ROWS_THREADS = 128;
__global__ void __launch_bounds__(SLICE_ROWS_THREADS) slice_rows_kernel(const double* __restrict__ X, int rows,
                                                                        int cols, long long rs,
                                                                        __nv_bfloat16* __restrict__ planes, int ldp,
                                                                        int* __restrict__ exps, float* absout,
                                                                        float* absT, float2* dfout) {
  pdl_entry();
  __shared__ double wmax[SLICE_ROWS_THREADS / 32];
  __shared__ int se;
  const int r = blockIdx.x, tid = threadIdx.x;
  const double* x = X + (long long)r * rs;
  if (r >= rows) {
    for (int k = tid; k < cols; k += SLICE_ROWS_THREADS) dfout[(long long)r * cols + k] = to_df(x[k]);
    return;
  }
  double mx = 0.0;
#pragma unroll 4
  for (int k = tid; k < cols; k += SLICE_ROWS_THREADS) mx = fmax(mx, fabs(x[k]));
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((tid & 31) == 0) wmax[tid >> 5] = mx;
  __syncthreads();
  if (tid == 0) {
    double m2 = wmax[0];
    for (int w = 1; w < SLICE_ROWS_THREADS / 32; ++w) m2 = fmax(m2, wmax[w]);
    se = expo_of(m2);
    exps[r] = se;
  }
  __syncthreads();
  const int e = se;
  __nv_bfloat16* out = planes + (size_t)r * 4 * ldp;
#pragma unroll 4
  for (int k = tid; k < cols; k += SLICE_ROWS_THREADS) {
    const double v = x[k];
    __nv_bfloat16 d[4];
    digits_bf16(__double2int_rn(scale_pow2(v, 31 - e)), d);
#pragma unroll
    for (int t = 0; t < 4; ++t) out[t * ldp + k] = d[t];
    if (absout) absout[(long long)r * cols + k] = (float)fabs(v);
    if (absT) absT[(long long)k * rows + r] = (float)fabs(v);
    if (dfout) dfout[(long long)r * cols + k] = to_df(v);
  }
}

// FP64 -> double-float pairs, elementwise.
__global__ void to_df_kernel(const double* __restrict__ x, long long n, float2* __restrict__ out) {
  pdl_entry();
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) out[i] = to_df(x[i]);
}

__device__ __forceinline__ float scale_pow2f(float x, int k) {
  return (k >= -126 && k <= 127) ? x * exp2_int(k) : ldexpf(x, k);
}
__device__ __forceinline__ int pair_to_int(float h, float l, int k) {
  const float hs = scale_pow2f(h, k), ls = scale_pow2f(l, k);  // |hs| < 2^30
  const float ih = rintf(hs);
  return __float2int_rn(ih) + __float2int_rn((hs - ih) + ls);
}
// J^(q) and K^(q) as digit rows, in two passes over the upper triangles that their GEMMs
// leave (matrix z of 2 N_O, double-float [z][n][ld], valid for nu >= mu): the maxima of the
// rows of the whole symmetric matrices, then the digits.  The lower triangles are never
// written as numbers, so the passes move 4 + 8 bytes of every upper element and the 8 of
// every digit row's element.  C20H40: 1200 us against 2440 for two mirror passes and a
// split over whole rows; with J^(q)'s rows packed to the triangle (5200 -> 4050 us: no
// 128-row block straddles it) the orbital half of the iteration went from 13.6 to 10.0
// ms.  (Gathering whole rows in shared memory in one pass instead
// took 2830 us at C20H40: too few loads in flight.)
//
// Maxima: rowmax[z][mu] (the FP32 pattern of a non-negative value, zero on entry) over row
// mu and column mu.  A block takes 32 rows of one matrix and keeps four columns' maxima per
// thread.  The low parts lie below the inflation of expo_of_inflated.
__global__ void __launch_bounds__(256) sym_max_kernel(const float* __restrict__ hi, int n, int ld,
                                                      unsigned int* __restrict__ rowmax) {
  pdl_entry();
  __shared__ unsigned int rm[32];
  const int mu0 = blockIdx.x * 32, lane = threadIdx.x % 32;
  if (threadIdx.x < 32) rm[threadIdx.x] = 0;
  __syncthreads();
  const float* h = hi + ((size_t)blockIdx.y * n + mu0) * ld;
  unsigned int* out = rowmax + (size_t)blockIdx.y * n;
  const int nr = min(32, n - mu0), c0 = mu0 / 4, c1 = (n + 3) / 4;
  for (int cw = c0 + (threadIdx.x & ~31); cw < c1; cw += 256) {  // a warp's 32 groups of four columns
    const int c = cw + lane, nu = 4 * c;
    float cm[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
    for (int r = 0; r < nr; ++r) {
      float4 v = c < c1 ? __ldg((const float4*)(h + (size_t)r * ld) + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      const int mu = mu0 + r;
      const float x[4] = {v.x, v.y, v.z, v.w};
      float m = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float a = (nu + j >= mu && nu + j < n) ? fabsf(x[j]) : 0.f;
        cm[j] = fmaxf(cm[j], a);
        m = fmaxf(m, a);
      }
      const unsigned int wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
      if (lane == 0) atomicMax(&rm[r], wm);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (nu + j < n && cm[j] > 0.f) atomicMax(out + nu + j, __float_as_uint(cm[j]));
  }
  __syncthreads();
  if (threadIdx.x < nr) atomicMax(out + mu0 + threadIdx.x, rm[threadIdx.x]);
}

// Digits: planes[((z n + mu) 4 + t) ldp + nu] and the row exponents.  A block takes one
// 64 x 64 tile on or above the diagonal: the digit rows of its rows mu, and through shared
// memory those of its columns nu (each value rounded at its own row's exponent).
__global__ void __launch_bounds__(256) sym_digits_kernel(const float* __restrict__ hi, const float* __restrict__ lo,
                                                         int n, int ld, const unsigned int* __restrict__ rowmax,
                                                         __nv_bfloat16* __restrict__ planes, int ldp,
                                                         int* __restrict__ exps) {
  pdl_entry();
  __shared__ float th[64][65], tl[64][65];
  __shared__ int er[64], ec[64];
  // tile (bi <= bj) of the block: the t-th of the upper triangle, rows of tiles first
  const int T = (n + 63) / 64;
  int bi = 0, t = blockIdx.x;
  while (t >= T - bi) t -= T - bi, ++bi;
  const int bj = bi + t, mu0 = bi * 64, nu0 = bj * 64;
  const size_t base = (size_t)blockIdx.y * n;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  if (threadIdx.x < 128) {
    const int i = threadIdx.x % 64, mu = (threadIdx.x < 64 ? mu0 : nu0) + i;
    const int e = mu < n ? expo_of_inflated(__uint_as_float(rowmax[base + mu])) : 0;
    (threadIdx.x < 64 ? er : ec)[i] = e;
    if (bi == bj && threadIdx.x < 64 && mu < n) exps[base + mu] = e;
  }
  const int c = 2 * tx;
  float2 hv[8], lv[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int mu = mu0 + ty + 8 * i, nu = nu0 + c;
    hv[i] = lv[i] = make_float2(0.f, 0.f);
    if (mu < n && nu < n) {  // ld is a multiple of 8: the pair lies within the row
      hv[i] = *(const float2*)(hi + (base + mu) * ld + nu);
      lv[i] = *(const float2*)(lo + (base + mu) * ld + nu);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = ty + 8 * i;
    th[r][c] = hv[i].x;
    th[r][c + 1] = hv[i].y;
    tl[r][c] = lv[i].x;
    tl[r][c + 1] = lv[i].y;
  }
  __syncthreads();
  if (bi == bj) {  // the diagonal tile's lower half from its upper one
    for (int i = threadIdx.x; i < 64 * 64; i += 256) {
      const int r = i / 64, k = i % 64;
      if (k < r) {
        th[r][k] = th[k][r];
        tl[r][k] = tl[k][r];
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = ty + 8 * i;
      hv[i] = make_float2(th[r][c], th[r][c + 1]);
      lv[i] = make_float2(tl[r][c], tl[r][c + 1]);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = ty + 8 * i, mu = mu0 + r, nu = nu0 + c;
    if (mu < n && nu < n) {
      const int k = 31 - er[r];
      __nv_bfloat162 dd[4];
      digits_bf16x2(pair_to_int(hv[i].x, lv[i].x, k), pair_to_int(hv[i].y, lv[i].y, k), dd);
      __nv_bfloat16* o = planes + (base + mu) * 4 * ldp + nu;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if (nu + 1 < n) *(__nv_bfloat162*)(o + (size_t)p * ldp) = dd[p];
        else o[(size_t)p * ldp] = dd[p].x;
      }
    }
  }
  if (bi == bj) return;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = ty + 8 * i, nu = nu0 + r, mu = mu0 + c;  // mu0 + 63 < n in a tile above the diagonal
    if (nu < n) {
      const int k = 31 - ec[r];
      __nv_bfloat162 dd[4];
      digits_bf16x2(pair_to_int(th[c][r], tl[c][r], k), pair_to_int(th[c + 1][r], tl[c + 1][r], k), dd);
      __nv_bfloat16* o = planes + (base + nu) * 4 * ldp + mu;
#pragma unroll
      for (int p = 0; p < 4; ++p) *(__nv_bfloat162*)(o + (size_t)p * ldp) = dd[p];
    }
  }
}

// Both passes in one for matrices whose triangle fits shared memory (up to 240 functions): a
// block per matrix gathers it once, so the numbers are read once and a launch is saved.
// Split at C6H12 / C10H20 / the square, with its launches (us): two passes 45 / 117 / 19, this
// 25 / 92 / 7.  (At 240 functions a block fills an SM and nothing overlaps its loads; larger
// matrices do not fit.)
__global__ void __launch_bounds__(1024) sym_split_kernel(const float* __restrict__ hi, const float* __restrict__ lo, int n,
                                                         int ld, __nv_bfloat16* __restrict__ planes, int ldp,
                                                         int* __restrict__ exps) {
  extern __shared__ float2 tri[];  // row mu from nu = mu on, at mu n - mu (mu - 1) / 2
  int* es = (int*)(tri + n * (n + 1) / 2);
  pdl_entry();
  const size_t base = (size_t)blockIdx.x * n;
  const int T = blockDim.x, tid = threadIdx.x, w = (n + 3) / 4;
  {
    // groups of four from the diagonal's on; rows mu and n - 1 - mu share a line of w + 2
    const int L = w + 2, total = (n + 1) / 2 * L;
    const unsigned int inv = 0xFFFFFFFFu / (unsigned int)L + 1;  // exact quotients below 2^32 / L
    const float4* h4 = (const float4*)(hi + base * ld);
    const float4* l4 = (const float4*)(lo + base * ld);
    constexpr int U = 4;
    for (int i0 = tid; i0 < total; i0 += U * T) {
      float4 h[U], l[U];
      int mu[U], nu[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * T, line = (int)__umulhi((unsigned int)i, inv);
        int g = i - line * L;
        const bool past = g >= w - line / 4;  // the end of row `line`
        if (past) g -= w - line / 4;
        mu[u] = past ? n - 1 - line : line;
        nu[u] = n;
        g += mu[u] / 4;
        if (i < total && g < w && (!past || mu[u] > line)) {
          nu[u] = 4 * g;
          h[u] = __ldg(h4 + mu[u] * (ld / 4) + g);
          l[u] = __ldg(l4 + mu[u] * (ld / 4) + g);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float2* row = tri + mu[u] * n - mu[u] * (mu[u] - 1) / 2 - mu[u];
        const float hv[4] = {h[u].x, h[u].y, h[u].z, h[u].w}, lv[4] = {l[u].x, l[u].y, l[u].z, l[u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (nu[u] + j >= mu[u] && nu[u] + j < n) row[nu[u] + j] = make_float2(hv[j], lv[j]);
      }
    }
  }
  __syncthreads();
  // row maxima: four lanes per row, over its column above the diagonal and its row
  for (int g0 = 0; g0 < n; g0 += T / 4) {
    const int mu = g0 + tid / 4, q = tid % 4;
    float mx = 0.f;
    if (mu < n) {
      for (int k = q; k < mu; k += 4) mx = fmaxf(mx, fabsf(tri[k * n - k * (k - 1) / 2 + mu - k].x));
      const float2* row = tri + mu * n - mu * (mu - 1) / 2 - mu;
      for (int k = mu + q; k < n; k += 4) mx = fmaxf(mx, fabsf(row[k].x));
    }
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    if (mu < n && q == 0) {
      const int e = expo_of_inflated(mx);
      es[mu] = e;
      exps[base + mu] = e;
    }
  }
  __syncthreads();
  // digits, four neighbouring nu per thread (the row's padding takes zeros)
  const int total = n * w;
  const unsigned int inv = w > 1 ? 0xFFFFFFFFu / (unsigned int)w + 1 : 0;
  for (int i = tid; i < total; i += T) {
    const int mu = w > 1 ? (int)__umulhi((unsigned int)i, inv) : i, nu = 4 * (i - mu * w), k = 31 - es[mu];
    const float2* row = tri + mu * n - mu * (mu - 1) / 2 - mu;
    int v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = nu + j;
      float2 x = make_float2(0.f, 0.f);
      if (c < n) x = c >= mu ? row[c] : tri[c * n - c * (c - 1) / 2 + mu - c];
      v[j] = pair_to_int(x.x, x.y, k);
    }
    __nv_bfloat162 d0[4], d1[4];
    digits_bf16x2(v[0], v[1], d0);
    digits_bf16x2(v[2], v[3], d1);
    __nv_bfloat16* o = planes + (base + mu) * 4 * ldp + nu;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      uint2 d;
      d.x = *(const unsigned int*)&d0[p];
      d.y = *(const unsigned int*)&d1[p];
      *(uint2*)(o + (size_t)p * ldp) = d;
    }
  }
}

static size_t sym_split_smem(int n) { return ((size_t)n * (n + 1) / 2) * 8 + (size_t)n * 4; }

// Upper bounds on |b^P_{p nu}| (Table 2/3 step 2), FP32 sums inflated by (1 + 2^-16):
//   e3[P][p] = expo(sum_mu rmaxB[P][mu] |C_{mu p}|)   (rows (P,p) of the full-transform operand)
//   e6[p][nu] = expo(sum_mu |C_{mu p}| maxB[mu][nu])   (rows (p,nu) of the K^(p) operand)
// and, for the half transform's output scale, either one less the exponent of C's row p
// and 17 (e3m [P][p], and e6m [nu][p] as int16).
// Both are out[i][j] = expo(sum_k A[i][k] B[k][j]) over a small FP32 product: 16 x 16
// outputs per block, K staged through shared memory in slices of 64, every sum
// taken in k order with one FMA chain (the bounds do not depend on the launch).
constexpr int BOUND_TILE = 16, BOUND_KC = 64;
struct BoundJob {
  int M, N;
  const float* A;
  int lda;
  const float* B;
  int ldb;
  int* out;
  int ldo;
  int* out_e3m;
  short* out_e6m;
  int ld6, bx, blocks;  // blocks along N, and in all
};
// Both products in one launch (beside each other on two streams they cost a fork and a join on
// the path to the half transform; small systems wait for little else).
__global__ void __launch_bounds__(256) bound_kernel(const __grid_constant__ BoundJob job3, const __grid_constant__ BoundJob job6,
                                                    int K, const int* __restrict__ eC) {
  pdl_entry();
  const bool second = (int)blockIdx.x >= job3.blocks;
  const BoundJob& job = second ? job6 : job3;
  const int blk = second ? (int)blockIdx.x - job3.blocks : (int)blockIdx.x;
  const int M = job.M, N = job.N, lda = job.lda, ldb = job.ldb, ldo = job.ldo, ld6 = job.ld6;
  const float* __restrict__ A = job.A;
  const float* __restrict__ B = job.B;
  int* __restrict__ out = job.out;
  int* __restrict__ out_e3m = job.out_e3m;
  short* __restrict__ out_e6m = job.out_e6m;
  __shared__ float As[BOUND_TILE][BOUND_KC + 1];
  __shared__ float Bs[BOUND_KC][BOUND_TILE + 1];
  __shared__ short es[BOUND_TILE][BOUND_TILE + 2];
  const int tid = threadIdx.x, tx = tid % BOUND_TILE, ty = tid / BOUND_TILE;
  const int i0 = blk / job.bx * BOUND_TILE, j0 = blk % job.bx * BOUND_TILE;
  float acc = 0.f;
  for (int k0 = 0; k0 < K; k0 += BOUND_KC) {
#pragma unroll
    for (int u = 0; u < BOUND_TILE * BOUND_KC / 256; ++u) {
      const int idx = tid + 256 * u;
      const int ar = idx / BOUND_KC, ac = idx % BOUND_KC;  // A: row i0 + ar, column k0 + ac
      As[ar][ac] = (i0 + ar < M && k0 + ac < K) ? A[(size_t)(i0 + ar) * lda + k0 + ac] : 0.f;
      const int br = idx / BOUND_TILE, bc = idx % BOUND_TILE;  // B: row k0 + br, column j0 + bc
      Bs[br][bc] = (k0 + br < K && j0 + bc < N) ? B[(size_t)(k0 + br) * ldb + j0 + bc] : 0.f;
    }
    __syncthreads();
    const int kn = K - k0 < BOUND_KC ? K - k0 : BOUND_KC;
    for (int kk = 0; kk < kn; ++kk) acc = fmaf(As[ty][kk], Bs[kk][tx], acc);
    __syncthreads();
  }
  if (i0 + ty < M && j0 + tx < N) {
    const int e = expo_of_inflated(acc);
    out[(size_t)(i0 + ty) * ldo + j0 + tx] = e;
    if (out_e3m) out_e3m[(size_t)(i0 + ty) * ldo + j0 + tx] = e - eC[j0 + tx] - 17;
    // transposed, rows nu: a block's 16 p are 32 contiguous bytes of each of its rows
    if (out_e6m) es[tx][ty] = (short)(e - eC[i0 + ty] - 17);
  }
  if (out_e6m) {
    __syncthreads();
    if (j0 + ty < N && i0 + tx < M) out_e6m[(size_t)(j0 + ty) * ld6 + i0 + tx] = es[ty][tx];
  }
}

// J_pq = 2^(ed_p + ed_q - 46) x (sum over splits of the exact int64 partials).
// Columns from `split` on belong to tiles of one half, whose units take more batches
// and write fewer partials.
__global__ void reduce_jmo_kernel(const long long* partial, S4Slots ns, int m, const int* ed, double* J) {
  pdl_entry();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m * m) return;
  long long s = 0;
#pragma unroll 8
  for (int k = 0; k < (i % m < ns.split ? ns.pair : ns.single); ++k) s += partial[(size_t)k * m * m + i];
  J[i] = ldexp((double)s, ed[i / m] + ed[i % m] - S4_SHIFT);
}

// Sum over the units of double-float partials, in double-float arithmetic (FP64 only
// for the final value).  Without outdf: out[i] = the sum (FP64).  With outdf: the
// [rows = p][cols = mu] partials of F^(p) C_p, written as the double-float Y^T
// [p][mu] with n_p (H C)^T added (HCt double-float).
__global__ void __launch_bounds__(256) reduce_df_kernel(const float2* partial, S4Slots ns, int rows, int cols,
                                                       double* out, float2* outdf, const double* n,
                                                       const float2* HCt) {
  pdl_entry();
  // 32 outputs per block, their partials dealt to 8 thread rows (split k to row
  // k % 8), each row summing its share in split order; the 8 row sums are then
  // added in row order, so the result does not depend on the launch beyond that
  // fixed order.
  __shared__ float2 part[8][32];
  const long long rc = (long long)rows * cols;
  const long long i = blockIdx.x * 32LL + threadIdx.x;
  float sh = 0.f, sl = 0.f;
  if (i < rc) {
    // the tile's column index is q for the squares, p (the row here) for F^(p) C_p
    const int pos = outdf ? (int)(i / cols) : (int)(i % cols);
    const int nsplit = pos < ns.split ? ns.pair : ns.single;
    for (int k = threadIdx.y; k < nsplit; k += 8) {
      const float2 v = partial[(size_t)k * rc + i];
      df_add(sh, sl, v.x, v.y);
    }
  }
  part[threadIdx.y][threadIdx.x] = make_float2(sh, sl);
  __syncthreads();
  if (threadIdx.y != 0 || i >= rc) return;
  float th = part[0][threadIdx.x].x, tl = part[0][threadIdx.x].y;
#pragma unroll
  for (int y = 1; y < 8; ++y) df_add(th, tl, part[y][threadIdx.x].x, part[y][threadIdx.x].y);
  if (outdf) {
    const float2 np = to_df(n[i / cols]), h = HCt[i];
    const float ph = np.x * h.x;
    const float pl = fmaf(np.x, h.x, -ph) + fmaf(np.x, h.y, np.y * h.x);
    df_add(th, tl, ph, pl);
    outdf[i] = make_float2(th, tl);
  } else {
    out[i] = (double)th + (double)tl;
  }
}

// The contracted Lagrangian's first operand,
//   X^P_qp = [q = p] w_pP - B_pq b^P_qp,  w_pP = sum_r A_pr b^P_rr,
// as digit rows (q, p) over P with the row's exact exponent: X digits
// [q][p][4][nxp], eX[q][p].  b^P_qp from bf [P][p][q] (FP64), w [p][P], B [p][q].
// Block (32, 8) per orbital p and 32 consecutive q: one pass for the row maxima (of |b|
// itself off the diagonal: rounding is monotonic, so max |B b| = |B max |b||), a second that
// rounds each value to its integer, turns a 64 x 32 (P, q) block around in shared memory and
// writes each digit row's 64 consecutive P at once.  One FP64 product per element and eight
// loads in flight per thread: with FP64 maxima, scalings and conversions in both passes it
// took 3.66 ms at 320 orbitals and 1680 auxiliary functions, 1.84 so (4.1 GB, read in pieces of
// 256 bytes, N_Omega^2 elements apart).
__global__ void __launch_bounds__(256) ctr_digits_kernel(const double* __restrict__ bf, const double* __restrict__ Bc,
                                                         const double* __restrict__ w, int m, int nx, int nxp,
                                                         __nv_bfloat16* __restrict__ Xd, int* __restrict__ eX) {
  pdl_entry();
  constexpr int TP = 64;
  __shared__ unsigned long long red[8][32];
  __shared__ int tile[TP][33];
  __shared__ int es[32];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int p = blockIdx.y, q0 = blockIdx.x * 32, q = q0 + tx;
  const bool qv = q < m;
  const double bqp = qv ? Bc[(size_t)p * m + q] : 0.0;
  const bool diag = qv && p == q;
  const double* b = bf + (size_t)p * m + q;
  const size_t m2 = (size_t)m * m;
  unsigned long long mx = 0;
  if (diag) {
    for (int P = ty; P < nx; P += 8) mx = max(mx, mag64(w[(size_t)p * nx + P] - bqp * b[P * m2]));
  } else if (qv) {
#pragma unroll 8
    for (int P = ty; P < nx; P += 8) mx = max(mx, mag64(__ldg(b + P * m2)));
    mx = mag64(bqp * __longlong_as_double((long long)mx));
  }
  red[ty][tx] = mx;
  __syncthreads();
  if (ty == 0) {
#pragma unroll
    for (int y = 1; y < 8; ++y) mx = max(mx, red[y][tx]);
    const int e = expo_of(__longlong_as_double((long long)mx));
    es[tx] = e;
    if (qv) eX[(size_t)q * m + p] = e;
  }
  __syncthreads();
  const int e = es[tx];
  for (int P0 = 0; P0 < nx; P0 += TP) {
    double v[TP / 8];
#pragma unroll
    for (int k = 0; k < TP / 8; ++k) {
      const int P = P0 + ty + 8 * k;
      v[k] = qv && P < nx ? __ldg(b + P * m2) : 0.0;
    }
#pragma unroll
    for (int k = 0; k < TP / 8; ++k) {
      const int P = P0 + ty + 8 * k;
      double x = -bqp * v[k];
      if (diag && P < nx) x = w[(size_t)p * nx + P] - bqp * v[k];
      tile[ty + 8 * k][tx] = fixed32(x, e);
    }
    __syncthreads();
    // pairs of P: past nx the tile holds zeros, and the row's padding takes one at most
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int pr = ty + 8 * k, P = P0 + 2 * tx;
      if (q0 + pr < m && P < nx) {
        __nv_bfloat162 d[4];
        digits_bf16x2(tile[2 * tx][pr], tile[2 * tx + 1][pr], d);
        __nv_bfloat16* o = Xd + ((size_t)(q0 + pr) * m + p) * 4 * nxp + P;
#pragma unroll
        for (int t = 0; t < 4; ++t) *(__nv_bfloat162*)(o + (size_t)t * nxp) = d[t];
      }
    }
    __syncthreads();
  }
}

// out[i][j] = sum_k A[i][k] B[j][k] in double-float arithmetic: each product as
// an FP32 pair (about 2^-46 relative), the high parts summed with TwoSum in k
// order and the low parts and rounding errors collected beside them.  A and B are
// double-float; out double-float or FP64.  The small products of the energy row
// (H C, lambda = Y^T C) run here rather than in DFMA, whose rate is a small
// fraction of FP32's on this part.  16 x 16 outputs per block, K staged through
// shared memory in slices of 64, the loads of a slice issued together.
__device__ __forceinline__ void df_store(float2& o, float h, float l) { o = make_float2(h, l); }
__device__ __forceinline__ void df_store(double& o, float h, float l) { o = (double)h + (double)l; }

constexpr int DFG_KC = 64, DFG_TI = 16, DFG_TJ = 16, DFG_THREADS = DFG_TI * DFG_TJ;
__device__ __forceinline__ float2 df_load(float2 x) { return x; }
__device__ __forceinline__ float2 df_load(double x) { return to_df(x); }
// A from FP64 (split as it is read) saves to_df_kernel's launch; every column block repeats the
// splits, on the FP64 pipe, so it pays up to DFG_FP64_A functions.
constexpr int DFG_FP64_A = 160;
template <typename TO, typename TA>
__global__ void __launch_bounds__(DFG_THREADS) df_gemm_nt_kernel(int M, int N, int K, const TA* __restrict__ A,
                                                                 int lda, const float2* __restrict__ B, int ldb,
                                                                 TO* __restrict__ out, int ldo) {
  pdl_entry();
  __shared__ float2 As[DFG_TI][DFG_KC + 1];  // [i][k]
  __shared__ float2 Bs[DFG_KC][DFG_TJ + 1];  // [k][j]
  const int tid = threadIdx.x, tx = tid % DFG_TJ, ty = tid / DFG_TJ;
  const int i0 = blockIdx.y * DFG_TI, j0 = blockIdx.x * DFG_TJ;
  constexpr int NA = DFG_TI * DFG_KC / DFG_THREADS, NB = DFG_TJ * DFG_KC / DFG_THREADS;
  float sum = 0.f, cmp = 0.f;
  for (int k0 = 0; k0 < K; k0 += DFG_KC) {
    float2 av[NA], bv[NB];
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int idx = tid + DFG_THREADS * u, r = idx / DFG_KC, c = idx % DFG_KC;
      av[u] = (i0 + r < M && k0 + c < K) ? df_load(A[(size_t)(i0 + r) * lda + k0 + c]) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int idx = tid + DFG_THREADS * u, r = idx / DFG_KC, c = idx % DFG_KC;
      bv[u] = (j0 + r < N && k0 + c < K) ? B[(size_t)(j0 + r) * ldb + k0 + c] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int idx = tid + DFG_THREADS * u;
      As[idx / DFG_KC][idx % DFG_KC] = av[u];
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int idx = tid + DFG_THREADS * u;
      Bs[idx % DFG_KC][idx / DFG_KC] = bv[u];
    }
    __syncthreads();
    const int kn = K - k0 < DFG_KC ? K - k0 : DFG_KC;
#pragma unroll 8
    for (int kk = 0; kk < kn; ++kk) {
      const float2 a = As[ty][kk], b = Bs[kk][tx];
      const float ph = a.x * b.x;
      const float pl = fmaf(a.x, b.x, -ph) + fmaf(a.x, b.y, a.y * b.x);
      float ns, e;
      two_sum_f(sum, ph, ns, e);
      sum = ns;
      cmp += e + pl;
    }
    __syncthreads();
  }
  if (i0 + ty < M && j0 + tx < N) {
    const float h = sum + cmp;
    df_store(out[(size_t)(i0 + ty) * ldo + j0 + tx], h, cmp - (h - sum));
  }
}

// E = E_nuc + sum_p (n_p H_pp + lambda_pp).  One warp per p: H_pp = C_p . (H C)_p
// in double-float arithmetic (lanes over mu, a fixed shuffle tree), the term in
// FP64 into eterm[p].  The last warp to finish (a ticket counter, which that warp
// resets for the next launch) adds the terms in a fixed order (lanes over p, then
// a shuffle tree).  No FP64 loop runs on one SM over a whole matrix, and no block
// waits for another.
__global__ void energy_terms_kernel(int nbf, int n_om, const float2* Cdf, const float2* HCt, const double* n,
                                    const double* lambda, const double* enuc, double* eterm, unsigned int* ticket,
                                    double* E) {
  pdl_entry();
  __shared__ int last;
  const int p = blockIdx.x, lane = threadIdx.x;
  float sum = 0.f, cmp = 0.f;
  for (int mu = lane; mu < nbf; mu += 32) {
    const float2 c = Cdf[(size_t)p * nbf + mu], h = HCt[(size_t)p * nbf + mu];
    const float ph = c.x * h.x;
    const float pl = fmaf(c.x, h.x, -ph) + fmaf(c.x, h.y, c.y * h.x);
    float ns, e;
    two_sum_f(sum, ph, ns, e);
    sum = ns;
    cmp += e + pl;
  }
  float sh = sum + cmp, sl = cmp - (sh - sum);
  for (int o = 16; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, sh, o), ol = __shfl_xor_sync(0xffffffffu, sl, o);
    df_add(sh, sl, oh, ol);
  }
  if (lane == 0) {
    eterm[p] = n[p] * ((double)sh + (double)sl) + lambda[(size_t)p * nbf + p];
    __threadfence();
    last = atomicAdd(ticket, 1u) == (unsigned int)(n_om - 1);
  }
  __syncwarp();
  if (!last) return;
  __threadfence();
  // lane l adds the terms q = l, l + 32, ... in order; then a fixed shuffle tree
  double v = 0.0;
  for (int q = lane; q < n_om; q += 32) v += __ldcg(eterm + q);
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) {
    *E = *enuc + v;
    *ticket = 0u;
  }
}

// FOCK weights as double-float pairs: W[q][p] = A_pq, W[N_O + q][p] = -B_pq.
__global__ void fock_weights_df_kernel(const double* A, const double* Bc, int m, float2* W) {
  pdl_entry();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * m * m) return;
  int qq = i / m, pc = i % m;
  const double v = qq < m ? A[(size_t)pc * m + qq] : -Bc[(size_t)pc * m + (qq - m)];
  const float h = (float)v;
  W[i] = make_float2(h, (float)(v - (double)h));
}

// Both digit layouts of b_half from the half transform's integers Xf [P][p][nu]
// (scale 2^(min(e3, e6) - 31)): L3 [P][p][t][nu] with exponent e3[P][p] and L6
// [p][nu][t][P] with exponent e6[p][nu], each a rounding right shift of Xf by
// the exponent difference.  A 64 x 64 (P, nu) tile per block, two adjacent
// elements per thread (8-byte loads, BF16 pairs stored as 4 bytes); L6 goes
// through a shared-memory transposition, so the reads and both digit stores are
// 128 contiguous bytes per warp.  Row strides (nbp, nxp) are even.
//
// The same pass accumulates the diagonal b^P_pp = sum_nu C_{nu p} b^P_{p nu} (Table 3
// step 3) from the L3 integers it has in hand: in the transposed half each thread
// sums its two rows P over its eight nu in double-float arithmetic (X3 = xh + xl
// exactly, C as a double-float pair), the eight thread rows are added in a fixed
// order through shared memory, and one partial per (nu tile, p, P) goes to dpart;
// diag_digits_kernel adds the tiles in a fixed order and applies the row scale.
__global__ void __launch_bounds__(256) xf_to_digits_kernel(const int* Xf, const int* e3, const int* e6, int nx, int nb,
                                                           int m, int mp, int nbp, int nxp, __nv_bfloat16* L3,
                                                           __nv_bfloat16* L6, const float2* Cdf, float2* dpart) {
  pdl_entry();
  __shared__ int tile[64][65];   // the integers Xf of the tile
  __shared__ int ytile[64][65];  // their L3 values (scale e3), for the diagonal partials
  __shared__ int s3[64], s6[64];
  __shared__ float2 sc[64];
  __shared__ float2 red[8][64];
  const int p = blockIdx.z, nu0 = blockIdx.x * 64, P0 = blockIdx.y * 64;
  const int tid = threadIdx.y * 32 + threadIdx.x;
  if (tid < 64) s3[tid] = (P0 + tid < nx) ? e3[(size_t)(P0 + tid) * m + p] : 0;
  else if (tid < 128) s6[tid - 64] = (nu0 + tid - 64 < nb) ? e6[(size_t)p * nb + nu0 + tid - 64] : 0;
  else if (tid < 192) sc[tid - 128] = (nu0 + tid - 128 < nb) ? Cdf[(size_t)p * nb + nu0 + tid - 128] : make_float2(0.f, 0.f);
  __syncthreads();
  const int c0 = 2 * threadIdx.x;  // this thread's column pair within the tile
  // rows P of the tile: L3 digits (nu contiguous).  The eight rows' loads are
  // issued before any of their stores, so that they are in flight together.
  int2 xv[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int P = P0 + threadIdx.y + 8 * i, nu = nu0 + c0;
    xv[i] = make_int2(0, 0);
    if (P < nx && nu < nb) {
      const int* src = Xf + ((size_t)P * m + p) * nbp + nu;
      if (nu + 1 < nb) xv[i] = *(const int2*)src;
      else xv[i].x = src[0];
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = threadIdx.y + 8 * i;
    const int P = P0 + r, nu = nu0 + c0;
    const int x0 = xv[i].x, x1 = xv[i].y;
    if (P < nx && nu < nb) {
      int d = s3[r] - s6[c0];
      const int y0 = rshift_round(x0, d > 0 ? d : 0);
      d = s3[r] - s6[c0 + 1];
      const int y1 = rshift_round(x1, d > 0 ? d : 0);
      __nv_bfloat162 dd[4];
      digits_bf16x2(y0, y1, dd);
      __nv_bfloat16* o = L3 + (((size_t)P * mp + p) * 4) * nbp + nu;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (nu + 1 < nb) *(__nv_bfloat162*)(o + (size_t)t * nbp) = dd[t];
        else o[(size_t)t * nbp] = dd[t].x;
      }
      ytile[r][c0] = y0;
      ytile[r][c0 + 1] = y1;
    } else {
      ytile[r][c0] = 0;
      ytile[r][c0 + 1] = 0;
    }
    tile[r][c0] = x0;
    tile[r][c0 + 1] = x1;
  }
  __syncthreads();
  // columns nu of the tile: L6 digits (P contiguous), and the diagonal partials of the
  // thread's two rows P over its eight nu in double-float arithmetic (the L3 value
  // y = yh + yl exactly in FP32, C as a double-float pair)
  float sum[2] = {0.f, 0.f}, cmp[2] = {0.f, 0.f};
  for (int r = threadIdx.y; r < 64; r += 8) {
    const int nu = nu0 + r, P = P0 + c0;
    if (nu < nb && P < nx) {
      int d = s6[r] - s3[c0];
      const int z0 = rshift_round(tile[c0][r], d > 0 ? d : 0);
      d = s6[r] - s3[c0 + 1];
      const int z1 = rshift_round(tile[c0 + 1][r], d > 0 ? d : 0);
      __nv_bfloat162 dd[4];
      digits_bf16x2(z0, z1, dd);
      __nv_bfloat16* o = L6 + ((size_t)p * nb + nu) * 4 * nxp + P;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (P + 1 < nx) *(__nv_bfloat162*)(o + (size_t)t * nxp) = dd[t];
        else o[(size_t)t * nxp] = dd[t].x;
      }
      const float2 cv = sc[r];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int y = ytile[c0 + k][r];
        const float yh = (float)(y >> 8) * 256.f, yl = (float)(y & 255);
        const float p0 = yh * cv.x;
        const float e0 = fmaf(yh, cv.x, -p0) + (yh * cv.y + yl * cv.x);
        float ns, e;
        two_sum_f(sum[k], p0, ns, e);
        sum[k] = ns;
        cmp[k] += e + e0;
      }
    }
  }
  red[threadIdx.y][c0] = make_float2(sum[0], cmp[0]);
  red[threadIdx.y][c0 + 1] = make_float2(sum[1], cmp[1]);
  __syncthreads();
  if (tid < 64 && P0 + tid < nx) {
    float sh = red[0][tid].x, sl = red[0][tid].y;
#pragma unroll
    for (int y = 1; y < 8; ++y) {
      float ns, e;
      two_sum_f(sh, red[y][tid].x, ns, e);
      sh = ns;
      sl += e + red[y][tid].y;
    }
    dpart[((size_t)blockIdx.x * m + p) * nx + P0 + tid] = make_float2(sh, sl);
  }
}

// d[p][P] = 2^(e3[P][p] - 31) sum over the nu tiles of the pass's double-float
// partials, added in tile order in double-float arithmetic; FP64 only for the
// final value.  Then the digits of row p (as slice_rows_kernel takes them): a block per row,
// which saves the path to the J products a launch.
constexpr int DIAG_THREADS = 256;
__global__ void __launch_bounds__(DIAG_THREADS) diag_digits_kernel(const float2* __restrict__ dpart, int ntiles, int nx,
                                                                   int m, const int* __restrict__ e3,
                                                                   double* __restrict__ d,
                                                                   __nv_bfloat16* __restrict__ planes, int ldp,
                                                                   int* __restrict__ exps, unsigned int* jkmax,
                                                                   long long njk) {
  pdl_entry();
  __shared__ unsigned long long wmax[DIAG_THREADS / 32];
  const int pc = blockIdx.x, tid = threadIdx.x;
  // the row maxima that the J^(q), K^(q) of these orbitals will raise
  for (long long k = pc * (long long)DIAG_THREADS + tid; k < njk; k += (long long)gridDim.x * DIAG_THREADS) jkmax[k] = 0;
  unsigned long long mx = 0;
  for (int P = tid; P < nx; P += DIAG_THREADS) {
    float sh = 0.f, sl = 0.f;
#pragma unroll 4
    for (int t = 0; t < ntiles; ++t) {
      const float2 v = dpart[((size_t)t * m + pc) * nx + P];
      df_add(sh, sl, v.x, v.y);
    }
    const double v = scale_pow2((double)sh + (double)sl, e3[(size_t)P * m + pc] - 31);
    d[(size_t)pc * nx + P] = v;
    mx = max(mx, mag64(v));
  }
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (tid % 32 == 0) wmax[tid / 32] = mx;
  __syncthreads();
  for (int w = 0; w < DIAG_THREADS / 32; ++w) mx = max(mx, wmax[w]);
  const int e = expo_of(__longlong_as_double((long long)mx));
  if (tid == 0) exps[pc] = e;
  __nv_bfloat16* out = planes + (size_t)pc * 4 * ldp;
  for (int P = tid; P < nx; P += DIAG_THREADS) {  // this thread's own values
    __nv_bfloat16 dg[4];
    digits_bf16(fixed32(d[(size_t)pc * nx + P], e), dg);
#pragma unroll
    for (int t = 0; t < 4; ++t) out[t * ldp + P] = dg[t];
  }
}

// Interleaved digits + row exponents -> FP64 values (the fetch path).
__global__ void unslice_kernel(const __nv_bfloat16* planes, int ldp, const int* exps, long long rows, int cols,
                               double* out) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= rows * cols) return;
  long long r = i / cols;
  int k = (int)(i % cols);
  const __nv_bfloat16* pr = planes + r * 4 * ldp + k;
  long long X = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t) X = X * 256 + (long long)__bfloat162float(pr[t * ldp]);
  out[i] = ldexp((double)X, exps[r] - 31);
}

// Matrices z of symmetric n x n double-float values, valid for nu >= mu -> FP64, whole.
__global__ void join_sym_kernel(const float* hi, const float* lo, long long nmat, int n, int ld, double* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= nmat * n * n) return;
  const long long z = i / ((long long)n * n);
  const int mu = (int)(i / n % n), nu = (int)(i % n);
  const size_t o = (size_t)z * n * ld + (nu >= mu ? (size_t)mu * ld + nu : (size_t)nu * ld + mu);
  out[i] = (double)hi[o] + (double)lo[o];
}

}  // namespace donof

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct donof::S4Buffers {
  int nbp, nxp, mp, ldo;
  __nv_bfloat16 *B1, *B5, *Ct, *L3, *L6, *Dp, *JKp;  // interleaved digits
  int* X6;                                            // L6 integers [nx][m][nbp] before digitisation
  int* tri;                                           // packed row of the upper triangle -> mu << 16 | nu
  unsigned int* jkmax;                                // row maxima of J^(q), K^(q) [2m][nb]
  int jk_merged;                                      // 1: J^(q) and K^(q) in one launch (S_JKAO)
  // Unit lists: [kind][0 / 1], the second one with twice the units (summed kinds).
  struct List {
    int4* d;
    int n;
    donof::S4Slots slots;
  } list[donof::S_NKINDS][2];
  int opt[donof::S_NKINDS];                           // the list in use
  int *eB1, *eB5, *eC, *e3, *e6, *ed, *eJK;          // row exponents
  int* e3m;                                           // e3 less eC[p] + 17 [nx][m], and e6 likewise as int16
  short* e6m;                                         // [nb][e6ld] (the half transform's scale)
  int e6ld;
  float *rmaxB, *maxB, *absC, *absCt;
  // Working basis: the orbital basis orthonormalised by the Cholesky factor of the
  // overlap, chi' = chi L^-T with S = L L^T.  Orbitals are C' = L^T C (C'^T C' = I),
  // the fitted tensor B'^P = L^-1 B^P L^-T and H' = L^-1 H L^-T; every GEMM operand
  // and the energy row work in it, and AO outputs are transformed back.
  double* Ls;     // L [mu][nu] row-major, lower triangle (FP64)
  float2* LsTdf;  // L^T [nu][mu] as double-float pairs
  float2* Cin;    // C^T rows [p][mu] (every p < nbf) as double-float pairs
  double* Cp;     // C'^T rows [p][mu'] (every p < nbf), FP64
  float2* Cinp;   // the energy prep's own double-float C^T rows (p < N_O)
  float2* Cdf;    // C' rows p (every p < nbf) as double-float pairs
  float2* Hdf;    // H' as double-float pairs (fixed at init)
  float2* Cdfp;   // C' rows p (< N_O) as double-float pairs, the energy prep's own copy (its stream
                  // may run ahead of the transform that writes Cdf)
  float2* dpart;  // diagonal partials [nu tile][m][nx] from the digit pass
  double* dmat;   // d [m][nx] FP64
  float *JKhi, *JKlo;
  float2* W;
  float2* HCt;  // (H C)^T [p][mu], double-float
  float2* Yt;   // Y^T [p][mu] = (F^(p) C_p)^T, double-float
  // contracted Lagrangian (allocated on its first call)
  double* bf;          // b^P_qp [P][p][q]
  double* wP;          // w [p][P]
  __nv_bfloat16* Xd;   // X digits [q][p][4][nxp]
  int* eX;             // their row exponents [q][p]
  double* eterm;          // the energy's per-orbital terms
  unsigned int* ticket;   // energy_terms_kernel's completion counter (zero between launches)
  void* partial;
  void* partial_j;  // J_pq's int64 partials (its launch group may run beside a3's)
  donof::S4Params plan[donof::S_NKINDS];
  PFN_cuTensorMapEncodeTiled_v12000 encode;
};

namespace donof {

static int s4_round_up(int a, int b) { return (a + b - 1) / b * b; }

// BF16 tensor map, 64-byte swizzle; dims innermost first, strides in elements.
static int s4_map(S4Buffers* sb, CUtensorMap* map, const void* base, int rank, const long long* dims,
                  const long long* strides_el, const int* box) {
  cuuint64_t gd[5], gs[4];
  cuuint32_t bd[5], es[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i < rank; ++i) {
    gd[i] = (cuuint64_t)dims[i];
    bd[i] = (cuuint32_t)box[i];
  }
  for (int i = 0; i < rank - 1; ++i) {
    gs[i] = (cuuint64_t)(strides_el[i] * 2);
    if (gs[i] % 16) return DONOF_RI_E_ARG;
  }
  if (((uintptr_t)base) % 16) return DONOF_RI_E_ARG;
  CUresult r = sb->encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, (void*)base, gd, gs, bd, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? DONOF_RI_OK : DONOF_RI_E_CUDA;
}

// An operand's map: rows [entry][row][digit][k] with row stride 4 ld, read in boxes of
// `brow` rows of `bent` entries, every digit plane, the planes outermost in the box.
static int s4_map_op(S4Buffers* sb, CUtensorMap* map, const void* base, int K, int rows, int ent, long long ld,
                     long long sent, int brow, int bent) {
  const long long d[4] = {K, rows, ent, S4_PLANES}, s[3] = {4 * ld, ent > 1 ? sent : 4 * ld * rows, ld};
  const int b[4] = {S4_BK, brow, bent, S4_PLANES};
  return s4_map(sb, map, base, 4, d, s, b);
}

// ---------------------------------------------------------------------------
// Unit lists
// ---------------------------------------------------------------------------
typedef std::vector<int4> S4Units;

static void s4_add_unit(S4Units& v, int b0, int nbat, int nh, int opi, int first, int mt, int nt, int slot) {
  v.push_back(make_int4(b0, (int)((unsigned)nbat | ((unsigned)nh << 28) | ((unsigned)opi << 30) | ((unsigned)first << 31)), mt, (int)((unsigned)nt | ((unsigned)slot << 16))));
}

// Units of a kind whose batches are summed: `mtiles` row tiles x `ncols` columns x
// `nbatch` batches of `nkb` K blocks.  A unit with two halves takes bpc batches, one
// with a single half twice as many (equal cost).  bpc minimises the modelled time of
// the launch (in cycles of one SM: whole turns of 152 CTAs, 624 cycles per K block and
// half, about 1500 per unit for its start and its sums) plus that of writing and
// reading the partials (`groups` per slot) at 6 TB/s; `finer` halves it.
// Returns the modelled cycles; with out == nullptr nothing else.
static double s4_sum_units(int mtiles, int ncols, int nbatch, int nkb, int groups, double out_bytes, int finer,
                           S4Units* out, S4Slots* slots) {
  const int ntiles = (ncols + S4_BN - 1) / S4_BN, pairs = ntiles / 2, single = ntiles & 1;
  double best = 1e300;
  int bpc = 1;
  for (int b2 = 1; b2 <= nbatch; ++b2) {
    const int b1 = 2 * b2 < nbatch ? 2 * b2 : nbatch;
    const long long n2 = (nbatch + b2 - 1) / b2, n1 = (nbatch + b1 - 1) / b1;
    const long long slots_used = (pairs ? n2 : n1) * groups;
    const double bytes = 2.0 * (double)slots_used * out_bytes;
    if (slots_used > 60000 || (bytes > 1e9 && b2 < nbatch)) continue;
    const long long units = (long long)mtiles * (pairs * n2 + single * n1);
    const long long turns = (units + S4_SMS - 1) / S4_SMS;
    const int halves = pairs ? 2 * b2 : b1;
    const double cyc = (double)turns * (624.0 * nkb * halves + 1500.0) + bytes / 6e12 * 1.9e9;
    if (cyc < best) {
      best = cyc;
      bpc = b2;
    }
  }
  if (!out) return best;
  if (finer) bpc = (bpc + 1) / 2;
  const int b1 = 2 * bpc < nbatch ? 2 * bpc : nbatch;
  // by first batch, so that the CTAs running at the same time share A's rows through L2
  for (int c = 0; c * bpc < nbatch; ++c)
    for (int mt = 0; mt < mtiles; ++mt) {
      for (int np = 0; np < pairs; ++np)
        s4_add_unit(*out, c * bpc, std::min(bpc, nbatch - c * bpc), 2, 0, np == 0, mt, 2 * np, c);
      if (single && (c * bpc) % b1 == 0)
        s4_add_unit(*out, c * bpc, std::min(b1, nbatch - c * bpc), 1, 0, pairs == 0, mt, ntiles - 1, c * bpc / b1);
    }
  slots->pair = (nbatch + bpc - 1) / bpc * groups;
  slots->single = (nbatch + b1 - 1) / b1 * groups;
  slots->split = pairs * 2 * S4_BN;
  return best;
}

// log2 of the rows per group that wastes the least of `mtiles` for nrows rows of each of
// nent entries (ties: the larger group), for the summed kinds with a shared B operand.
static int s4_best_rshift(int nrows, int nent, int ncols, int nc, int nkb, double out_bytes) {
  int best = 7;
  double cost = 1e300;
  for (int rs = 7; rs >= 4; --rs) {
    const int groups = 128 >> rs, ents = (nent + groups - 1) / groups;
    const double c = s4_sum_units((nrows + (1 << rs) - 1) >> rs, ncols, ents * nc, nkb, groups, out_bytes, 0, nullptr,
                                  nullptr);
    if (c < 0.99 * cost) {
      cost = c;
      best = rs;
    }
  }
  return best;
}

// Units of a row block x every column tile (pairs of halves), one batch.
static void s4_row_units(S4Units& v, int b, int mt, int nt0, int ntiles, int opi) {
  for (int nt = nt0; nt < ntiles; nt += 2) s4_add_unit(v, b, 1, nt + 1 < ntiles ? 2 : 1, opi, nt == nt0, mt, nt, 0);
}

static int s4_upload(S4Buffers* sb, int kind, int opt, const S4Units& v) {
  S4Buffers::List& l = sb->list[kind][opt];
  l.n = (int)v.size();
  if (cudaMalloc((void**)&l.d, (v.size() + 1) * sizeof(int4)) != cudaSuccess) {
    cudaGetLastError();
    return DONOF_RI_E_OOM;
  }
  if (!v.empty() && cudaMemcpy(l.d, v.data(), v.size() * sizeof(int4), cudaMemcpyHostToDevice) != cudaSuccess)
    return DONOF_RI_E_CUDA;
  return DONOF_RI_OK;
}

// Makes list `opt` of a kind the one its next launch takes.
static void s4_use(S4Buffers* sb, int kind, int opt) {
  sb->opt[kind] = opt;
  sb->plan[kind].units = sb->list[kind][opt].d;
  sb->plan[kind].nunits = sb->list[kind][opt].n;
}

static int s4_grid(const S4Params& p) { return p.nunits < S4_SMS ? p.nunits : S4_SMS; }
static size_t s4_smem(const S4Params& p) { return S4_FIXED_SMEM + (size_t)p.stages * S4_STAGE_BYTES; }

// Every unit list of the context, and the bytes of the partial sums.
static int s4_build_lists(donof_ri_ctx* ctx, size_t* pbytes, size_t* jbytes) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, nx = ctx->naux, m = ctx->n_omega;
  const int KBb = (nb + S4_BK - 1) / S4_BK, KBx = (nx + S4_BK - 1) / S4_BK;
  const int tm = (m + S4_BN - 1) / S4_BN, tb = (nb + S4_BN - 1) / S4_BN;
  int rc;
  for (int k = 0; k < S_NKINDS; ++k) {
    S4Params& p = sb->plan[k];
    p.stages = S4_MAX_STAGES;
    p.nc = 1;
    p.nkb = p.nkb_all = KBx;
    for (S4Operands& o : p.op) o.rshift = 7;
  }
  {
    S4Params& p = sb->plan[S_HALF];
    p.nkb = p.nkb_all = KBb;
    p.op[0].rshift = 4;  // 16 nu of 8 auxiliary functions: nbf fills multiples of 16, and a store is a full sector
    S4Units v;
    for (int b = 0; b < (nx + 7) / 8; ++b)
      for (int mt = 0; mt < (nb + 15) / 16; ++mt) s4_row_units(v, b, mt, 0, tm, 0);
    if ((rc = s4_upload(sb, S_HALF, 0, v))) return rc;
  }
  *pbytes = 0;
  const double m2 = (double)m * m * 8, mn = (double)m * nb * 8;
  struct Sum {
    int kind, nrows, nent, nc, nkb, nkb_all;
    bool grouped;
    double bytes;
  };
  const int ncf = (KBb + s4_chunk_kb(S_FOCK) - 1) / s4_chunk_kb(S_FOCK), ncj = (KBx + S4_CHUNK_KB - 1) / S4_CHUNK_KB;
  const Sum sums[4] = {
      {S_FULLSQ, m, nx, 1, KBb, KBb, true, m2},                                             // rows (P, p)
      {S_FOCK, nb, 2 * m, ncf, ncf > 1 ? s4_chunk_kb(S_FOCK) : KBb, KBb, true, mn},         // rows (q', mu)
      {S_JMO, m, 1, ncj, ncj > 1 ? S4_CHUNK_KB : KBx, KBx, false, m2},                      // rows p
      {S_CTR, nb, m, 1, KBx, KBx, false, mn}};                                              // rows mu
  for (const Sum& s : sums) {
    S4Params& p = sb->plan[s.kind];
    p.nc = s.nc;
    p.nkb = s.nkb;
    p.nkb_all = s.nkb_all;
    const int rs = s.grouped ? s4_best_rshift(s.nrows, s.nent, m, s.nc, s.nkb, s.bytes) : 7;
    p.op[0].rshift = rs;
    const int groups = 128 >> rs, ents = (s.nent + groups - 1) / groups;
    for (int o = 0; o < 2; ++o) {
      S4Units v;
      S4Slots sl;
      s4_sum_units((s.nrows + (1 << rs) - 1) >> rs, m, ents * s.nc, s.nkb, groups, s.bytes, o, &v, &sl);
      if ((rc = s4_upload(sb, s.kind, o, v))) return rc;
      sb->list[s.kind][o].slots = sl;
      const size_t bytes = (size_t)(sl.pair > sl.single ? sl.pair : sl.single) * (size_t)s.bytes;
      size_t* dst = s.kind == S_JMO ? jbytes : pbytes;
      if (s.kind == S_JMO && o == 0) *dst = 0;
      if (bytes > *dst) *dst = bytes;
    }
  }
  // K^(q): only the tiles that reach the diagonal or lie above it (the split mirrors the rest)
  S4Units kao, kao2;
  for (int q = 0; q < m; ++q)
    for (int mt = 0; mt < (nb + S4_BM - 1) / S4_BM; ++mt) {
      int nt0 = 0;
      while (nt0 * S4_BN + S4_BN - 1 < mt * S4_BM) ++nt0;
      s4_row_units(kao, q, mt, nt0, tb, 0);
      s4_row_units(kao2, q, mt, nt0, tb, 1);
    }
  if ((rc = s4_upload(sb, S_KAO, 0, kao))) return rc;
  // J^(q): the packed rows of the upper triangle, alone and followed by the K^(q) units
  {
    S4Units v;
    const long long rows = (long long)nb * (nb + 1) / 2;
    for (long long mt = 0; mt < (rows + S4_BM - 1) / S4_BM; ++mt) s4_row_units(v, 0, (int)mt, 0, tm, 0);
    if ((rc = s4_upload(sb, S_JAO, 0, v))) return rc;
    v.insert(v.end(), kao2.begin(), kao2.end());
    if ((rc = s4_upload(sb, S_JKAO, 0, v))) return rc;
  }
  for (int k = 0; k < S_NKINDS; ++k) s4_use(sb, k, 0);
  return DONOF_RI_OK;
}

// The merged J^(q) + K^(q) launch takes the two kinds' operands.
static void s4_plan_jkao(S4Buffers* sb) {
  S4Params& p = sb->plan[S_JKAO];
  p.op[0] = sb->plan[S_JAO].op[0];
  p.op[1] = sb->plan[S_KAO].op[0];
  p.ohi = sb->JKhi;
  p.olo = sb->JKlo;
  p.tri = sb->tri;
  p.stages = std::max(sb->plan[S_JAO].stages, sb->plan[S_KAO].stages);
}

// X^T as double-float pairs.
__global__ void transpose_df_kernel(const double* X, int n, float2* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)n * n) return;
  const int r = (int)(i / n), c = (int)(i % n);
  out[i] = to_df(X[(size_t)c * n + r]);
}

__global__ void identity64_kernel(int n, double* X) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)n * n) return;
  X[i] = (i / n == i % n) ? 1.0 : 0.0;
}

// X^P <- (X^P + X^P^T) / 2 for each of `batch` n x n matrices: the two-sided products
// below are symmetric only up to rounding, and the digit layouts take B' as symmetric.
__global__ void symmetrize_kernel(double* X, int n, long long batch) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long n2 = (long long)n * n;
  if (i >= batch * n2) return;
  const long long b = i / n2;
  const int r = (int)((i % n2) / n), c = (int)(i % n);
  if (c <= r) return;
  double* M = X + b * n2;
  const double v = 0.5 * (M[(size_t)r * n + c] + M[(size_t)c * n + r]);
  M[(size_t)r * n + c] = v;
  M[(size_t)c * n + r] = v;
}

// out = Li X Li^T for `batch` symmetric n x n matrices X and a lower-triangular Li.
// On the tensor cores (launch_xgemm) where they take the size: only the triangle that Li
// leaves in the first product, and only the lower triangle of the second, a workspace's
// worth of matrices at a time (512 MB, or what there is room for).  Otherwise two FP64
// products and the mean of both triangles (240 functions, 840 matrices: 42 ms).
static int s4_congruence(donof_ri_ctx* ctx, const double* Li, const double* X, int n, int batch, double* out) {
  const long long n2 = (long long)n * n;
  cudaStream_t s = ctx->stream;
  Gemm64 g{};  // T = Li X
  g.M = n; g.N = n; g.K = n;
  g.A = Li; g.sAb = 0; g.sAm = n; g.sAk = 1;
  g.sBb = n2; g.sBk = 1; g.sBn = n;  // X symmetric: rows along k
  g.sCb = n2; g.sCm = n; g.sCn = 1;
  g.alpha = 1.0; g.beta = 0.0;
  Gemm64 h{};  // out = T Li^T
  h.M = n; h.N = n; h.K = n;
  h.sAb = n2; h.sAm = n; h.sAk = 1;
  h.B = Li; h.sBb = 0; h.sBk = 1; h.sBn = n;  // element (k, n) of Li^T = Li[n][k]
  h.sCb = n2; h.sCm = n; h.sCn = 1;
  h.alpha = 1.0; h.beta = 0.0;
  int rc;
  g.batch = 1;
  const size_t per = n2 * sizeof(double) + xgemm_operand_bytes(n, n, 1);
  int step = (int)((size_t)512e6 / per);
  if (step > batch) step = batch;
  if (step < 1) step = 1;
  if (xgemm_takes(g)) {
    size_t tbytes;
    char* ws;
    for (;; step = (step + 1) / 2) {
      tbytes = ((size_t)step * n2 * sizeof(double) + 255) / 256 * 256;
      const size_t bytes = tbytes + xgemm_operand_bytes(n, n, step) + xgemm_operand_bytes(n, n, 1);
      rc = xgemm_workspace(ctx, bytes, bytes, (void**)&ws);
      if (rc != DONOF_RI_E_OOM || step == 1) break;
    }
    if (rc) return rc;
    double* T = (double*)ws;
    for (int b = 0; b < batch; b += step) {
      g.batch = h.batch = batch - b < step ? batch - b : step;
      g.B = X + b * n2;
      g.C = T;
      h.A = T;
      h.C = out + b * n2;
      if ((rc = launch_xgemm(ctx, g, ws + tbytes, XG_A_LOWER))) return rc;
      if ((rc = launch_xgemm(ctx, h, ws + tbytes, XG_B_LOWER | XG_C_LOWER))) return rc;
    }
    return launch_mirror_lower(ctx, out, n, batch);
  }
  double* T = nullptr;
  if (cudaMalloc((void**)&T, (size_t)batch * n2 * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    return DONOF_RI_E_OOM;
  }
  g.batch = h.batch = batch;
  g.B = X; g.sBk = n; g.sBn = 1;
  g.C = T;
  h.A = T;
  h.C = out;
  rc = launch_dgemm(ctx, g);
  if (!rc) rc = launch_dgemm(ctx, h);
  if (!rc) {
    symmetrize_kernel<<<ceil_div_u((long long)batch * n2, 256), 256, 0, s>>>(out, n, batch);
    ctx->launches++;
    if (cudaGetLastError() != cudaSuccess) rc = DONOF_RI_E_CUDA;
  }
  cudaStreamSynchronize(s);
  cudaFree(T);
  return rc;
}

// L L^T = S (FP64 Cholesky of the overlap) into sb->Ls, Li = L^-1, and the fitted
// tensor and core Hamiltonian in the working basis: Bw^P = Li B^P Li^T,
// Hw = Li H Li^T; L^T as double-float pairs into sb->LsTdf.
static int s4_working_basis(donof_ri_ctx* ctx, double* Li, double* Bw, double* Hw) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, nx = ctx->naux;
  const long long n2 = (long long)nb * nb;
  cudaStream_t s = ctx->stream;
  int rc;
  DONOF_CUDA_TRY(cudaMemcpyAsync(sb->Ls, ctx->d_S, n2 * sizeof(double), cudaMemcpyDeviceToDevice, s));
  if ((rc = cholesky_lower(ctx, sb->Ls, nb, ctx->d_scratch_max, 1e-14))) return rc;
  identity64_kernel<<<ceil_div_u(n2, 256), 256, 0, s>>>(nb, Li);
  DONOF_LAUNCH_CHECK(ctx);
  if ((rc = forward_subst(ctx, sb->Ls, nb, Li, nb))) return rc;  // Li = L^-1
  transpose_df_kernel<<<ceil_div_u(n2, 256), 256, 0, s>>>(sb->Ls, nb, sb->LsTdf);
  DONOF_LAUNCH_CHECK(ctx);
  if ((rc = s4_congruence(ctx, Li, ctx->d_B, nb, nx, Bw))) return rc;
  return s4_congruence(ctx, Li, ctx->d_H, nb, 1, Hw);
}

static int s4_init_buffers(donof_ri_ctx* ctx) {
  S4Buffers* sb = (S4Buffers*)calloc(1, sizeof(S4Buffers));
  if (!sb) return DONOF_RI_E_OOM;
  ctx->s4 = sb;
  {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !f) {
      cudaGetLastError();
      return DONOF_RI_E_UNSUPPORTED;
    }
    sb->encode = (PFN_cuTensorMapEncodeTiled_v12000)f;
  }
  const int nb = ctx->nbf, nx = ctx->naux, m = ctx->n_omega;
  // Digit rows padded to 16 elements (32 bytes) so that full-sector stores stay aligned.
  const int nbp = s4_round_up(nb, 16), nxp = s4_round_up(nx, 16), mp = s4_round_up(m, 4), ldo = s4_round_up(nb, 8);
  sb->nbp = nbp; sb->nxp = nxp; sb->mp = mp; sb->ldo = ldo;
  const long long nbs = nb, nxs = nx, ms = m;
  const int bn = S4_BN;
  size_t pbytes = 0, jbytes = 0;
  int rc;

#define ALLOC(ptr, bytes)                                             \
  do {                                                                \
    if (cudaMalloc((void**)&(ptr), (size_t)(bytes)) != cudaSuccess) { \
      cudaGetLastError();                                             \
      return DONOF_RI_E_OOM;                                          \
    }                                                                 \
  } while (0)
  ALLOC(sb->B1, nxs * nbs * 4 * nbp * 2);
  const long long ntri = nbs * (nbs + 1) / 2;
  ALLOC(sb->B5, ntri * 4 * nxp * 2);
  ALLOC(sb->tri, ntri * sizeof(int));
  ALLOC(sb->jkmax, 2 * ms * nbs * 4);
  ALLOC(sb->Ct, ms * 4 * nbp * 2);
  ALLOC(sb->L3, nxs * mp * 4 * nbp * 2);
  ALLOC(sb->L6, ms * nbs * 4 * nxp * 2);
  ALLOC(sb->X6, nxs * ms * nbp * 4);
  ALLOC(sb->Dp, ms * 4 * nxp * 2);
  ALLOC(sb->JKp, 2 * ms * nbs * 4 * nbp * 2);
  ALLOC(sb->eB1, nxs * nbs * 4);
  ALLOC(sb->eB5, ntri * 4);
  ALLOC(sb->eC, ms * 4);
  ALLOC(sb->e3, nxs * ms * 4);
  ALLOC(sb->e6, ms * nbs * 4);
  ALLOC(sb->e3m, nxs * ms * 4);
  sb->e6ld = s4_round_up(m, S4_BN);
  ALLOC(sb->e6m, nbs * sb->e6ld * 2);
  ALLOC(sb->ed, ms * 4);
  ALLOC(sb->eJK, 2 * ms * nbs * 4);
  ALLOC(sb->rmaxB, nxs * nbs * 4);
  ALLOC(sb->maxB, nbs * nbs * 4);
  ALLOC(sb->absC, ms * nbs * 4);
  ALLOC(sb->absCt, ms * nbs * 4);
  ALLOC(sb->Ls, nbs * nbs * 8);
  ALLOC(sb->LsTdf, nbs * nbs * 8);
  ALLOC(sb->Cin, nbs * nbs * 8);
  ALLOC(sb->Cp, nbs * nbs * 8);
  ALLOC(sb->Cinp, ms * nbs * 8);
  ALLOC(sb->Cdf, nbs * nbs * 8);
  ALLOC(sb->Hdf, nbs * nbs * 8);
  ALLOC(sb->Cdfp, ms * nbs * 8);
  ALLOC(sb->eterm, ms * 8);
  ALLOC(sb->ticket, 4);
  ALLOC(sb->dpart, (size_t)((nb + 63) / 64) * ms * nxs * 8);
  ALLOC(sb->dmat, ms * nxs * 8);
  ALLOC(sb->JKhi, 2 * ms * nbs * ldo * 4);
  ALLOC(sb->JKlo, 2 * ms * nbs * ldo * 4);
  ALLOC(sb->W, 2 * ms * ms * 8);
  ALLOC(sb->HCt, ms * nbs * 8);
  ALLOC(sb->Yt, ms * nbs * 8);
  // host memory only for what the device has room for: the lists hold 16 bytes for every 12288
  // elements of K^(q)
  if ((rc = s4_build_lists(ctx, &pbytes, &jbytes))) return rc;
  ALLOC(sb->partial, pbytes);
  ALLOC(sb->partial_j, jbytes);
#undef ALLOC
  {
    std::vector<int> tri;
    tri.reserve((size_t)ntri);
    for (int mu = 0; mu < nb; ++mu)
      for (int nu = mu; nu < nb; ++nu) tri.push_back((int)((unsigned)mu << 16 | (unsigned)nu));
    if (cudaMemcpy(sb->tri, tri.data(), tri.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
      return DONOF_RI_E_CUDA;
  }

  // The working basis (see S4Buffers): L from the overlap, then B' = L^-1 B L^-T and
  // H' = L^-1 H L^-T in FP64 (temporaries freed after the digitisation), L^T as
  // double-float pairs for the per-iteration C' = L^T C.
  cudaStream_t s = ctx->stream;
  double *Li = nullptr, *Bw = nullptr, *Hw = nullptr;
  auto free_tmp = [&]() {
    if (Li) cudaFree(Li);
    if (Bw) cudaFree(Bw);
    if (Hw) cudaFree(Hw);
  };
  if (cudaMalloc((void**)&Li, nbs * nbs * 8) != cudaSuccess ||
      cudaMalloc((void**)&Bw, nxs * nbs * nbs * 8) != cudaSuccess || cudaMalloc((void**)&Hw, nbs * nbs * 8) != cudaSuccess) {
    cudaGetLastError();
    free_tmp();
    return DONOF_RI_E_OOM;
  }
  if ((rc = s4_working_basis(ctx, Li, Bw, Hw))) {
    cudaStreamSynchronize(s);
    free_tmp();
    return rc;
  }
  // one-time digitisation of B' in both operand layouts, and its maxima for the bounds
  to_df_kernel<<<ceil_div_u(nbs * nbs, 256), 256, 0, s>>>(Hw, nbs * nbs, sb->Hdf);
  if (cudaMemsetAsync(sb->ticket, 0, sizeof(unsigned int), s) != cudaSuccess) return DONOF_RI_E_CUDA;
  {
    long long rows = nxs * nbs;  // rows (P, nu) over mu (B' symmetric)
    slice_f64_kernel<<<ceil_div_u(rows * 32, 256), 256, 0, s>>>(Bw, rows, nb, sb->B1, nbp, sb->eB1, sb->rmaxB);
    DONOF_LAUNCH_CHECK(ctx);
    // rows (mu, nu), mu <= nu, over P
    slice_tri_kernel<<<ceil_div_u(ntri, 32), dim3(32, 8), 0, s>>>(Bw, sb->tri, (int)ntri, nb, nx, sb->B5, nxp, sb->eB5,
                                                                  sb->maxB);
    DONOF_LAUNCH_CHECK(ctx);
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) {
    free_tmp();
    return DONOF_RI_E_CUDA;
  }
  free_tmp();

  for (int k = 0; k < S_NKINDS; ++k) {
    S4Params& p = sb->plan[k];
    p.nb = nb; p.nx = nx; p.m = m; p.nbp = nbp;
    p.status = ctx->d_status;
    p.partial = k == S_JMO ? sb->partial_j : sb->partial;
    p.ldo = ldo;
    p.prow = m;
    p.pcol = (k == S_FOCK || k == S_CTR) ? nb : m;
  }
  // operand maps: A (k, row, entry, digit) in boxes of 128 rows, B (k, column, entry, digit)
  // in boxes of one half; a box brings all four digit planes, one above the other
  struct Op {
    int kind;
    const void* a;
    int K, nrows, nent;
    long long lda, sent;  // row stride (four planes apart: 4 lda) and entry stride of A, elements
    const int* ea;
    const void* b;
    int ncols, batched;
    long long ldb, sbent;
    const int* eb;
  };
  const long long bp = nbp, xp = nxp;
  const Op ops[] = {
      // HALF: B1 [nx][nb][4][nbp] rows (P, nu) over mu; C^T digits [m][4][nbp]
      {S_HALF, sb->B1, nb, nb, nx, bp, nbs * 4 * bp, sb->eB1, sb->Ct, m, 0, bp, 0, sb->eC},
      // FULLSQ: L3 [nx][mp][4][nbp] rows (P, p) over nu; C^T digits
      {S_FULLSQ, sb->L3, nb, m, nx, bp, (long long)mp * 4 * bp, sb->e3, sb->Ct, m, 0, bp, 0, sb->eC},
      // JMO: d digits [m][4][nxp] over P, both operands
      {S_JMO, sb->Dp, nx, m, 1, xp, 0, sb->ed, sb->Dp, m, 0, xp, 0, sb->ed},
      // JAO: B5 [nb (nb + 1) / 2][4][nxp] rows (mu, nu), mu <= nu, over P; d digits
      {S_JAO, sb->B5, nx, (int)ntri, 1, xp, 0, sb->eB5, sb->Dp, m, 0, xp, 0, sb->ed},
      // KAO: L6 [m][nb][4][nxp] rows (q, mu) over P, both operands
      {S_KAO, sb->L6, nx, nb, m, xp, nbs * 4 * xp, sb->e6, sb->L6, nb, 1, xp, nbs * 4 * xp, sb->e6},
      // FOCK: JK digits [2m][nb][4][nbp] rows (q', mu) over nu; C^T digits.  Rows over (q', mu)
      // fill the tiles whatever N_Omega is; the weight W[q'][p] is per entry and column.
      {S_FOCK, sb->JKp, nb, nb, 2 * m, bp, nbs * 4 * bp, sb->eJK, sb->Ct, m, 0, bp, 0, sb->eC},
  };
  for (const Op& o : ops) {
    S4Operands& op = sb->plan[o.kind].op[0];
    op.nrows = o.nrows; op.nent = o.nent; op.ncols = o.ncols; op.batched = o.batched;
    op.ea = o.ea; op.eb = o.eb;
    if ((rc = s4_map_op(sb, &op.a, o.a, o.K, o.nrows, o.nent, o.lda, o.sent, 1 << op.rshift, 128 >> op.rshift)) ||
        (rc = s4_map_op(sb, &op.b, o.b, o.K, o.ncols, o.batched ? o.nent : 1, o.ldb, o.sbent, bn, 1)))
      return rc;
  }
  sb->plan[S_HALF].x6 = sb->X6; sb->plan[S_HALF].e3m = sb->e3m; sb->plan[S_HALF].e6m = sb->e6m; sb->plan[S_HALF].e6ld = sb->e6ld;
  sb->plan[S_FOCK].w = sb->W;
  for (int k : {S_JAO, S_KAO}) { sb->plan[k].ohi = sb->JKhi; sb->plan[k].olo = sb->JKlo; }
  sb->plan[S_JAO].tri = sb->tri;
  s4_plan_jkao(sb);
  // J^(q) and K^(q) in one persistent launch while every unit is one K chunk: it saves a
  // launch and its tail (iterations without the full transform, two launches / one, us:
  // C6H12 307 / 293, nbf 240 and naux 512 826 / 810).  Beyond 512 auxiliary functions two
  // launches are the default, which is the same at C16H32 and C20H40 (7.27 / 7.27 and
  // 26.57 / 26.53 ms) and 2 % behind between (naux 544 912 / 892 us, C10H20 1204 / 1179);
  // s4_autotune measures both.
  sb->jk_merged = nx <= S4_CHUNK_KB * S4_BK ? 1 : 0;
#define OPTIN(KIND, ...)                                                                                      \
  if (cudaFuncSetAttribute(s4_gemm_kernel<KIND, __VA_ARGS__>, cudaFuncAttributeMaxDynamicSharedMemorySize,           \
                           (int)(S4_FIXED_SMEM + S4_MAX_STAGES * (size_t)S4_STAGE_BYTES)) != cudaSuccess ||   \
      cudaFuncSetAttribute(s4_gemm_kernel<KIND, __VA_ARGS__>, cudaFuncAttributePreferredSharedMemoryCarveout,        \
                           (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess)                               \
    return DONOF_RI_E_CUDA;
  OPTIN(S_HALF, 0) OPTIN(S_HALF, 1) OPTIN(S_FULLSQ, 0) OPTIN(S_FULLSQ, 1) OPTIN(S_FULLSQ, 0, true) OPTIN(S_FULLSQ, 1, true) OPTIN(S_JMO, 0) OPTIN(S_JAO, 0) OPTIN(S_JAO, 1)
  OPTIN(S_KAO, 0) OPTIN(S_KAO, 1) OPTIN(S_FOCK, 1) OPTIN(S_JKAO, 0) OPTIN(S_JKAO, 1) OPTIN(S_CTR, 0)
#undef OPTIN
  DONOF_CUDA_TRY(allow_full_smem(sym_split_kernel));
  return DONOF_RI_OK;
}

int s4_init(donof_ri_ctx* ctx) {
  try {
    return s4_init_buffers(ctx);
  } catch (const std::bad_alloc&) {  // no exception crosses the ABI
    return DONOF_RI_E_OOM;
  }
}

void s4_free(donof_ri_ctx* ctx) {
  S4Buffers* sb = ctx->s4;
  if (!sb) return;
  void* bufs[] = {sb->tri,   sb->jkmax, sb->X6,    sb->B1,   sb->B5,   sb->Ct,   sb->L3,   sb->L6, sb->Dp,  sb->JKp,  sb->eB1,   sb->eB5,
                  sb->eC,    sb->e3,   sb->e6,   sb->e3m,  sb->e6m,   sb->ed,   sb->eJK, sb->rmaxB, sb->maxB, sb->absC, sb->absCt,
                  sb->Ls,    sb->LsTdf, sb->Cin,   sb->Cp,   sb->Cinp,
                  sb->Cdf,   sb->Hdf,   sb->Cdfp,  sb->eterm, sb->ticket, sb->dpart, sb->dmat, sb->JKhi, sb->JKlo, sb->W,  sb->HCt, sb->Yt,   sb->partial, sb->partial_j,
                  sb->bf,    sb->wP,    sb->Xd,    sb->eX};
  for (void* b : bufs)
    if (b) cudaFree(b);
  for (auto& k : sb->list)
    for (S4Buffers::List& l : k)
      if (l.d) cudaFree(l.d);
  free(sb);
  ctx->s4 = nullptr;
}

template <int KIND>
static int launch_s4(donof_ri_ctx* ctx) {
  const S4Params& p = ctx->s4->plan[KIND];
  if (p.nunits <= 0) return DONOF_RI_OK;
  ProfScope ps(ctx, KIND == S_JKAO  ? DONOF_RI_GEMM_JAO
                    : KIND == S_CTR ? DONOF_RI_GEMM_FOCK
                                    : DONOF_RI_GEMM_HALF + KIND);
  // single-chunk epilogue where every batch's K fits one chunk (F^(p) C_p: always)
  const dim3 g(s4_grid(p)), t(S4_THREADS);
  const size_t sm = s4_smem(p);
  if constexpr (KIND == S_FOCK) {
    launch_pdl(s4_gemm_kernel<KIND, 1>, g, t, sm, ctx->stream, p);
  } else if constexpr (KIND == S_FULLSQ) {
    const bool one = p.nkb <= s4_chunk_kb(KIND);
    if (p.bfull && one) launch_pdl(s4_gemm_kernel<KIND, 1, true>, g, t, sm, ctx->stream, p);
    else if (p.bfull) launch_pdl(s4_gemm_kernel<KIND, 0, true>, g, t, sm, ctx->stream, p);
    else if (one) launch_pdl(s4_gemm_kernel<KIND, 1>, g, t, sm, ctx->stream, p);
    else launch_pdl(s4_gemm_kernel<KIND, 0>, g, t, sm, ctx->stream, p);
  } else if constexpr (KIND == S_JMO || KIND == S_CTR) {
    launch_pdl(s4_gemm_kernel<KIND, 0>, g, t, sm, ctx->stream, p);
  } else {
    if (p.nkb <= s4_chunk_kb(KIND)) launch_pdl(s4_gemm_kernel<KIND, 1>, g, t, sm, ctx->stream, p);
    else launch_pdl(s4_gemm_kernel<KIND, 0>, g, t, sm, ctx->stream, p);
  }
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

static const S4Slots& s4_slots(const S4Buffers* sb, int kind) { return sb->list[kind][sb->opt[kind]].slots; }

int s4_transform(donof_ri_ctx* ctx, int mode) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, nx = ctx->naux, m = ctx->n_omega;
  cudaStream_t s = ctx->stream;
  int rc;
  {
    ProfScope ps(ctx, DONOF_RI_ROW_OTHER);
    // the orbitals in the working basis, C' = L^T C: rows of C'^T [p][mu'] =
    // sum_mu C^T[p][mu] L[mu][mu'] (C column-major = rows p contiguous), in double-float
    const dim3 cg((nb + DFG_TJ - 1) / DFG_TJ, (nb + DFG_TI - 1) / DFG_TI);
    if (nb <= DFG_FP64_A) {
      launch_pdl(df_gemm_nt_kernel<double, double>, cg, dim3(DFG_THREADS), 0, s, nb, nb, nb, (const double*)ctx->d_C, nb,
                 (const float2*)sb->LsTdf, nb, sb->Cp, nb);
    } else {
      launch_pdl(to_df_kernel, dim3(ceil_div_u((long long)nb * nb, 256)), dim3(256), 0, s, (const double*)ctx->d_C,
                 (long long)nb * nb, sb->Cin);
      DONOF_LAUNCH_CHECK(ctx);
      launch_pdl(df_gemm_nt_kernel<double, float2>, cg, dim3(DFG_THREADS), 0, s, nb, nb, nb, (const float2*)sb->Cin, nb,
                 (const float2*)sb->LsTdf, nb, sb->Cp, nb);
    }
    DONOF_LAUNCH_CHECK(ctx);
    // C'^T rows p over mu' (and every row of C' as double-float pairs, for lambda)
    launch_pdl(slice_rows_kernel, dim3(nb), dim3(SLICE_ROWS_THREADS), 0, s, (const double*)sb->Cp, m, nb,
               (long long)nb, sb->Ct, sb->nbp, sb->eC, sb->absC, sb->absCt, sb->Cdf);
    DONOF_LAUNCH_CHECK(ctx);
    auto blocks = [](int n) { return (n + BOUND_TILE - 1) / BOUND_TILE; };
    const BoundJob j3{nx, m, sb->rmaxB, nb, sb->absCt, m, sb->e3, m, sb->e3m, nullptr, 0, blocks(m), blocks(m) * blocks(nx)};
    const BoundJob j6{m, nb, sb->absC, nb, sb->maxB, nb, sb->e6, nb, nullptr, sb->e6m, sb->e6ld, blocks(nb),
                      blocks(nb) * blocks(m)};
    launch_pdl(bound_kernel, dim3(j3.blocks + j6.blocks), dim3(256), 0, s, j3, j6, nb, (const int*)sb->eC);
    DONOF_LAUNCH_CHECK(ctx);
  }
  {
    ProfScope ps(ctx, DONOF_RI_ROW_HALF);
    if ((rc = launch_s4<S_HALF>(ctx))) return rc;
    dim3 g((nb + 63) / 64, (nx + 63) / 64, m), b(32, 8);
    ProfScope pm(ctx, DONOF_RI_MEM_DIGITS);
    launch_pdl(xf_to_digits_kernel, g, b, 0, s, (const int*)sb->X6, (const int*)sb->e3, (const int*)sb->e6, nx, nb, m,
               sb->mp, sb->nbp, sb->nxp, sb->L3, sb->L6, (const float2*)sb->Cdf, sb->dpart);
    DONOF_LAUNCH_CHECK(ctx);
  }
  {
    ProfScope ps(ctx, DONOF_RI_ROW_DIAG);
    launch_pdl(diag_digits_kernel, dim3(m), dim3(DIAG_THREADS), 0, s, (const float2*)sb->dpart, (nb + 63) / 64, nx, m,
               (const int*)sb->e3, sb->dmat, sb->Dp, sb->nxp, sb->ed, sb->jkmax, 2LL * m * nb);
    DONOF_LAUNCH_CHECK(ctx);
  }
  if (mode == DONOF_RI_FULL) {
    // J_pq (a few CTAs, its own partial buffer) runs on the second stream beside the
    // full transform, on the SMs the latter leaves free; the shared-memory footprint
    // of both kinds keeps their CTAs off each other's SMs.
    cudaStream_t main_stream;
    const bool forked = fork_begin(ctx, &main_stream);
    int rcj;
    {
      ProfScope ps(ctx, DONOF_RI_ROW_J);
      rcj = launch_s4<S_JMO>(ctx);
      if (!rcj) {
        const S4Params& p = sb->plan[S_JMO];
        launch_pdl(reduce_jmo_kernel, dim3(ceil_div_u((long long)m * m, 256)), dim3(256), 0, ctx->stream,
                   (const long long*)p.partial, s4_slots(sb, S_JMO), m, (const int*)sb->ed, ctx->d_J);
        rcj = cudaGetLastError() == cudaSuccess ? DONOF_RI_OK : DONOF_RI_E_CUDA;
        ctx->launches++;
      }
    }
    if (forked) fork_end(ctx, main_stream);
    {
      ProfScope ps(ctx, DONOF_RI_ROW_FULL_K);
      if ((rc = launch_s4<S_FULLSQ>(ctx))) return rc;
      const S4Params& p = sb->plan[S_FULLSQ];
      launch_pdl(reduce_df_kernel, dim3(ceil_div_u((long long)m * m, 32)), dim3(32, 8), 0, s, (const float2*)p.partial,
                 s4_slots(sb, S_FULLSQ), m, m, ctx->d_K, (float2*)nullptr, (const double*)nullptr, (const float2*)nullptr);
      DONOF_LAUNCH_CHECK(ctx);
    }
    if (forked && (rc = fork_join(ctx))) return rc;
    if (rcj) return rcj;
  }
  return DONOF_RI_OK;
}

int s4_jk_ao(donof_ri_ctx* ctx) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, m = ctx->n_omega;
  int rc;
  if (sb->jk_merged && !ctx->prof_enabled) {
    // one persistent launch for every J^(q) and K^(q) unit.  Per-row profiling keeps the
    // two launches apart so that each row has its own events.
    if ((rc = launch_s4<S_JKAO>(ctx))) return rc;
  } else {
    {
      ProfScope ps(ctx, DONOF_RI_ROW_JAO);
      if ((rc = launch_s4<S_JAO>(ctx))) return rc;
    }
    {
      ProfScope ps(ctx, DONOF_RI_ROW_KAO);
      if ((rc = launch_s4<S_KAO>(ctx))) return rc;
    }
  }
  {
    ProfScope ps(ctx, DONOF_RI_ROW_OTHER);
    ProfScope pm(ctx, DONOF_RI_MEM_SPLIT);
    const size_t smem = sym_split_smem(nb);
    if (smem <= SMEM_BLOCK_BYTES) {
      launch_pdl(sym_split_kernel, dim3(2 * m), dim3(nb <= 48 ? 256 : smem <= 113 * 1024 ? 512 : 1024), smem, ctx->stream,
                 (const float*)sb->JKhi, (const float*)sb->JKlo, nb, sb->ldo, sb->JKp, sb->nbp, sb->eJK);
      DONOF_LAUNCH_CHECK(ctx);
      return DONOF_RI_OK;
    }
    const int T = (nb + 63) / 64;
    launch_pdl(sym_max_kernel, dim3((nb + 31) / 32, 2 * m), dim3(256), 0, ctx->stream, (const float*)sb->JKhi, nb, sb->ldo,
               sb->jkmax);
    DONOF_LAUNCH_CHECK(ctx);
    launch_pdl(sym_digits_kernel, dim3(T * (T + 1) / 2, 2 * m), dim3(256), 0, ctx->stream, (const float*)sb->JKhi,
               (const float*)sb->JKlo, nb, sb->ldo, (const unsigned int*)sb->jkmax, sb->JKp, sb->nbp, sb->eJK);
    DONOF_LAUNCH_CHECK(ctx);
  }
  return DONOF_RI_OK;
}

int s4_energy(donof_ri_ctx* ctx, int part) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, m = ctx->n_omega;
  cudaStream_t s = ctx->stream;
  int rc;
  ProfScope ps(ctx, DONOF_RI_ROW_ENERGY);
  if (part & ENERGY_PREP) {
    if ((rc = launch_occupations_coupling(ctx))) return rc;
    launch_pdl(fock_weights_df_kernel, dim3(ceil_div_u(2LL * m * m, 256)), dim3(256), 0, s, (const double*)ctx->d_A,
               (const double*)ctx->d_Bc, m, sb->W);
    DONOF_LAUNCH_CHECK(ctx);
    // (H' C')^T [p][mu'] as double-float pairs, from the prep's own double-float copy of
    // C' = L^T C (this part may run on a second stream beside the transform)
    const dim3 cg((nb + DFG_TJ - 1) / DFG_TJ, (m + DFG_TI - 1) / DFG_TI);
    if (nb <= DFG_FP64_A) {
      launch_pdl(df_gemm_nt_kernel<float2, double>, cg, dim3(DFG_THREADS), 0, s, m, nb, nb, (const double*)ctx->d_C, nb,
                 (const float2*)sb->LsTdf, nb, sb->Cdfp, nb);
    } else {
      launch_pdl(to_df_kernel, dim3(ceil_div_u((long long)m * nb, 256)), dim3(256), 0, s, (const double*)ctx->d_C,
                 (long long)m * nb, sb->Cinp);
      DONOF_LAUNCH_CHECK(ctx);
      launch_pdl(df_gemm_nt_kernel<float2, float2>, cg, dim3(DFG_THREADS), 0, s, m, nb, nb, (const float2*)sb->Cinp, nb,
                 (const float2*)sb->LsTdf, nb, sb->Cdfp, nb);
    }
    DONOF_LAUNCH_CHECK(ctx);
    launch_pdl(df_gemm_nt_kernel<float2, float2>, dim3((nb + DFG_TJ - 1) / DFG_TJ, (m + DFG_TI - 1) / DFG_TI), dim3(DFG_THREADS),
               0, s, m, nb, nb,
               (const float2*)sb->Cdfp, nb, (const float2*)sb->Hdf, nb, sb->HCt, nb);
    DONOF_LAUNCH_CHECK(ctx);
  }
  if (!(part & ENERGY_MAIN)) return DONOF_RI_OK;
  if ((rc = launch_s4<S_FOCK>(ctx))) return rc;
  const S4Params& p = sb->plan[S_FOCK];
  launch_pdl(reduce_df_kernel, dim3(ceil_div_u((long long)nb * m, 32)), dim3(32, 8), 0, s, (const float2*)p.partial,
             s4_slots(sb, S_FOCK), m, nb, (double*)nullptr, sb->Yt, (const double*)ctx->d_n, (const float2*)sb->HCt);
  DONOF_LAUNCH_CHECK(ctx);
  // lambda[p][q] = Y^T_p . C_q for every q < nbf
  launch_pdl(df_gemm_nt_kernel<double, float2>, dim3((nb + DFG_TJ - 1) / DFG_TJ, (m + DFG_TI - 1) / DFG_TI), dim3(DFG_THREADS),
             0, s, m, nb, nb,
             (const float2*)sb->Yt, nb, (const float2*)sb->Cdf, nb, ctx->d_lambda, nb);
  DONOF_LAUNCH_CHECK(ctx);
  launch_pdl(energy_terms_kernel, dim3(m), dim3(32), 0, s, nb, m, (const float2*)sb->Cdf, (const float2*)sb->HCt,
             (const double*)ctx->d_n, (const double*)ctx->d_lambda, (const double*)ctx->d_enuc, sb->eterm, sb->ticket,
             ctx->d_E);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

// ---------------------------------------------------------------------------
// Contracted Lagrangian on the digit path.  With w_pP = sum_q A_pq b^P_qq and
// X^P_qp = [q = p] w_pP - B_pq b^P_qp,
//   F^(p) C_p = n_p H C_p + sum_q sum_P X^P_qp b^P_{q .}
// (J^(q) C_p = sum_P b^P_qq b^P_{p .}, K^(q) C_p = sum_P b^P_{q .} b^P_qp), one
// digit-plane GEMM of N_b N_Omega^2 N_aux products (S_CTR) in place of J^(q),
// K^(q) and the Fock sum.  b^P_qp comes from the full transform's GEMM run once more
// with its store switched on, w from an FP64 GEMM, X's digits from
// ctr_digits_kernel; Y, lambda and E then as in s4_energy.
// ---------------------------------------------------------------------------
static int s4_ctr_setup(donof_ri_ctx* ctx) {
  S4Buffers* sb = ctx->s4;
  const long long nb = ctx->nbf, nx = ctx->naux, m = ctx->n_omega, nxp = sb->nxp;
  // every buffer and both tensor maps first, then the context's pointers: a failed
  // set-up leaves nothing behind and the next call starts again
  double *bf = nullptr, *wP = nullptr;
  __nv_bfloat16* Xd = nullptr;
  int* eX = nullptr;
  void* hws = nullptr;
  auto release = [&]() {
    cudaFree(bf);
    cudaFree(wP);
    cudaFree(Xd);
    cudaFree(eX);
    cudaFree(hws);
  };
  // digits of w = A d's operands (xgemm.cu: 40 us at 320 orbitals and 1680 auxiliary functions,
  // 330 by the FP64 kernel)
  const size_t hws_bytes = xgemm_operand_bytes((int)m, (int)m, 1) + xgemm_operand_bytes((int)nx, (int)m, 1);
  if (cudaMalloc((void**)&bf, (size_t)(nx * m * m * 8)) != cudaSuccess ||
      cudaMalloc((void**)&wP, (size_t)(m * nx * 8)) != cudaSuccess ||
      cudaMalloc((void**)&Xd, (size_t)(m * m * 4 * nxp * 2)) != cudaSuccess ||
      cudaMalloc((void**)&eX, (size_t)(m * m * 4)) != cudaSuccess || cudaMalloc(&hws, hws_bytes) != cudaSuccess) {
    cudaGetLastError();
    release();
    return DONOF_RI_E_OOM;
  }
  // A = L6 [m][nb][4][nxp] rows mu (per q) over P; B = X digits [m][m][4][nxp] rows p (per q) over P
  CUtensorMap ma, mb;
  int rc;
  if ((rc = s4_map_op(sb, &ma, sb->L6, (int)nx, (int)nb, (int)m, nxp, nb * 4 * nxp, S4_BM, 1)) ||
      (rc = s4_map_op(sb, &mb, Xd, (int)nx, (int)m, (int)m, nxp, m * 4 * nxp, S4_BN, 1))) {
    release();
    return rc;
  }
  S4Operands& op = sb->plan[S_CTR].op[0];
  op.a = ma; op.b = mb;
  op.nrows = (int)nb; op.nent = (int)m; op.ncols = (int)m; op.batched = 1;
  op.ea = sb->e6; op.eb = eX;
  sb->bf = bf; sb->wP = wP; sb->Xd = Xd; sb->eX = eX;
  ctx->d_hws = hws;
  ctx->hws_bytes = hws_bytes;
  return DONOF_RI_OK;
}

int s4_energy_contracted(donof_ri_ctx* ctx) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, nx = ctx->naux, m = ctx->n_omega;
  cudaStream_t s = ctx->stream;
  int rc;
  if (!sb->Xd && (rc = s4_ctr_setup(ctx))) return rc;
  // occupations, couplings A and B, (H' C')^T
  if ((rc = s4_energy(ctx, ENERGY_PREP))) return rc;
  ProfScope ps(ctx, DONOF_RI_ROW_ENERGY);
  {
    S4Params& pf = sb->plan[S_FULLSQ];
    pf.bfull = sb->bf;
    rc = launch_s4<S_FULLSQ>(ctx);
    pf.bfull = nullptr;
    if (rc) return rc;
  }
  Gemm64 g{};  // w[p][P] = sum_q A_pq d[q][P]
  g.M = m; g.N = nx; g.K = m; g.batch = 1;
  g.A = ctx->d_A; g.sAm = m; g.sAk = 1;
  g.B = sb->dmat; g.sBk = nx; g.sBn = 1;
  g.C = sb->wP; g.sCm = nx; g.sCn = 1;
  g.alpha = 1.0; g.beta = 0.0;
  if ((rc = launch_gemm64(ctx, g, ctx->d_hws, ctx->hws_bytes, 0))) return rc;
  launch_pdl(ctr_digits_kernel, dim3((m + 31) / 32, m), dim3(32, 8), 0, s, (const double*)sb->bf,
             (const double*)ctx->d_Bc, (const double*)sb->wP, m, nx, sb->nxp, sb->Xd, sb->eX);
  DONOF_LAUNCH_CHECK(ctx);
  if ((rc = launch_s4<S_CTR>(ctx))) return rc;
  const S4Params& p = sb->plan[S_CTR];
  launch_pdl(reduce_df_kernel, dim3(ceil_div_u((long long)nb * m, 32)), dim3(32, 8), 0, s, (const float2*)p.partial,
             s4_slots(sb, S_CTR), m, nb, (double*)nullptr, sb->Yt, (const double*)ctx->d_n, (const float2*)sb->HCt);
  DONOF_LAUNCH_CHECK(ctx);
  launch_pdl(df_gemm_nt_kernel<double, float2>, dim3((nb + DFG_TJ - 1) / DFG_TJ, (m + DFG_TI - 1) / DFG_TI), dim3(DFG_THREADS),
             0, s, m, nb, nb,
             (const float2*)sb->Yt, nb, (const float2*)sb->Cdf, nb, ctx->d_lambda, nb);
  DONOF_LAUNCH_CHECK(ctx);
  launch_pdl(energy_terms_kernel, dim3(m), dim3(32), 0, s, nb, m, (const float2*)sb->Cdf, (const float2*)sb->HCt,
             (const double*)ctx->d_n, (const double*)ctx->d_lambda, (const double*)ctx->d_enuc, sb->eterm, sb->ticket,
             ctx->d_E);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

// ---------------------------------------------------------------------------
// Autotuning: every digit-plane GEMM kind is timed on the live problem for each
// pipeline depth that fits its shared memory, the summed kinds (a3, a4, a7) also
// with twice the units.  Each timed launch starts from a flushed L2 (a 256 MB write
// outside the events), as inside an iteration, and a setting replaces the
// default only when it is at least 3 % faster.  Each launch rewrites its
// outputs, so the inputs stay valid.
// ---------------------------------------------------------------------------
template <int KIND>
static int s4_time(donof_ri_ctx* ctx, int reps, cudaEvent_t a, cudaEvent_t b, void* flush, size_t flush_bytes,
                   float* ms) {
  int rc;
  if ((rc = launch_s4<KIND>(ctx))) return rc;  // warm-up
  float total = 0.f;
  for (int r = 0; r < reps; ++r) {
    DONOF_CUDA_TRY(cudaMemsetAsync(flush, r & 255, flush_bytes, ctx->stream));
    DONOF_CUDA_TRY(cudaEventRecord(a, ctx->stream));
    if ((rc = launch_s4<KIND>(ctx))) return rc;
    DONOF_CUDA_TRY(cudaEventRecord(b, ctx->stream));
    DONOF_CUDA_TRY(cudaEventSynchronize(b));
    float t = 0.f;
    DONOF_CUDA_TRY(cudaEventElapsedTime(&t, a, b));
    total += t;
  }
  *ms = total / reps;
  return DONOF_RI_OK;
}

static bool s4_has_options(int kind) { return kind == S_FULLSQ || kind == S_JMO || kind == S_FOCK; }

template <int KIND>
static int s4_tune_kind(donof_ri_ctx* ctx, int reps, cudaEvent_t a, cudaEvent_t b, void* flush, size_t fbytes,
                        int* report, int* tried) {
  S4Buffers* sb = ctx->s4;
  S4Params& p = sb->plan[KIND];
  const int dS = p.stages, dO = sb->opt[KIND];
  int bestS = dS, bestO = dO, rc;
  float best = 1e30f, dflt = 1e30f;
  for (int o = 0; o < (s4_has_options(KIND) ? 2 : 1); ++o) {
    s4_use(sb, KIND, o);
    for (int S = 2; S <= S4_MAX_STAGES; ++S) {
      p.stages = S;
      float ms = 0.f;
      if ((rc = s4_time<KIND>(ctx, reps, a, b, flush, fbytes, &ms))) return rc;
      ++*tried;
      if (S == dS && o == dO) dflt = ms;
      if (ms < best) {
        best = ms;
        bestS = S;
        bestO = o;
      }
    }
  }
  if (!(best < 0.97f * dflt)) {  // keep the default unless clearly beaten
    best = dflt;
    bestS = dS;
    bestO = dO;
  }
  p.stages = bestS;
  s4_use(sb, KIND, bestO);
  if (report) {
    const S4Slots& sl = s4_slots(sb, KIND);
    report[KIND * 4 + 0] = bestS;
    report[KIND * 4 + 1] = s4_has_options(KIND) ? std::max(sl.pair, sl.single) : (KIND == S_JAO ? 1 : 0);
    report[KIND * 4 + 2] = s4_grid(p);
    report[KIND * 4 + 3] = (int)(best * 1000.f + 0.5f);  // microseconds
  }
  return DONOF_RI_OK;
}

// A kind's schedule set by the caller (the choices the autotuner makes): pipeline
// depth, and option = 1 or 2 for the summed kinds (the default units, or units of half
// the batches), one launch together with J^(q) (1) or its own (0) for K^(q).  The half
// transform and J^(q) have one kernel whatever the option, which is 0 or 1 because callers
// pass either; so is the limit of 2 stages on the half transform's option 0.
int s4_set_schedule(donof_ri_ctx* ctx, int kind, int stages, int option) {
  S4Buffers* sb = ctx->s4;
  if (kind < 0 || kind > S_FOCK) return DONOF_RI_E_ARG;
  const bool split = (kind == S_FULLSQ || kind == S_JMO || kind == S_FOCK);
  if (stages < 2 || stages > (kind == S_HALF && option != 1 ? 2 : 4)) return DONOF_RI_E_ARG;
  if (split ? (option != 1 && option != 2)
            : ((kind == S_JAO || kind == S_HALF || kind == S_KAO) ? (option != 0 && option != 1) : option != 0))
    return DONOF_RI_E_ARG;
  sb->plan[kind].stages = std::min(stages, S4_MAX_STAGES);
  if (kind == S_KAO) sb->jk_merged = option;
  if (split) s4_use(sb, kind, option - 1);
  if (kind == S_JAO || kind == S_KAO) s4_plan_jkao(sb);
  return DONOF_RI_OK;
}

// J^(q) and K^(q) as one launch or as two, each timed from a
// flushed L2; the merged launch stays unless the pair of launches is 3 % faster.
static int s4_tune_jk_merge(donof_ri_ctx* ctx, int reps, cudaEvent_t a, cudaEvent_t b, void* flush, size_t fbytes,
                            int* tried) {
  S4Buffers* sb = ctx->s4;
  float t[2] = {0.f, 0.f};
  int rc;
  for (int merged = 0; merged < 2; ++merged) {
    sb->jk_merged = merged;
    for (int r = 0; r <= reps; ++r) {  // r = 0: warm-up
      DONOF_CUDA_TRY(cudaMemsetAsync(flush, r & 255, fbytes, ctx->stream));
      DONOF_CUDA_TRY(cudaEventRecord(a, ctx->stream));
      if (merged) {
        if ((rc = launch_s4<S_JKAO>(ctx))) return rc;
      } else {
        if ((rc = launch_s4<S_JAO>(ctx))) return rc;
        if ((rc = launch_s4<S_KAO>(ctx))) return rc;
      }
      DONOF_CUDA_TRY(cudaEventRecord(b, ctx->stream));
      DONOF_CUDA_TRY(cudaEventSynchronize(b));
      float ms = 0.f;
      DONOF_CUDA_TRY(cudaEventElapsedTime(&ms, a, b));
      if (r > 0) t[merged] += ms;
    }
    ++*tried;
  }
  sb->jk_merged = (t[0] < 0.97f * t[1]) ? 0 : 1;
  return DONOF_RI_OK;
}

int s4_autotune(donof_ri_ctx* ctx, int reps, int* report, int* tried) {
  const size_t fbytes = (size_t)256 << 20;
  void* flush = nullptr;
  if (cudaMalloc(&flush, fbytes) != cudaSuccess) {
    cudaGetLastError();
    return DONOF_RI_E_OOM;
  }
  cudaEvent_t a, b;
  if (cudaEventCreate(&a) != cudaSuccess) {
    cudaFree(flush);
    return DONOF_RI_E_CUDA;
  }
  if (cudaEventCreate(&b) != cudaSuccess) {
    cudaEventDestroy(a);
    cudaFree(flush);
    return DONOF_RI_E_CUDA;
  }
  int rc = DONOF_RI_OK;
  *tried = 0;
  if (!rc) rc = s4_tune_kind<S_HALF>(ctx, reps, a, b, flush, fbytes, report, tried);
  if (!rc) rc = s4_tune_kind<S_FULLSQ>(ctx, reps, a, b, flush, fbytes, report, tried);
  if (!rc) rc = s4_tune_kind<S_JMO>(ctx, reps, a, b, flush, fbytes, report, tried);
  if (!rc) rc = s4_tune_kind<S_JAO>(ctx, reps, a, b, flush, fbytes, report, tried);
  if (!rc) rc = s4_tune_kind<S_KAO>(ctx, reps, a, b, flush, fbytes, report, tried);
  if (!rc) rc = s4_tune_kind<S_FOCK>(ctx, reps, a, b, flush, fbytes, report, tried);
  s4_plan_jkao(ctx->s4);  // the merged J^(q) + K^(q) launch follows the tuned tile lists
  if (!rc) rc = s4_tune_jk_merge(ctx, reps, a, b, flush, fbytes, tried);
  if (!rc && report) report[S_KAO * 4 + 1] = ctx->s4->jk_merged;
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cudaFree(flush);
  return rc;
}

int s4_fetch(donof_ri_ctx* ctx, int what, double* dst, size_t count) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, nx = ctx->naux, m = ctx->n_omega;
  cudaError_t e = cudaSuccess;
  if (what == DONOF_RI_FETCH_BHALF) {
    double* tmp = nullptr;
    if (cudaMalloc((void**)&tmp, count * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      return DONOF_RI_E_OOM;
    }
    double* ao = nullptr;
    if (cudaMalloc((void**)&ao, count * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      cudaFree(tmp);
      return DONOF_RI_E_OOM;
    }
    // rows (P, p) of the L3 digits over nu'; consecutive P are mp rows apart
    for (int P = 0; P < nx && e == cudaSuccess; ++P) {
      unslice_kernel<<<ceil_div_u((long long)m * nb, 256), 256, 0, ctx->stream>>>(
          sb->L3 + (size_t)P * sb->mp * 4 * sb->nbp, sb->nbp, sb->e3 + (size_t)P * m, m, nb,
          tmp + (size_t)P * m * nb);
      e = cudaGetLastError();
    }
    // back to the AO basis: b^P_{p nu} = sum_nu' b'^P_{p nu'} L_{nu nu'}
    int rc = DONOF_RI_OK;
    if (e == cudaSuccess) {
      Gemm64 g{};
      g.M = nx * m; g.N = nb; g.K = nb; g.batch = 1;
      g.A = tmp; g.sAm = nb; g.sAk = 1;
      g.B = sb->Ls; g.sBk = 1; g.sBn = nb;
      g.C = ao; g.sCm = nb; g.sCn = 1;
      g.alpha = 1.0; g.beta = 0.0;
      rc = launch_dgemm(ctx, g);
    }
    if (e == cudaSuccess && !rc) e = cudaMemcpyAsync(dst, ao, count * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    cudaFree(tmp);
    cudaFree(ao);
    if (rc) return rc;
    return e == cudaSuccess ? DONOF_RI_OK : DONOF_RI_E_CUDA;
  }
  // d is kept as FP64 [p][P]; the fetch layout is [P][p]
  double* hostbuf = (double*)malloc(count * sizeof(double));
  if (!hostbuf) return DONOF_RI_E_OOM;
  e = cudaMemcpyAsync(hostbuf, sb->dmat, count * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e == cudaSuccess)
    for (int P = 0; P < nx; ++P)
      for (int pc = 0; pc < m; ++pc) dst[(size_t)P * m + pc] = hostbuf[(size_t)pc * nx + P];
  free(hostbuf);
  return e == cudaSuccess ? DONOF_RI_OK : DONOF_RI_E_CUDA;
}

int s4_copy_ao(donof_ri_ctx* ctx, double* Jao, double* Kao, bool jao_dev, bool kao_dev) {
  S4Buffers* sb = ctx->s4;
  const int nb = ctx->nbf, m = ctx->n_omega;
  const size_t n = (size_t)m * nb * nb;
  double *tmp = nullptr, *tmp2 = nullptr;
  if (cudaMalloc((void**)&tmp, n * sizeof(double)) != cudaSuccess ||
      cudaMalloc((void**)&tmp2, n * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    if (tmp) cudaFree(tmp);
    return DONOF_RI_E_OOM;
  }
  cudaError_t e = cudaSuccess;
  for (int which = 0; which < 2 && e == cudaSuccess; ++which) {
    double* dst = which == 0 ? Jao : Kao;
    bool dev = which == 0 ? jao_dev : kao_dev;
    if (!dst) continue;
    size_t off = (size_t)which * m * nb * sb->ldo;
    join_sym_kernel<<<ceil_div_u((long long)n, 256), 256, 0, ctx->stream>>>(sb->JKhi + off, sb->JKlo + off, m, nb,
                                                                             sb->ldo, tmp);
    e = cudaGetLastError();
    // back to the AO basis: X^(q) = L X'^(q) L^T for every orbital q
    if (e == cudaSuccess) {
      const long long n2 = (long long)nb * nb;
      Gemm64 g{};
      g.M = nb; g.N = nb; g.K = nb; g.batch = m;
      g.A = sb->Ls; g.sAb = 0; g.sAm = nb; g.sAk = 1;
      g.B = tmp; g.sBb = n2; g.sBk = nb; g.sBn = 1;
      g.C = tmp2; g.sCb = n2; g.sCm = nb; g.sCn = 1;
      g.alpha = 1.0; g.beta = 0.0;
      int rc = launch_dgemm(ctx, g);
      Gemm64 h{};
      h.M = nb; h.N = nb; h.K = nb; h.batch = m;
      h.A = tmp2; h.sAb = n2; h.sAm = nb; h.sAk = 1;
      h.B = sb->Ls; h.sBb = 0; h.sBk = 1; h.sBn = nb;  // element (k, n) of L^T = L[n][k]
      h.C = tmp; h.sCb = n2; h.sCm = nb; h.sCn = 1;
      h.alpha = 1.0; h.beta = 0.0;
      if (!rc) rc = launch_dgemm(ctx, h);
      if (rc) {
        cudaFree(tmp);
        cudaFree(tmp2);
        return rc;
      }
    }
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(dst, tmp, n * sizeof(double), dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                          ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  }
  cudaFree(tmp);
  cudaFree(tmp2);
  return e == cudaSuccess ? DONOF_RI_OK : DONOF_RI_E_CUDA;
}

}  // namespace donof
