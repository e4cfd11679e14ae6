// Setup on the device, all FP64: s-type Gaussian integrals, the Cholesky
// factorisation of the Coulomb metric and the fitted three-index tensor.
//
// Paper: Table 2 / Table 3 steps 0-1 (evaluation of (mu nu|k), G_kl = (k|l)
// and the solve for b), Eq. (AOERI), Sec. 3 (integrals evaluated once and
// stored).  The engine factorises G = L L^T with a plain Cholesky (no
// pivoting, no eigenvalue correction) and forms B = L^-1 (Q|mu nu).
#include "common.cuh"
#include "numeric.cuh"
#include "pairs.cuh"

#include <math.h>

namespace donof {

// ---------------------------------------------------------------------------
// Generic strided batched FP64 GEMM (CUDA cores).  T x T output tile per CTA, 256
// threads, (T / 16)^2 outputs per thread, K staged through shared memory in slices of
// 16.  Loads are ordered along whichever operand stride is unit so that global reads
// coalesce for every layout the engine uses.  Every output is one chain of FMAs in k
// order, whatever T.
//
// T = 64 keeps the FP64 pipe (2 lanes a clock per SM) at 85-90 % while there are CTAs for
// every SM; a product with fewer 64 x 64 tiles than two per SM (H C at nbf 720, 400
// orbitals: 84 tiles, 700 us) takes T = 32 (299 tiles; all of an energy and gradient of the
// occupations with this product: 490 us).
// ---------------------------------------------------------------------------
constexpr int DG_TK = 16;

template <int T>
__global__ void __launch_bounds__(256) dgemm_kernel(Gemm64 g) {
  constexpr int R = T / 16, L = T / 16;  // outputs per thread and dimension; loads per thread
  __shared__ double As[DG_TK][T + 1];
  __shared__ double Bs[DG_TK][T + 1];
  const int b = blockIdx.z;
  const int m0 = blockIdx.y * T;
  const int n0 = blockIdx.x * T;
  if (g.lower && n0 >= m0 + T) return;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const double* A = g.A + (long long)b * g.sAb;
  const double* B = g.B + (long long)b * g.sBb;
  double acc[R][R];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) acc[i][j] = 0.0;

  for (int k0 = 0; k0 < g.K; k0 += DG_TK) {
#pragma unroll
    for (int it = 0; it < L; ++it) {
      int e = threadIdx.x + it * 256;
      int mm, kk;
      if (g.sAm == 1) { mm = e % T; kk = e / T; } else { kk = e % DG_TK; mm = e / DG_TK; }
      int gm = m0 + mm, gk = k0 + kk;
      As[kk][mm] = (gm < g.M && gk < g.K) ? A[(long long)gm * g.sAm + (long long)gk * g.sAk] : 0.0;
      int nn;
      if (g.sBn == 1) { nn = e % T; kk = e / T; } else { kk = e % DG_TK; nn = e / DG_TK; }
      int gn = n0 + nn;
      gk = k0 + kk;
      Bs[kk][nn] = (gn < g.N && gk < g.K) ? B[(long long)gk * g.sBk + (long long)gn * g.sBn] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < DG_TK; ++kk) {
      double a[R], bb[R];
#pragma unroll
      for (int i = 0; i < R; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < R; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }
  double* C = g.C + (long long)b * g.sCb;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int m = m0 + ty + 16 * i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      int n = n0 + tx + 16 * j;
      if (n >= g.N) continue;
      double* c = C + (long long)m * g.sCm + (long long)n * g.sCn;
      double v = g.alpha * acc[i][j];
      if (g.beta != 0.0) v += g.beta * (*c);
      *c = v;
    }
  }
}

int launch_dgemm(donof_ri_ctx* ctx, const Gemm64& g) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return DONOF_RI_OK;
  if (g.K <= 0) return DONOF_RI_E_ARG;
  const long long tiles64 = ((g.M + 63LL) / 64) * ((g.N + 63LL) / 64) * g.batch;
  const int T = tiles64 < 2 * 152 ? 32 : 64;
  long long gy = (g.M + T - 1) / T;
  if (gy > 65535 || g.batch > 65535) return DONOF_RI_E_ARG;
  dim3 grid(ceil_div_u(g.N, T), (unsigned)gy, (unsigned)g.batch);
  if (T == 32) dgemm_kernel<32><<<grid, 256, 0, ctx->stream>>>(g);
  else dgemm_kernel<64><<<grid, 256, 0, ctx->stream>>>(g);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

// ---------------------------------------------------------------------------
// Integrals over normalised s-type Gaussians.
//   orbital basis:   N_a = (2a/pi)^(3/4)
//   auxiliary basis: N_k = (2k/pi)^(3/4) sqrt(k / (4 pi))   ((k|k) = 1)
// Boys F0(T) = 1/2 sqrt(pi/T) erf(sqrt(T)), with the series 1 - T/3 + T^2/10
// below T = 1e-8.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double boys_f0(double t) {
  if (t < 1e-8) return 1.0 - t / 3.0 + t * t / 10.0;
  double st = sqrt(t);
  return 0.5 * sqrt(M_PI / t) * erf(st);
}

__device__ __forceinline__ double norm_orb(double a) { return pow(2.0 * a / M_PI, 0.75); }
__device__ __forceinline__ double norm_aux(double k) {
  return pow(2.0 * k / M_PI, 0.75) * sqrt(k / (4.0 * M_PI));
}

// S, H = T + V for every orbital pair.
__global__ void one_electron_kernel(int nbf, int n_atoms, const double* xyz, const double* charge,
                                    const int* bf_atom, const double* bf_alpha, double* S, double* H) {
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)nbf * nbf) return;
  int i = (int)(idx / nbf), j = (int)(idx % nbf);
  double a = bf_alpha[i], b = bf_alpha[j];
  const double* A = xyz + 3 * bf_atom[i];
  const double* Bc = xyz + 3 * bf_atom[j];
  double p = a + b, mu = a * b / p;
  double dx = A[0] - Bc[0], dy = A[1] - Bc[1], dz = A[2] - Bc[2];
  double r2 = dx * dx + dy * dy + dz * dz;
  double kab = exp(-mu * r2);
  double nn = norm_orb(a) * norm_orb(b);
  double s = nn * pow(M_PI / p, 1.5) * kab;
  double t = nn * mu * (3.0 - 2.0 * mu * r2) * pow(M_PI / p, 1.5) * kab;
  double Px = (a * A[0] + b * Bc[0]) / p, Py = (a * A[1] + b * Bc[1]) / p, Pz = (a * A[2] + b * Bc[2]) / p;
  double v = 0.0;
  for (int c = 0; c < n_atoms; ++c) {
    double ex = Px - xyz[3 * c], ey = Py - xyz[3 * c + 1], ez = Pz - xyz[3 * c + 2];
    v -= charge[c] * nn * (2.0 * M_PI / p) * kab * boys_f0(p * (ex * ex + ey * ey + ez * ez));
  }
  S[idx] = s;
  H[idx] = t + v;
}

// G_kl = (k|l) over the auxiliary basis.  A 32 x 32 tile on or below the diagonal per block
// (every factor is symmetric in k and l to the last bit), the norms once per tile: 560 -> 181 us
// at 840 functions.
__global__ void __launch_bounds__(256) metric_kernel(int naux, const double* xyz, const int* aux_atom,
                                                     const double* aux_alpha, double* G) {
  __shared__ double nrm[2][32], t[32][33];
  if (blockIdx.x > blockIdx.y) return;
  const int k0 = blockIdx.y * 32, l0 = blockIdx.x * 32, tx = threadIdx.x, ty = threadIdx.y;
  if (ty < 2) {
    const int i = (ty == 0 ? k0 : l0) + tx;
    if (i < naux) nrm[ty][tx] = norm_aux(aux_alpha[i]);
  }
  __syncthreads();
  const double two_pi52 = 2.0 * pow(M_PI, 2.5);
  const int l = l0 + tx;
  for (int y = ty; y < 32; y += 8) {
    const int k = k0 + y;
    if (k >= naux || l >= naux) continue;
    double c = aux_alpha[k], d = aux_alpha[l];
    const double* X = xyz + 3 * aux_atom[k];
    const double* Y = xyz + 3 * aux_atom[l];
    double dx = X[0] - Y[0], dy = X[1] - Y[1], dz = X[2] - Y[2];
    double r2 = dx * dx + dy * dy + dz * dz;
    const double pref = two_pi52 / (c * d * sqrt(c + d));
    const double g = nrm[0][y] * nrm[1][tx] * pref * boys_f0(c * d / (c + d) * r2);
    G[(size_t)k * naux + l] = g;
    t[y][tx] = g;
  }
  __syncthreads();
  if (blockIdx.x == blockIdx.y) return;
  for (int y = ty; y < 32; y += 8)
    if (l0 + y < naux && k0 + tx < naux) G[(size_t)(l0 + y) * naux + k0 + tx] = t[tx][y];
}

// (k|mu nu) into out[k][mu][nu].
__global__ void eri3_kernel(int nbf, int naux, const double* xyz, const int* bf_atom, const double* bf_alpha,
                            const int* aux_atom, const double* aux_alpha, double* out) {
  long long nb2 = (long long)nbf * nbf;
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)naux * nb2) return;
  int k = (int)(idx / nb2);
  int rem = (int)(idx % nb2);
  int i = rem / nbf, j = rem % nbf;
  double a = bf_alpha[i], b = bf_alpha[j], c = aux_alpha[k];
  const double* A = xyz + 3 * bf_atom[i];
  const double* Bc = xyz + 3 * bf_atom[j];
  const double* Cc = xyz + 3 * aux_atom[k];
  double p = a + b, mu = a * b / p;
  double dx = A[0] - Bc[0], dy = A[1] - Bc[1], dz = A[2] - Bc[2];
  double kab = exp(-mu * (dx * dx + dy * dy + dz * dz));
  double Px = (a * A[0] + b * Bc[0]) / p, Py = (a * A[1] + b * Bc[1]) / p, Pz = (a * A[2] + b * Bc[2]) / p;
  double ex = Px - Cc[0], ey = Py - Cc[1], ez = Pz - Cc[2];
  double pref = 2.0 * pow(M_PI, 2.5) / (p * c * sqrt(p + c));
  out[idx] = norm_orb(a) * norm_orb(b) * norm_aux(c) * pref * kab *
             boys_f0(p * c / (p + c) * (ex * ex + ey * ey + ez * ez));
}

// Tiles of 16 x 16 pairs (mu, nu) on and above the diagonal.
constexpr int PAIR_T = 16;
// Tile t of the pairs: t = J (J + 1) / 2 + I, I <= J.
__device__ __forceinline__ void pair_tile(int t, int& I, int& J) {
  J = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((J + 1) * (J + 2) / 2 <= t) ++J;
  while (J * (J + 1) / 2 > t) --J;
  I = t - J * (J + 1) / 2;
}

// ---------------------------------------------------------------------------
// The three-centre integrals of the larger contexts.  FP64 is the bound (two lanes a clock per
// SM), so the kernel above, which takes three powers, an exponential, an error function and
// half a dozen roots and quotients for every (k|mu nu) of both triangles, ran at 49 ms for 840
// x 240 x 240.  Here a thread keeps one pair (mu <= nu) and runs over auxiliary functions:
//   (k|mu nu) = [N_mu N_nu 2 pi^(5/2) K_ab / p] [N_k / c] (p + c)^(-1/2) F0(p c r^2 / (p + c)),
// the brackets once per pair and function, and F0 from its Taylor series about the nearest
// multiple of 1/16 below 36,
//   F0(t) = sum_k F_k(t0) (t0 - t)^k / k!  (dF_k/dt = -F_{k+1}), k <= 7: next term below 1.4e-18,
// and (pi / t)^(1/2) / 2 from there on (erfc(6) = 2e-17): about 30 FP64 instructions, 1.9 ms; errors as the kernel above
// (1.8e-15 rms against exact, from the rounded exponents).
// From 256 auxiliary functions on, like the fit (below it the sums and integrals keep their
// bits, see path64_init), and not for TF32X3, which rounds B to FP32: other last bits of B move
// its results by 1e-9, as far as a rearranged FP32 sum would.
// ---------------------------------------------------------------------------
constexpr int BOYS_N = 8, BOYS_PER = 16, BOYS_MAX = 36, BOYS_ROWS = BOYS_MAX * BOYS_PER + 1;

// F_k(t0) / k!: F_7 from its ascending series (positive terms), the others by the downward
// recursion F_{k-1} = (2 t F_k + e^-t) / (2 k - 1); F_0, the only one whose last bits reach the
// result, from its closed form.
__global__ void boys_table_kernel(double* tab) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= BOYS_ROWS) return;
  const double t = (double)i / BOYS_PER, e = exp(-t);
  double term = 1.0 / (2 * BOYS_N - 1), s = term;
  for (int j = 1; j < 400 && term > 1e-18 * s; ++j) {
    term *= 2.0 * t / (2 * (BOYS_N - 1 + j) + 1);
    s += term;
  }
  double F[BOYS_N], fact = 1.0;
  F[BOYS_N - 1] = e * s;
  for (int k = BOYS_N - 1; k > 0; --k) F[k - 1] = (2.0 * t * F[k] + e) / (2 * k - 1);
  for (int k = 0; k < BOYS_N; ++k) {
    if (k) fact *= k;
    tab[i * BOYS_N + k] = k ? F[k] / fact : boys_f0(t);
  }
}

__device__ __forceinline__ double boys_f0_tab(double t, const double* __restrict__ tab) {
  if (!(t < (double)BOYS_MAX)) return 0.886226925452758014 * rsqrt(t);
  constexpr double R = 6755399441055744.0;  // 1.5 2^52: the sum's low bits are the rounded integer
  const double u = fma(t, (double)BOYS_PER, R);
  const double d = fma(u - R, 1.0 / BOYS_PER, -t);
  const double2* f = (const double2*)(tab + (unsigned int)__double_as_longlong(u) * BOYS_N);
  const double2 f0 = __ldg(f), f2 = __ldg(f + 1), f4 = __ldg(f + 2), f6 = __ldg(f + 3);
  double v = fma(f6.y, d, f6.x);
  v = fma(v, d, f4.y);
  v = fma(v, d, f4.x);
  v = fma(v, d, f2.y);
  v = fma(v, d, f2.x);
  v = fma(v, d, f0.y);
  return fma(v, d, f0.x);
}

constexpr int ERI_K = 64, ERI_U = 4;  // auxiliary functions per block, and per turn through shared memory
__global__ void __launch_bounds__(256) eri3_pairs_kernel(int nbf, int naux, const double* __restrict__ xyz,
                                                         const int* __restrict__ bf_atom,
                                                         const double* __restrict__ bf_alpha,
                                                         const int* __restrict__ aux_atom,
                                                         const double* __restrict__ aux_alpha,
                                                         const double* __restrict__ tab, double* __restrict__ out) {
  __shared__ double ks[5][ERI_K];
  __shared__ double s[ERI_U][PAIR_T][PAIR_T + 1];
  int I, J;
  pair_tile(blockIdx.x, I, J);
  const int a = threadIdx.x / PAIR_T, b = threadIdx.x % PAIR_T;
  const int mu = I * PAIR_T + a, nu = J * PAIR_T + b, k0 = blockIdx.y * ERI_K, nk = min(ERI_K, naux - k0);
  if (threadIdx.x < nk) {
    const double c = aux_alpha[k0 + threadIdx.x];
    const double* C = xyz + 3 * aux_atom[k0 + threadIdx.x];
    ks[0][threadIdx.x] = C[0];
    ks[1][threadIdx.x] = C[1];
    ks[2][threadIdx.x] = C[2];
    ks[3][threadIdx.x] = c;
    ks[4][threadIdx.x] = norm_aux(c) / c;
  }
  double p = 1.0, f = 0.0, Px = 0.0, Py = 0.0, Pz = 0.0;
  if (mu < nbf && nu < nbf) {
    const int i = min(mu, nu), j = max(mu, nu);
    const double ea = bf_alpha[i], eb = bf_alpha[j];
    const double *A = xyz + 3 * bf_atom[i], *B = xyz + 3 * bf_atom[j];
    p = ea + eb;
    const double dx = A[0] - B[0], dy = A[1] - B[1], dz = A[2] - B[2];
    f = norm_orb(ea) * norm_orb(eb) * exp(-ea * eb / p * (dx * dx + dy * dy + dz * dz)) * (2.0 * pow(M_PI, 2.5) / p);
    Px = (ea * A[0] + eb * B[0]) / p;
    Py = (ea * A[1] + eb * B[1]) / p;
    Pz = (ea * A[2] + eb * B[2]) / p;
  }
  __syncthreads();
  const size_t n2 = (size_t)nbf * nbf;
  double* o = out + (size_t)k0 * n2 + (size_t)mu * nbf + nu;
  double* ot = out + (size_t)k0 * n2 + (size_t)(J * PAIR_T + a) * nbf + I * PAIR_T + b;
  const bool st = mu < nbf && nu < nbf, stt = I != J && J * PAIR_T + a < nbf && I * PAIR_T + b < nbf;
  for (int k = 0; k < nk; k += ERI_U) {
    double v[ERI_U];
#pragma unroll
    for (int u = 0; u < ERI_U; ++u) {
      const int q = min(k + u, nk - 1);
      const double c = ks[3][q], ex = Px - ks[0][q], ey = Py - ks[1][q], ez = Pz - ks[2][q];
      const double w = rsqrt(p + c);
      const double r2 = fma(ex, ex, fma(ey, ey, ez * ez));
      v[u] = f * ks[4][q] * w * boys_f0_tab(p * c * (w * w) * r2, tab);
    }
#pragma unroll
    for (int u = 0; u < ERI_U; ++u) s[u][a][b] = v[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < ERI_U; ++u)
      if (k + u < nk) {
        if (st) o[(size_t)(k + u) * n2] = v[u];
        if (stt) ot[(size_t)(k + u) * n2] = s[u][b][a];
      }
    __syncthreads();
  }
}

// E_nuc: the terms in parallel, their sum by one thread in the order i, j < i.
__global__ void __launch_bounds__(256) enuc_kernel(int n_atoms, const double* xyz, const double* charge, double* out) {
  __shared__ double term[1024];
  double e = 0.0;
  const long long n = pair_count(n_atoms);
  for (long long t0 = 0; t0 < n; t0 += 1024) {
    const int nt = (int)min(1024LL, n - t0);
    for (int q = threadIdx.x; q < nt; q += 256) {
      int i, j;
      pair_at(t0 + q, i, j);
      double dx = xyz[3 * i] - xyz[3 * j], dy = xyz[3 * i + 1] - xyz[3 * j + 1], dz = xyz[3 * i + 2] - xyz[3 * j + 2];
      term[q] = charge[i] * charge[j] / sqrt(dx * dx + dy * dy + dz * dz);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll 8
      for (int q = 0; q < nt; ++q) e += term[q];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = e;
}

int setup_integrals(donof_ri_ctx* ctx) {
  const int nb = ctx->nbf, nx = ctx->naux;
  long long n1 = (long long)nb * nb;
  one_electron_kernel<<<ceil_div_u(n1, 256), 256, 0, ctx->stream>>>(
      nb, ctx->n_atoms, ctx->d_atom_xyz, ctx->d_atom_charge, ctx->d_bf_atom, ctx->d_bf_alpha, ctx->d_S, ctx->d_H);
  DONOF_LAUNCH_CHECK(ctx);
  const unsigned int mt = (nx + 31) / 32;
  metric_kernel<<<dim3(mt, mt), dim3(32, 8), 0, ctx->stream>>>(nx, ctx->d_atom_xyz, ctx->d_aux_atom, ctx->d_aux_alpha,
                                                               ctx->d_G);
  DONOF_LAUNCH_CHECK(ctx);
  if (nx >= 256 && ctx->precision != DONOF_RI_TF32X3) {
    double* tab = nullptr;
    const size_t bytes = BOYS_ROWS * BOYS_N * sizeof(double);
    const int rc = xgemm_workspace(ctx, bytes, bytes, (void**)&tab);
    if (rc) return rc;
    boys_table_kernel<<<(BOYS_ROWS + 63) / 64, 64, 0, ctx->stream>>>(tab);
    DONOF_LAUNCH_CHECK(ctx);
    const int T = (nb + PAIR_T - 1) / PAIR_T;
    eri3_pairs_kernel<<<dim3(T * (T + 1) / 2, (nx + ERI_K - 1) / ERI_K), 256, 0, ctx->stream>>>(
        nb, nx, ctx->d_atom_xyz, ctx->d_bf_atom, ctx->d_bf_alpha, ctx->d_aux_atom, ctx->d_aux_alpha, tab, ctx->d_B);
    DONOF_LAUNCH_CHECK(ctx);
  } else {
    const long long n3 = (long long)nx * n1;
    eri3_kernel<<<ceil_div_u(n3, 256), 256, 0, ctx->stream>>>(nb, nx, ctx->d_atom_xyz, ctx->d_bf_atom,
                                                               ctx->d_bf_alpha, ctx->d_aux_atom,
                                                               ctx->d_aux_alpha, ctx->d_B);
    DONOF_LAUNCH_CHECK(ctx);
  }
  enuc_kernel<<<1, 256, 0, ctx->stream>>>(ctx->n_atoms, ctx->d_atom_xyz, ctx->d_atom_charge, ctx->d_enuc);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

// ---------------------------------------------------------------------------
// Blocked right-looking Cholesky of G (row-major, lower factor in place).
// ---------------------------------------------------------------------------
constexpr int CH_NB = 64;

__global__ void max_diag_kernel(int n, const double* G, double* out) {
  __shared__ double red[256];
  double m = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, G[(long long)i * n + i]);
  red[threadIdx.x] = m;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

// Factor the nbk x nbk diagonal block at (k0, k0) in shared memory.  A pivot
// below rel_min * max(diag G) sets DEV_METRIC_NOT_PD (the factorisation then
// continues on a clamped pivot so that the kernel always terminates).
__global__ void __launch_bounds__(1024) potrf_block_kernel(int n, double* G, int k0, int nbk, const double* maxdiag,
                                                          double rel_min, int* status) {
  __shared__ double s[CH_NB][CH_NB + 1], dg[CH_NB];
  for (int e = threadIdx.x; e < nbk * nbk; e += blockDim.x) {
    int i = e / nbk, j = e % nbk;
    s[i][j] = G[(long long)(k0 + i) * n + k0 + j];
  }
  __syncthreads();
  // Right-looking, a warp per row of the trailing block (FP64 issues two lanes a clock, so the
  // 44 k multiplications of a block are its bound): 98 -> 79 us per block, most of
  // it the root and the quotient that each column waits for.
  const double thresh = rel_min * (*maxdiag);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int j = 0; j < nbk; ++j) {
    if (threadIdx.x < CH_NB) {
      double d = s[j][j];
      if (!(d > thresh)) {
        if (threadIdx.x == 0) atomicCAS(status, 0, (int)DEV_METRIC_NOT_PD);
        d = fmax(thresh, 1e-300);
      }
      d = sqrt(d);
      if (threadIdx.x == 0) dg[j] = d;
      const int i = j + 1 + threadIdx.x;
      if (i < nbk) s[i][j] /= d;
    }
    __syncthreads();
    for (int i = j + 1 + warp; i < nbk; i += 32) {
      const double sij = s[i][j];
      for (int k = j + 1 + lane; k <= i; k += 32) s[i][k] -= sij * s[k][j];
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < nbk * nbk; e += blockDim.x) {
    int i = e / nbk, j = e % nbk;
    G[(long long)(k0 + i) * n + k0 + j] = (j < i) ? s[i][j] : j == i ? dg[i] : 0.0;
  }
}

// Forward substitution x <- T^-1 x of a 64-vector held by a warp (lane: elements lane and
// lane + 32), T unit-stride columns Tt[j][i] = T_ij; right-looking, so that every element takes
// its subtractions in the order of j and only a quotient and one step are ever waited for.
__device__ __forceinline__ void warp_subst(const double (*Tt)[CH_NB + 1], const double* rd, double& x0, double& x1) {
  const int lane = threadIdx.x % 32;
#pragma unroll 4
  for (int j = 0; j < CH_NB; ++j) {
    const double x = quotient(__shfl_sync(0xffffffffu, j < 32 ? x0 : x1, j & 31), Tt[j][j], rd[j]);
    if (lane > j) x0 -= x * Tt[j][lane];
    if (lane + 32 > j) x1 -= x * Tt[j][lane + 32];
    if (lane == j) x0 = x;
    if (lane + 32 == j) x1 = x;
  }
}

// L21 = A21 L11^-T for the rows below a full diagonal block: a warp per row.  (One thread per row
// waited for FP64 results: 218 us per panel from memory, 185 from registers; 34 so.)
__global__ void __launch_bounds__(128) trsm_panel_kernel(int n, double* G, int k0) {
  __shared__ double Lt[CH_NB][CH_NB + 1], rd[CH_NB];
  for (int e = threadIdx.x; e < CH_NB * CH_NB; e += 128) {
    const int i = e / CH_NB, j = e % CH_NB;
    if (j <= i) {
      const double v = G[(long long)(k0 + i) * n + k0 + j];
      Lt[j][i] = v;
      if (i == j) rd[i] = 1.0 / v;
    }
  }
  __syncthreads();
  const int r = k0 + CH_NB + blockIdx.x * 4 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (r >= n) return;
  double* row = G + (long long)r * n + k0;
  double x0 = row[lane], x1 = row[lane + 32];
  warp_subst(Lt, rd, x0, x1);
  row[lane] = x0;
  row[lane + 32] = x1;
}

__global__ void zero_upper_kernel(int n, double* G) {
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)n * n) return;
  int i = (int)(idx / n), j = (int)(idx % n);
  if (j > i) G[idx] = 0.0;
}

// Solve L X = R in place for rows [i0, i0+nbk) of R (one thread per column):
// X_m = (R_m - sum_{j<m} L_{m j} X_j) / L_{m m} with the diagonal block of L
// staged in shared memory.
// One thread per column, the column in registers, right-looking as the panels.  Past nbk the
// block is padded with a unit diagonal.
__global__ void __launch_bounds__(64) trsm_rows_kernel(int nx, const double* L, double* R, long long ncol, int i0, int nbk) {
  __shared__ double Lt[CH_NB][CH_NB + 1];  // Lt[j][i] = L[i][j]
  for (int e = threadIdx.x; e < CH_NB * CH_NB; e += blockDim.x) {
    const int i = e / CH_NB, j = e % CH_NB;
    if (j <= i) Lt[j][i] = i < nbk ? L[(long long)(i0 + i) * nx + i0 + j] : i == j ? 1.0 : 0.0;
  }
  __syncthreads();
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= ncol) return;
  double* col = R + (long long)i0 * ncol + c;
  double x[CH_NB];
#pragma unroll
  for (int m = 0; m < CH_NB; ++m) x[m] = m < nbk ? col[(long long)m * ncol] : 0.0;
#pragma unroll
  for (int j = 0; j < CH_NB; ++j) {
    x[j] = x[j] / Lt[j][j];
#pragma unroll
    for (int m = j + 1; m < CH_NB; ++m) x[m] -= Lt[j][m] * x[j];
  }
#pragma unroll
  for (int m = 0; m < CH_NB; ++m)
    if (m < nbk) col[(long long)m * ncol] = x[m];
}

// The same with a warp per column, for the few columns of a square right-hand side (240 columns
// leave three warps per SM waiting: 217 us a call before, 33 so).
__global__ void __launch_bounds__(128) trsm_cols_kernel(int nx, const double* L, double* R, int ncol, int i0, int nbk) {
  __shared__ double Lt[CH_NB][CH_NB + 1], rd[CH_NB];
  for (int e = threadIdx.x; e < CH_NB * CH_NB; e += 128) {
    const int i = e / CH_NB, j = e % CH_NB;
    if (j <= i) {
      const double v = i < nbk ? L[(long long)(i0 + i) * nx + i0 + j] : i == j ? 1.0 : 0.0;
      Lt[j][i] = v;
      if (i == j) rd[i] = 1.0 / v;
    }
  }
  __syncthreads();
  const int c = blockIdx.x * 4 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (c >= ncol) return;
  double* col = R + (long long)i0 * ncol + c;
  double x0 = lane < nbk ? col[(long long)lane * ncol] : 0.0;
  double x1 = lane + 32 < nbk ? col[(long long)(lane + 32) * ncol] : 0.0;
  warp_subst(Lt, rd, x0, x1);
  if (lane < nbk) col[(long long)lane * ncol] = x0;
  if (lane + 32 < nbk) col[(long long)(lane + 32) * ncol] = x1;
}

// A = L L^T in place for a symmetric positive definite n x n A (row-major; lower
// factor, upper triangle zeroed).  maxdiag: one device double of scratch.  A pivot
// below rel_min * max A_kk sets DEV_METRIC_NOT_PD in the context's status word.
int cholesky_lower(donof_ri_ctx* ctx, double* A, int n, double* maxdiag, double rel_min) {
  max_diag_kernel<<<1, 256, 0, ctx->stream>>>(n, A, maxdiag);
  DONOF_LAUNCH_CHECK(ctx);
  for (int k0 = 0; k0 < n; k0 += CH_NB) {
    int nbk = n - k0 < CH_NB ? n - k0 : CH_NB;
    potrf_block_kernel<<<1, 1024, 0, ctx->stream>>>(n, A, k0, nbk, maxdiag, rel_min, ctx->d_status);
    DONOF_LAUNCH_CHECK(ctx);
    int rows = n - k0 - nbk;
    if (rows <= 0) break;
    trsm_panel_kernel<<<ceil_div_u(rows, 4), 128, 0, ctx->stream>>>(n, A, k0);  // rows are left: nbk = CH_NB
    DONOF_LAUNCH_CHECK(ctx);
    Gemm64 g{};
    g.M = rows; g.N = rows; g.K = nbk; g.batch = 1;
    g.A = A + (long long)(k0 + nbk) * n + k0; g.sAm = n; g.sAk = 1;
    g.B = A + (long long)(k0 + nbk) * n + k0; g.sBk = 1; g.sBn = n;
    g.C = A + (long long)(k0 + nbk) * n + (k0 + nbk); g.sCm = n; g.sCn = 1;
    g.alpha = -1.0; g.beta = 1.0;
    g.lower = 1;
    int rc = launch_dgemm(ctx, g);
    if (rc) return rc;
  }
  zero_upper_kernel<<<ceil_div_u((long long)n * n, 256), 256, 0, ctx->stream>>>(n, A);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

// R <- L^-1 R for a lower-triangular n x n L (row-major, zero upper triangle) and an
// n x ncol row-major R: forward substitution over row blocks of R.
int forward_subst(donof_ri_ctx* ctx, const double* L, int n, double* R, long long ncol) {
  for (int i0 = 0; i0 < n; i0 += CH_NB) {
    int nbk = n - i0 < CH_NB ? n - i0 : CH_NB;
    if (i0 > 0) {
      // N can exceed the grid limit in x only for ncol > 4e9; never for supported sizes.
      Gemm64 g{};
      g.M = nbk; g.N = (int)ncol; g.K = i0; g.batch = 1;
      g.A = L + (long long)i0 * n; g.sAm = n; g.sAk = 1;
      g.B = R; g.sBk = ncol; g.sBn = 1;
      g.C = R + (long long)i0 * ncol; g.sCm = ncol; g.sCn = 1;
      g.alpha = -1.0; g.beta = 1.0;
      int rc = launch_dgemm(ctx, g);
      if (rc) return rc;
    }
    if (ncol <= 4096)
      trsm_cols_kernel<<<ceil_div_u(ncol, 4), 128, 0, ctx->stream>>>(n, L, R, (int)ncol, i0, nbk);
    else
      trsm_rows_kernel<<<ceil_div_u(ncol, 64), 64, 0, ctx->stream>>>(n, L, R, ncol, i0, nbk);
    DONOF_LAUNCH_CHECK(ctx);
  }
  return DONOF_RI_OK;
}

int setup_cholesky_and_fit(donof_ri_ctx* ctx) {
  int rc = cholesky_lower(ctx, ctx->d_G, ctx->naux, ctx->d_scratch_max, 1e-14);
  if (rc) return rc;
  return fit_forward(ctx);
}

void max_diag_public(donof_ri_ctx* ctx, const double* G, double* out) {
  max_diag_kernel<<<1, 256, 0, ctx->stream>>>(ctx->naux, G, out);
  ctx->launches++;
}

// ---------------------------------------------------------------------------
// The fit B <- L^-1 B on the tensor cores (launch_xgemm), over the pairs mu <= nu only.
//
// Right-looking in blocks of 128 auxiliary functions: X_j = D^-1 R_j for the diagonal block
// D, then R_i -= L_ij X_j below it.  The inverse of D alone would lose cond(D) roundings (X
// 50 times further off than by substitution for the even-tempered sets); one step of
// refinement, X = X0 + D^-1 (R_j - D X0) with the residual formed before it is rounded,
// makes it better than FP64 substitution (2e-14 against 4e-14 at 72 functions, cond(G) 5e6).
//
// With s4_congruence, of a SLICE4 context's set-up at 240 orbital and 840 auxiliary
// functions: 146 -> 15 ms with the integrals and the factorisation above.
//
// Columns are the 16 x 16 tiles I <= J of (mu, nu), in chunks of about 32768, so that the
// workspace stays at a few hundred MB and both triangles are written in full sectors.
// ---------------------------------------------------------------------------
constexpr int FIT_NB = 128;
constexpr long long FIT_CHUNK = 32768;

// The diagonal blocks' inverses: four CTAs per block, each every fourth column, four lanes
// per column (FP64 bound again: one CTA per block took 430 us).  L lies in the lower triangle
// of fs and X^T in the upper one; the diagonal keeps L_mm.
__global__ void __launch_bounds__(FIT_NB) fit_inverse_kernel(int nx, const double* __restrict__ L,
                                                             double* __restrict__ inv) {
  extern __shared__ double fs[];
  constexpr int LD = FIT_NB + 1;
  const int i0 = blockIdx.x * FIT_NB, n = min(FIT_NB, nx - i0), u = threadIdx.x % 4;
  const int c = blockIdx.y + 4 * (threadIdx.x / 4), warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int i = warp; i < n; i += 4)
    for (int j = lane; j <= i; j += 32) fs[i * LD + j] = L[(size_t)(i0 + i) * nx + i0 + j];
  __syncthreads();
  double* out = inv + (size_t)blockIdx.x * FIT_NB * FIT_NB;
  const bool on = c < n;
  double* x = fs + (on ? c : 0) * LD;  // x[j], j > c: X_jc
  const double xc = on ? 1.0 / x[c] : 0.0;
  if (on) {
    for (int m = u; m < c; m += 4) out[m * n + c] = 0.0;
    if (u == 0) out[c * n + c] = xc;
  }
  for (int m = 1; m < n; ++m) {  // every lane takes part in the shuffles
    const double* l = fs + m * LD;
    const bool act = on && m > c;
    double a0 = 0.0, a1 = 0.0;
    if (act) {
      if (u == 0) a0 = l[c] * xc;
      int j = c + 1 + u;
      for (; j + 4 < m; j += 8) {
        a0 = fma(l[j], x[j], a0);
        a1 = fma(l[j + 4], x[j + 4], a1);
      }
      if (j < m) a0 = fma(l[j], x[j], a0);
    }
    a0 += a1;
    a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
    a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
    if (act && u == 0) {
      const double v = -a0 / l[m];
      x[m] = v;
      out[m * n + c] = v;
    }
    __syncwarp();
  }
}

// W[k][c] = B[k][mu][nu] for the columns of tiles t0, t0 + 1, ...: a block per tile and k.
__global__ void __launch_bounds__(256) fit_gather_kernel(const double* __restrict__ B, int nbf, int t0, long long cw,
                                                         double* __restrict__ W) {
  int I, J;
  pair_tile(t0 + blockIdx.x, I, J);
  const int mu = I * PAIR_T + threadIdx.x / PAIR_T, nu = J * PAIR_T + threadIdx.x % PAIR_T;
  W[blockIdx.y * cw + blockIdx.x * 256 + threadIdx.x] =
      mu < nbf && nu < nbf ? B[((size_t)blockIdx.y * nbf + mu) * nbf + nu] : 0.0;
}

__global__ void __launch_bounds__(256) fit_scatter_kernel(const double* __restrict__ W, int nbf, int t0, long long cw,
                                                          double* __restrict__ B) {
  __shared__ double s[PAIR_T][PAIR_T + 1];
  int I, J;
  pair_tile(t0 + blockIdx.x, I, J);
  const int a = threadIdx.x / PAIR_T, b = threadIdx.x % PAIR_T;
  double* Bk = B + (size_t)blockIdx.y * nbf * nbf;
  const double v = W[blockIdx.y * cw + blockIdx.x * 256 + threadIdx.x];
  s[a][b] = v;
  __syncthreads();
  if (I * PAIR_T + a < nbf && J * PAIR_T + b < nbf) Bk[(size_t)(I * PAIR_T + a) * nbf + J * PAIR_T + b] = v;
  if (I != J && J * PAIR_T + a < nbf && I * PAIR_T + b < nbf) Bk[(size_t)(J * PAIR_T + a) * nbf + I * PAIR_T + b] = s[b][a];
}

// C = alpha A B + beta C for a row-major A (ld_a) and chunk rows B, C (ld cw)
static int fit_gemm(donof_ri_ctx* ctx, int M, int K, const double* A, long long lda, const double* B, double* C,
                    long long cw, double alpha, double beta, void* ws) {
  Gemm64 g{};
  g.M = M; g.N = (int)cw; g.K = K; g.batch = 1;
  g.A = A; g.sAm = lda; g.sAk = 1;
  g.B = B; g.sBk = cw; g.sBn = 1;
  g.C = C; g.sCm = cw; g.sCn = 1;
  g.alpha = alpha; g.beta = beta;
  return launch_xgemm(ctx, g, ws, 0);
}

static int fit_forward_tc(donof_ri_ctx* ctx, double* inv, double* W, double* X, void* ws, long long cw, int ntiles) {
  const int nb = ctx->nbf, nx = ctx->naux;
  const double* L = ctx->d_G;
  const int smem = FIT_NB * (FIT_NB + 1) * (int)sizeof(double);
  DONOF_CUDA_TRY(cudaFuncSetAttribute(fit_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  fit_inverse_kernel<<<dim3((nx + FIT_NB - 1) / FIT_NB, 4), FIT_NB, smem, ctx->stream>>>(nx, L, inv);
  DONOF_LAUNCH_CHECK(ctx);
  int rc;
  for (int t0 = 0; t0 < ntiles; t0 += (int)(cw / 256)) {
    const int nt = ntiles - t0 < cw / 256 ? ntiles - t0 : (int)(cw / 256);
    const long long w = nt * 256LL;
    fit_gather_kernel<<<dim3(nt, nx), 256, 0, ctx->stream>>>(ctx->d_B, nb, t0, w, W);
    DONOF_LAUNCH_CHECK(ctx);
    for (int i0 = 0; i0 < nx; i0 += FIT_NB) {
      const int n = nx - i0 < FIT_NB ? nx - i0 : FIT_NB, rows = nx - i0 - n;
      const double *D = L + (size_t)i0 * nx + i0, *Di = inv + (size_t)i0 * FIT_NB;
      double* R = W + (size_t)i0 * w;
      if ((rc = fit_gemm(ctx, n, n, Di, n, R, X, w, 1.0, 0.0, ws))) return rc;    // X = D^-1 R
      if ((rc = fit_gemm(ctx, n, n, D, nx, X, R, w, -1.0, 1.0, ws))) return rc;   // R -= D X
      if ((rc = fit_gemm(ctx, n, n, Di, n, R, X, w, 1.0, 1.0, ws))) return rc;    // X += D^-1 R
      DONOF_CUDA_TRY(cudaMemcpyAsync(R, X, (size_t)n * w * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream));
      if (rows > 0 &&
          (rc = fit_gemm(ctx, rows, n, D + (size_t)n * nx, nx, X, R + (size_t)n * w, w, -1.0, 1.0, ws)))
        return rc;
    }
    fit_scatter_kernel<<<dim3(nt, nx), 256, 0, ctx->stream>>>(W, nb, t0, w, ctx->d_B);
    DONOF_LAUNCH_CHECK(ctx);
  }
  return DONOF_RI_OK;
}

// B <- L^-1 B for the lower-triangular L in ctx->d_G (row-major, zero upper triangle):
// forward substitution over row blocks of B.  B is symmetric in (mu, nu).  By the tensor
// cores from 256 auxiliary and 64 orbital functions on, where the products fill the chip, in
// narrower chunks of columns (the same bits) where there is no room for the wide ones.  Set-up
// at 96 orbital functions with 255 / 256 auxiliary ones (integrals too): FP64 4.9 / 2.4 ms, SLICE4
// 6.3 / 3.7.
int fit_forward(donof_ri_ctx* ctx) {
  const int nb = ctx->nbf, nx = ctx->naux;
  if (nx >= 256 && nb >= 64 && nx <= 65535 && ctx->precision != DONOF_RI_TF32X3) {
    const int T = (nb + PAIR_T - 1) / PAIR_T, ntiles = T * (T + 1) / 2;
    const size_t inv = (size_t)((nx + FIT_NB - 1) / FIT_NB) * FIT_NB * FIT_NB * sizeof(double);
    for (long long chunks = (ntiles * 256LL + FIT_CHUNK - 1) / FIT_CHUNK;; chunks *= 2) {
      const long long cw = (ntiles + chunks - 1) / chunks * 256LL;
      const size_t digits = xgemm_operand_bytes((int)cw, FIT_NB, 1) + xgemm_operand_bytes(nx, FIT_NB, 1);
      const size_t bytes = inv + (size_t)(nx + FIT_NB) * cw * sizeof(double) + digits;
      char* ws;
      const int rc = xgemm_workspace(ctx, bytes, bytes, (void**)&ws);
      if (rc == DONOF_RI_E_OOM && cw > 256) continue;
      if (rc) return rc;
      double* W = (double*)(ws + inv);
      double* X = W + (size_t)nx * cw;
      return fit_forward_tc(ctx, (double*)ws, W, X, X + FIT_NB * cw, cw, ntiles);
    }
  }
  return forward_subst(ctx, ctx->d_G, nx, ctx->d_B, (long long)nb * nb);
}

}  // namespace donof
