// Orbital rotation step for fixed occupations (Sec. 2, "Orbital Optimization with
// RI"): C -> C expm(kappa) with kappa = -r G / max|G|, G_qp = lambda_qp - lambda_pq
// the rotation gradient (dE/dkappa_qp = 4 G_qp) from the Lagrangian of the last
// donof_ri_energy_lagrangian, and r a trust radius chosen by the caller.  This is
// the plain rotation driver's step; the paper's own step (iterative
// diagonalisation of F^lambda) is a later addition.
//
// expm by scaling and squaring: X = kappa / 2^s with s the smallest for which the bound
// ||X^13||_1 / 13! <= 1e-18 holds, from the 1-norms of kappa, kappa^2 and kappa^4 (their
// products bound ||kappa^13||; the norm of kappa alone overestimates the powers of an
// antisymmetric matrix by up to sqrt(n) each, which costs squarings); Taylor polynomial of
// degree 12 in X, ..., X^4 by Paterson and Stockmeyer's scheme (five products), then s
// squarings; the rotated orbitals are re-orthonormalised in the overlap metric by one
// Newton-Schulz step C <- C (3 I - C^T S C) / 2, which removes the rounding drift
// of repeated steps (the orbitals are orthonormal functions, C^T S C = I; a
// rotation in orbital space keeps that exactly, so the step only corrects
// rounding and expects orbitals that are S-orthonormal on entry).
// All FP64: the products by launch_xgemm (tensor cores, FP64 accuracy) from 96 functions
// on, by the tiled DGEMM below.  At 720 functions: Horner's 11 products, squarings until the
// 1-norm was below 1/4, and one block for the norms took 18.4 ms; now 1.47 ms with the copies
// of kappa and C (8 MB) from and to the host.
#include "common.cuh"

#include <math.h>

namespace donof {

// kappa[q][p] (row-major) = scale (lambda_qp - lambda_pq); lambda column-major.
__global__ void rot_kappa_kernel(const double* lam, int nb, double scale, double* kappa) {
  __shared__ double t[32][33];
  const int p0 = blockIdx.x * 32, q0 = blockIdx.y * 32;
  // lambda_pq = lam[q nb + p]: read along p; lambda_qp = lam[p nb + q]: through the tile
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int p = p0 + i, q = q0 + threadIdx.x;
    t[i][threadIdx.x] = p < nb && q < nb ? lam[(size_t)p * nb + q] : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int q = q0 + i, p = p0 + threadIdx.x;
    if (p < nb && q < nb) kappa[(size_t)q * nb + p] = scale * (t[threadIdx.x][i] - lam[(size_t)q * nb + p]);
  }
}

// out[0] <- max(out[0], 1-norm of X) (max over columns of the sums of |X|), and with out + 1
// the same for the largest |X|, NaN left out of it; the patterns of non-negative doubles
// order like integers (NaN above everything).  32 columns per block.
__global__ void __launch_bounds__(256) rot_norms_kernel(const double* __restrict__ X, int n, unsigned long long* sum,
                                                        unsigned long long* mx) {
  __shared__ double rs[8][32], rm[8][32];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32, c = blockIdx.x * 32 + tx;
  double s = 0.0, m = 0.0;
  if (c < n) {
#pragma unroll 8
    for (int r = ty; r < n; r += 8) {
      const double a = fabs(X[(size_t)r * n + c]);
      s += a;
      m = fmax(m, a);
    }
  }
  rs[ty][tx] = s;
  rm[ty][tx] = m;
  __syncthreads();
  if (ty == 0 && c < n) {
    for (int y = 1; y < 8; ++y) {
      s += rs[y][tx];
      m = fmax(m, rm[y][tx]);
    }
    atomicMax(sum, (unsigned long long)__double_as_longlong(s));
    if (mx) atomicMax(mx, (unsigned long long)__double_as_longlong(m));
  }
}

// out = a[0] I + a[1] X + a[2] X2 + a[3] X3 + a[4] X4 (row-major n x n; a null matrix counts as zero)
struct RotPoly {
  double a[5];
};
__global__ void rot_poly_kernel(int n, RotPoly c, const double* X, const double* X2, const double* X3, const double* X4,
                                double* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)n * n) return;
  double v = (i / n == i % n) ? c.a[0] : 0.0;
  if (X) v = fma(c.a[1], X[i], v);
  if (X2) v = fma(c.a[2], X2[i], v);
  if (X3) v = fma(c.a[3], X3[i], v);
  if (X4) v = fma(c.a[4], X4[i], v);
  out[i] = v;
}

size_t rotation_scratch_doubles(int n) { return 6 * (size_t)n * n + 4; }

static int rot_gemm(donof_ri_ctx* ctx, const Gemm64& g) {
  if (!xgemm_takes(g)) return launch_dgemm(ctx, g);
  void* ws;
  const size_t a = xgemm_operand_bytes(g.M, g.K, 1), b = xgemm_operand_bytes(g.N, g.K, 1);
  const int rc = xgemm_workspace(ctx, a + b, a + xgemm_operand_bytes(128, g.K, 1), &ws);
  return rc ? rc : launch_gemm64(ctx, g, ws, ctx->xws_bytes, 0);
}

static int gemm_rr(donof_ri_ctx* ctx, int n, const double* A, bool At, const double* B, double* C, double alpha,
                   double beta) {
  // C = alpha op(A) B + beta C, all row-major n x n; op(A) = A or A^T
  Gemm64 g{};
  g.M = n; g.N = n; g.K = n; g.batch = 1;
  g.A = A;
  g.sAm = At ? 1 : n;
  g.sAk = At ? n : 1;
  g.B = B; g.sBk = n; g.sBn = 1;
  g.C = C; g.sCm = n; g.sCn = 1;
  g.alpha = alpha; g.beta = beta;
  return rot_gemm(ctx, g);
}

// C <- C expm(K) for K (row-major kappa, the first n^2 of the scratch), then one
// Newton-Schulz step in the overlap metric.  must_be_finite: refuse a K that is not.
static int rotate_by(donof_ri_ctx* ctx, double* scratch, bool must_be_finite) {
  const int n = ctx->nbf;
  const long long n2 = (long long)n * n;
  double *K = scratch, *X2 = K + n2, *X3 = X2 + n2, *X4 = X3 + n2, *U = X4 + n2, *T = U + n2;
  unsigned long long* nrm = (unsigned long long*)(scratch + 6 * n2);
  const unsigned int nblk = ceil_div_u(n2, 256), cblk = ceil_div_u(n, 32);
  int rc;
  if ((rc = gemm_rr(ctx, n, K, false, K, X2, 1.0, 0.0))) return rc;
  if ((rc = gemm_rr(ctx, n, X2, false, X2, X4, 1.0, 0.0))) return rc;
  DONOF_CUDA_TRY(cudaMemsetAsync(nrm, 0, 3 * sizeof(double), ctx->stream));
  const double* mats[3] = {K, X2, X4};
  for (int i = 0; i < 3; ++i) {
    rot_norms_kernel<<<cblk, 256, 0, ctx->stream>>>(mats[i], n, nrm + i, nullptr);
    DONOF_LAUNCH_CHECK(ctx);
  }
  double h[3];
  DONOF_CUDA_TRY(cudaMemcpyAsync(h, nrm, 3 * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
  if ((rc = gemm_rr(ctx, n, X2, false, K, X3, 1.0, 0.0))) return rc;
  DONOF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  if (must_be_finite && !isfinite(h[0])) return DONOF_RI_E_NONFINITE;
  int s = 0;
  for (; s < 60; ++s) {
    const double a1 = ldexp(h[0], -s), a2 = ldexp(h[1], -2 * s), a4 = ldexp(h[2], -4 * s);
    const double b = fmin(fmin(a4 * a4 * a4, pow(a2, 6.0)) * a1, pow(a1, 13.0));
    if (!(a1 > 4.0) && !(b / 6227020800.0 > 1e-18)) break;
  }
  // Taylor coefficients c_k 2^(-s k) of kappa^k, k = 0..12
  double c[13], f = 1.0;
  for (int k = 0; k <= 12; ++k) {
    if (k) f /= k;
    c[k] = ldexp(f, -s * k);
  }
  // U = ((c12 X4 + c11 X3 + ... + c8) X4 + c7 X3 + ... + c4) X4 + c3 X3 + ... + c0, with the
  // powers of two of c8.. and c4.. taken out of the bracket (c_k / 2^(-4 s) and so on)
  const double up4 = ldexp(1.0, 4 * s), up8 = ldexp(1.0, 8 * s);
  rot_poly_kernel<<<nblk, 256, 0, ctx->stream>>>(n, RotPoly{{c[8] * up8, c[9] * up8, c[10] * up8, c[11] * up8, c[12] * up8}},
                                                K, X2, X3, X4, U);
  DONOF_LAUNCH_CHECK(ctx);
  rot_poly_kernel<<<nblk, 256, 0, ctx->stream>>>(n, RotPoly{{c[4] * up4, c[5] * up4, c[6] * up4, c[7] * up4, 0.0}}, K, X2,
                                                X3, nullptr, T);
  DONOF_LAUNCH_CHECK(ctx);
  if ((rc = gemm_rr(ctx, n, U, false, X4, T, ldexp(1.0, -4 * s), 1.0))) return rc;
  rot_poly_kernel<<<nblk, 256, 0, ctx->stream>>>(n, RotPoly{{c[0], c[1], c[2], c[3], 0.0}}, K, X2, X3, nullptr, U);
  DONOF_LAUNCH_CHECK(ctx);
  if ((rc = gemm_rr(ctx, n, T, false, X4, U, ldexp(1.0, -4 * s), 1.0))) return rc;
  for (int k = 0; k < s; ++k) {  // U <- U U
    if ((rc = gemm_rr(ctx, n, U, false, U, T, 1.0, 0.0))) return rc;
    double* t = U;
    U = T;
    T = t;
  }
  // d_C is column-major, i.e. row-major C^T: (C U)^T = U^T C^T
  if ((rc = gemm_rr(ctx, n, U, true, ctx->d_C, T, 1.0, 0.0))) return rc;
  // Newton-Schulz in the overlap metric: C <- C (3 I - C^T S C) / 2.  With Ct = C^T
  // (row-major, in T): X = S C = S Ct^T (into K, free after the exponential), then
  // W = Ct X = C^T S C; Ct <- Z Ct with Z = (3 I - W) / 2 (symmetric).
  {
    Gemm64 g{};
    g.M = n; g.N = n; g.K = n; g.batch = 1;
    g.A = ctx->d_S; g.sAm = n; g.sAk = 1;
    g.B = T; g.sBk = 1; g.sBn = n;
    g.C = K; g.sCm = n; g.sCn = 1;
    g.alpha = 1.0; g.beta = 0.0;
    if ((rc = rot_gemm(ctx, g))) return rc;  // K = S C
    if ((rc = gemm_rr(ctx, n, T, false, K, X2, 1.0, 0.0))) return rc;  // X2 = C^T S C
  }
  rot_poly_kernel<<<nblk, 256, 0, ctx->stream>>>(n, RotPoly{{1.5, -0.5, 0.0, 0.0, 0.0}}, X2, nullptr, nullptr, nullptr,
                                                U);  // Z = (3 I - W) / 2
  DONOF_LAUNCH_CHECK(ctx);
  return gemm_rr(ctx, n, U, false, T, ctx->d_C, 1.0, 0.0);
}

// Rotates ctx->d_C in place; gnorm[0] = max|G| (host).  Scratch: rotation_scratch_doubles.
int rotate_orbitals(donof_ri_ctx* ctx, double radius, double* scratch, double* gnorm) {
  const int n = ctx->nbf;
  const long long n2 = (long long)n * n;
  unsigned long long* nrm = (unsigned long long*)(scratch + 6 * n2);
  const dim3 kb(ceil_div_u(n, 32), ceil_div_u(n, 32));
  // G in place of kappa, for its largest element
  rot_kappa_kernel<<<kb, dim3(32, 8), 0, ctx->stream>>>(ctx->d_lambda, n, 1.0, scratch);
  DONOF_LAUNCH_CHECK(ctx);
  DONOF_CUDA_TRY(cudaMemsetAsync(nrm, 0, 2 * sizeof(double), ctx->stream));
  rot_norms_kernel<<<ceil_div_u(n, 32), 256, 0, ctx->stream>>>(scratch, n, nrm, nrm + 1);
  DONOF_LAUNCH_CHECK(ctx);
  double g = 0.0;
  DONOF_CUDA_TRY(cudaMemcpyAsync(&g, nrm + 1, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
  DONOF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  *gnorm = g;
  if (!(g > 0.0) || !(radius > 0.0)) return DONOF_RI_OK;
  rot_kappa_kernel<<<kb, dim3(32, 8), 0, ctx->stream>>>(ctx->d_lambda, n, -radius / g, scratch);
  DONOF_LAUNCH_CHECK(ctx);
  return rotate_by(ctx, scratch, false);
}

// Rotates ctx->d_C in place by expm(kappa), kappa a device copy (row-major n x n) in the
// scratch's first n^2 doubles.
int apply_rotation(donof_ri_ctx* ctx, double* scratch) { return rotate_by(ctx, scratch, true); }

}  // namespace donof
