// Occupation optimisation for fixed orbitals (Sec. 2, "Occupancy Optimization
// with RI"): J_pq and K_pq of the current orbitals stay fixed while the PNOF7
// energy, Eq. (PNOF), is minimised over the unconstrained angles gamma that
// parametrise the occupations.  The paper names neither the optimiser nor the
// gradient.  Here the gradient is the chain rule
//   dE/dgamma_k = sum_p dE/dn_p dn_p/dgamma_k,
//   dE/dn_p = 2 H_pp + J_pp - sum_{q in g(p), q != p} s_pq K_pq sqrt(n_q / n_p)
//             + sum_{q not in g(p)} (4 n_q J_pq - 2 n_q K_pq - 2 Phi'_p Phi_q K_pq),
// (s_pq = +1 when p or q is the subspace's strong orbital, -1 when both are
// weak; Phi = sqrt(n (1 - n)), Phi' = (1 - 2n)/(2 Phi)), and the minimiser is
// L-BFGS (8 pairs of history, backtracking Armijo line search), all in FP64.
//
// The problem is small (N_Omega^2 terms per evaluation) but FP64, which this part issues
// at two lanes a clock per SM, so the evaluation runs on as many SMs as there are
// pairing subspaces (one cooperative launch per outer iteration, no host round trips):
// the CTA of subspace g takes the trigonometry and the occupations of its orbitals, their
// rows of J and K (read along q, coalesced), and the gradient of its angles; two grid
// barriers per evaluation exchange the occupations and then the row energies and the
// gradient.  The L-BFGS vectors are kept and updated by every CTA alike, so every CTA
// takes the same decisions.  Row sums are added in q order and all other sums in fixed
// trees, so the result does not depend on the number of CTAs.
// Twenty iterations at N_Omega = 400: 27.0 ms in one CTA (one thread per row, uncoalesced,
// the sines of an angle recomputed up to N_g^2 times) -> 1.9 ms; at 60 orbitals 3.7 -> 1.0.
// Every loop and every wait has a fixed bound; __syncthreads() is only reached in uniform
// control flow (loop decisions are read from shared memory after a barrier).
#include "common.cuh"

namespace donof {

constexpr int ON_THREADS = 512;
constexpr int ON_HIST = 8;
constexpr int ON_MAX_WEAK = 16;

struct OnParams {
  int n_strong, n_weak_per, m, ng;
  const int* subspace;
  const int* weak_rank;
  const double* J;
  const double* K;
  const double* Hd;
  const double* enuc;
  double* gamma;     // in: start, out: result
  double* E_out;     // [1]
  double* grad_out;  // [ng]
  int* info_out;     // [2]: iterations, stop reason (0 gradient below gtol, 1 iteration cap,
                     //      2 line search found no decrease, 3 relative energy decrease below etol)
  int max_iter;
  double gtol, etol;
  int mode;  // 0: evaluate E and the gradient at gamma; 1: optimise
  int chunk;       // orbitals q per step of the row sums
  int nown;        // subspaces of a CTA at most
  double* xch;     // exchanged between CTAs: n, phi, dphi, row energies [m] each, gradient [ng]
  unsigned int* bar;  // [2]: arrivals at the grid barrier, abort flag (zero at launch)
  int* status;
};

// H_pp = C_p^T (H C)_p for the pairing-space orbitals: one warp per p.
__global__ void on_hdiag_kernel(int nb, int m, const double* C, const double* HC, double* Hd) {
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x % 32;
  if (w >= m) return;
  double s = 0.0;
  for (int mu = lane; mu < nb; mu += 32) s = fma(C[(size_t)w * nb + mu], HC[(size_t)mu * m + w], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) Hd[w] = s;
}

struct OnShared {
  double *n, *phi, *dphi, *red, *red2;
  double *x, *g, *xn, *gn, *d, *S, *Y, *rho, *al;
  double* trig;              // per subspace of the CTA: cos x, sin 2x of the strong angle; sin, cos, sin 2w of the weak ones
  double* dE;                // [N_g + 1] dE/dn of the rows in hand
  double *sk, *sv, *se;      // [N_g + 1][N_g + 1] pairs within the subspace: s K_pq, sqrt(n_q / n_p), sqrt(n_p n_q)
  double *tv, *te;           // [2][N_g + 1][chunk] terms of the other orbitals q
  int* mk;                   // [2][chunk] member index of q in the subspace in hand, or -1
  unsigned int* mb;          // [2][2] the same as bits: members among the 64 orbitals of a chunk
  int* orb;  // orb[g * (N_g + 1) + r + 1] = orbital of rank r (-1 strong) in subspace g
  unsigned int* epoch;
};

// Barrier over the grid's CTAs (a cooperative launch, so all are resident), with a time
// limit: false, for every thread, once a CTA has waited for two seconds.
__device__ bool on_grid_sync(const OnParams& p, const OnShared& sh) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int target = (*sh.epoch += gridDim.x);
    __threadfence();
    atomicAdd(p.bar, 1u);
    ok = 1;
    unsigned long long t0 = 0;
    while ((int)(*(volatile unsigned int*)p.bar - target) < 0) {
      unsigned long long now;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (!t0) t0 = now;
      if (*(volatile unsigned int*)(p.bar + 1) || now - t0 > 2000000000ull) {
        atomicExch(p.bar + 1, 1u);
        atomicCAS(p.status, 0, (int)DEV_TIMEOUT);
        ok = 0;
        break;
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// Block-wide sum of v over all threads: the tree of strides 256, 128, ..., 1 over the
// threads' values, the same additions in three barriers.
__device__ double on_block_sum(double v, const OnShared& sh) {
  const int t = threadIdx.x;
  sh.red[t] = v;
  __syncthreads();
  if (t < 128) sh.red2[t] = (sh.red[t] + sh.red[t + 256]) + (sh.red[t + 128] + sh.red[t + 384]);
  __syncthreads();
  if (t < 32) {
    double s = (sh.red2[t] + sh.red2[t + 64]) + (sh.red2[t + 32] + sh.red2[t + 96]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (t == 0) sh.red2[128] = s;
  }
  __syncthreads();
  return sh.red2[128];
}

__device__ double on_block_max(double v, const OnShared& sh) {
  const int t = threadIdx.x;
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (t % 32 == 0) sh.red[t / 32] = v;
  __syncthreads();
  if (t < 32) {
    double s = t < ON_THREADS / 32 ? sh.red[t] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
    if (t == 0) sh.red2[129] = s;
  }
  __syncthreads();
  return sh.red2[129];
}

__device__ double on_dot(const double* a, const double* b, int n, const OnShared& sh) {
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += ON_THREADS) s = fma(a[i], b[i], s);
  return on_block_sum(s, sh);
}

// alpha_i of a subspace with N_g weak orbitals, from the sines and cosines of its angles.
__device__ double on_alpha(const double* sw, const double* cw, int Ng, int i) {
  const double tail = i < Ng - 1 ? cw[i] * cw[i] : 1.0;
  double prod = 1.0;
  for (int k = 0; k < i; ++k) prod *= sw[k] * sw[k];
  return prod * tail;
}

// d alpha_i / d w_j.
__device__ double on_dalpha(const double* sw, const double* cw, const double* s2w, int Ng, int i, int j) {
  const double tail = i < Ng - 1 ? cw[i] * cw[i] : 1.0;
  double v = 0.0;
  if (j < i) {
    double others = 1.0;
    for (int k = 0; k < i; ++k)
      if (k != j) others *= sw[k] * sw[k];
    v = others * s2w[j] * tail;
  } else if (j == i) {
    double prod = 1.0;
    for (int k = 0; k < i; ++k) prod *= sw[k] * sw[k];
    v = -prod * s2w[i];
  }
  return v;
}

// E(x) and dE/dx into E and gout (every CTA gets all of them); false when a grid barrier
// gave up.
__device__ bool on_evaluate(const OnParams& p, const OnShared& sh, const double* x, double* gout, double* E) {
  const int NI = p.n_strong, Ng = p.n_weak_per, m = p.m, na = Ng - 1, M = Ng + 1;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  double *g_n = p.xch, *g_phi = g_n + m, *g_dphi = g_phi + m, *g_e = g_dphi + m, *g_grad = g_e + m;
  const int TR = 3 * Ng + 2;
  // occupations of the CTA's subspaces: a warp each, a lane per angle and per orbital
  for (int k = warp; (int)blockIdx.x + k * (int)gridDim.x < NI; k += ON_THREADS / 32) {
    const int g = blockIdx.x + k * gridDim.x;
    double* tr = sh.trig + (size_t)k * TR;
    double *sw = tr + 2, *cw = sw + Ng, *s2w = cw + Ng;
    if (lane < na) {
      const double w = x[NI + g * na + lane];
      sw[lane] = sin(w);
      cw[lane] = cos(w);
      s2w[lane] = sin(2.0 * w);
    }
    if (lane == 31) {
      tr[0] = cos(x[g]);
      tr[1] = sin(2.0 * x[g]);
    }
    __syncwarp();
    if (lane < M) {
      const double c = tr[0];
      const double ngv = 0.5 * (1.0 + c * c), hg = 1.0 - ngv;
      const double nq = lane == 0 ? ngv : hg * on_alpha(sw, cw, Ng, lane - 1);
      const double ph = sqrt(nq * (1.0 - nq));
      const int q = sh.orb[g * M + lane];
      g_n[q] = nq;
      g_phi[q] = ph;
      g_dphi[q] = ph > 0.0 ? (1.0 - 2.0 * nq) / (2.0 * ph) : 0.0;
    }
  }
  if (!on_grid_sync(p, sh)) return false;
  for (int q = threadIdx.x; q < m; q += ON_THREADS) {
    sh.n[q] = __ldcg(g_n + q);
    sh.phi[q] = __ldcg(g_phi + q);
    sh.dphi[q] = __ldcg(g_dphi + q);
  }
  __syncthreads();
  const int CH = p.chunk, nch = (m + CH - 1) / CH;
  for (int k = 0; (int)blockIdx.x + k * (int)gridDim.x < NI; ++k) {
    const int g = blockIdx.x + k * gridDim.x;
    const int* orb = sh.orb + g * M;
    // the pairs within the subspace
    for (int i = threadIdx.x; i < M * M; i += ON_THREADS) {
      const int r = i / M, o = i % M;
      const double s = (r == 0 || o == 0) ? 1.0 : -1.0;
      const double np_ = sh.n[orb[r]], nq = sh.n[orb[o]];
      sh.sk[i] = s * p.K[(size_t)orb[r] * m + orb[o]];
      sh.sv[i] = np_ > 0.0 ? sqrt(nq / np_) : 0.0;
      sh.se[i] = sqrt(np_ * nq);
    }
    // the other orbitals' terms of chunk c, into buffer c % 2
    auto terms = [&](int c, int t0, int nt) {
      const int q0 = c * CH, cn = m - q0 < CH ? m - q0 : CH;
      double *tv = sh.tv + (size_t)(c & 1) * M * CH, *te = sh.te + (size_t)(c & 1) * M * CH;
      int* mk = sh.mk + (c & 1) * CH;
      if (t0 < M) {  // the subspace's members in this chunk (a chunk has at most 64 orbitals)
        const int qi = orb[t0] - q0;
        if (qi >= 0 && qi < cn) {
          mk[qi] = t0;
          atomicOr(sh.mb + 2 * (c & 1) + qi / 32, 1u << (qi % 32));
        }
      }
      for (int i = t0; i < M * cn; i += nt) {
        const int r = i / cn, qi = i % cn, q = q0 + qi, pp = orb[r];
        if (p.subspace[q] != g) {
          const double np_ = sh.n[pp], php = sh.phi[pp], dphp = sh.dphi[pp];
          const double nq = sh.n[q], phq = sh.phi[q];
          const double j = p.J[(size_t)pp * m + q], kk = p.K[(size_t)pp * m + q];
          tv[r * CH + qi] = 4.0 * nq * j - 2.0 * nq * kk - 2.0 * dphp * phq * kk;
          te[r * CH + qi] = 2.0 * np_ * nq * j - (np_ * nq + php * phq) * kk;
        }
      }
    };
    terms(0, threadIdx.x, ON_THREADS);
    __syncthreads();
    // dE/dn_p (warp 0) and the row energies (warp 1), a lane per row, q in order; the other
    // warps prepare the next chunk's terms meanwhile
    double acc = 0.0, np_ = 0.0;
    if (warp < 2 && lane < M) {
      const int pp = orb[lane];
      np_ = sh.n[pp];
      acc = warp == 0 ? 2.0 * p.Hd[pp] + p.J[(size_t)pp * m + pp]
                      : 2.0 * np_ * p.Hd[pp] + np_ * p.J[(size_t)pp * m + pp];
    }
    for (int c = 0; c < nch; ++c) {
      if (warp < 2) {
        if (lane < M) {
          const int cn = m - c * CH < CH ? m - c * CH : CH;
          const double* tt = (warp == 0 ? sh.tv : sh.te) + ((size_t)(c & 1) * M + lane) * CH;
          const int* mk = sh.mk + (c & 1) * CH;
          unsigned long long left = (unsigned long long)sh.mb[2 * (c & 1) + 1] << 32 | sh.mb[2 * (c & 1)];
          for (int qi = 0; qi < cn;) {
            // the other orbitals up to the next member, whose loads run ahead of the sum
            const int end = left ? __ffsll((long long)left) - 1 : cn;
#pragma unroll 8
            for (; qi < end; ++qi) acc += tt[qi];
            if (qi == cn) break;
            left &= left - 1;
            const int o = mk[qi++];
            if (o != lane) {
              const int i = lane * M + o;
              if (warp == 0) {
                if (np_ > 0.0) acc = fma(-sh.sk[i], sh.sv[i], acc);
              } else {
                acc = fma(-sh.se[i], sh.sk[i], acc);
              }
            }
          }
        }
      } else if (c + 1 < nch) {
        terms(c + 1, threadIdx.x - 64, ON_THREADS - 64);
      }
      __syncthreads();
      if (threadIdx.x < 2) sh.mb[2 * (c & 1) + threadIdx.x] = 0;  // for chunk c + 2
      __syncthreads();
    }
    if (warp == 0 && lane < M) sh.dE[lane] = acc;
    if (warp == 1 && lane < M) __stcg(g_e + orb[lane], acc);
    __syncthreads();
    // chain rule: a lane per angle
    if (warp == 0) {
      const double* tr = sh.trig + (size_t)k * TR;
      const double *sw = tr + 2, *cw = sw + Ng, *s2w = cw + Ng;
      if (lane == 31) {
        const double dh = 0.5 * tr[1];
        double gs = -dh * sh.dE[0];
        for (int i = 0; i < Ng; ++i) gs += dh * on_alpha(sw, cw, Ng, i) * sh.dE[i + 1];
        __stcg(g_grad + g, gs);
      }
      if (lane < na) {
        const double c = tr[0];
        const double hg = 1.0 - 0.5 * (1.0 + c * c);
        double gw = 0.0;
        for (int i = 0; i < Ng; ++i) gw += hg * on_dalpha(sw, cw, s2w, Ng, i, lane) * sh.dE[i + 1];
        __stcg(g_grad + NI + g * na + lane, gw);
      }
    }
    __syncthreads();
  }
  if (!on_grid_sync(p, sh)) return false;
  double epart = 0.0;
  for (int pp = threadIdx.x; pp < m; pp += ON_THREADS) epart += __ldcg(g_e + pp);
  for (int i = threadIdx.x; i < p.ng; i += ON_THREADS) gout[i] = __ldcg(g_grad + i);
  *E = on_block_sum(epart, sh) + p.enuc[0];  // (the sum's barriers also publish gout)
  return true;
}

__global__ void __launch_bounds__(ON_THREADS, 1) on_opt_kernel(const OnParams p) {
  extern __shared__ double onsm[];
  __shared__ unsigned int epoch, members[4];
  const int m = p.m, ng = p.ng, Ng = p.n_weak_per, M = Ng + 1;
  OnShared sh;
  double* ptr = onsm;
  auto take = [&](size_t n) {
    double* r = ptr;
    ptr += n;
    return r;
  };
  sh.n = take(m);
  sh.phi = take(m);
  sh.dphi = take(m);
  // the pairs of a subspace are dead when the block sums run: they share their space
  sh.red = take(3 * M * M > ON_THREADS ? 3 * M * M : ON_THREADS);
  sh.sk = sh.red;
  sh.sv = sh.sk + M * M;
  sh.se = sh.sv + M * M;
  sh.red2 = take(130);
  sh.x = take(ng);
  sh.g = take(ng);
  sh.xn = take(ng);
  sh.gn = take(ng);
  sh.d = take(ng);
  sh.S = take((size_t)ON_HIST * ng);
  sh.Y = take((size_t)ON_HIST * ng);
  sh.rho = take(ON_HIST);
  sh.al = take(ON_HIST);
  sh.trig = take((size_t)p.nown * (3 * Ng + 2));
  sh.dE = take(M);
  sh.tv = take((size_t)2 * M * p.chunk);
  sh.te = take((size_t)2 * M * p.chunk);
  sh.mk = (int*)ptr;
  sh.orb = sh.mk + 2 * p.chunk;
  sh.epoch = &epoch;
  sh.mb = members;
  if (threadIdx.x == 0) epoch = 0;
  if (threadIdx.x < 4) members[threadIdx.x] = 0;

  for (int q = threadIdx.x; q < m; q += ON_THREADS) {
    const int r = p.weak_rank[q];
    sh.orb[p.subspace[q] * (p.n_weak_per + 1) + r + 1] = q;
  }
  for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.x[i] = p.gamma[i];
  __syncthreads();

  double E = 0.0;
  bool ok = on_evaluate(p, sh, sh.x, sh.g, &E);
  int iters = 0, reason = 1, hist = 0, head = 0;
  if (p.mode == 1) {
    for (int it = 0; ok && it < p.max_iter; ++it) {
      double gmax = 0.0;
      for (int i = threadIdx.x; i < ng; i += ON_THREADS) gmax = fmax(gmax, fabs(sh.g[i]));
      gmax = on_block_max(gmax, sh);
      if (gmax <= p.gtol) {
        reason = 0;
        break;
      }
      // two-loop recursion: d = -H g
      for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.d[i] = sh.g[i];
      __syncthreads();
      for (int k = 0; k < hist; ++k) {
        const int slot = (head - 1 - k + ON_HIST) % ON_HIST;
        const double a = sh.rho[slot] * on_dot(sh.S + (size_t)slot * ng, sh.d, ng, sh);
        if (threadIdx.x == 0) sh.al[slot] = a;
        for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.d[i] -= a * sh.Y[(size_t)slot * ng + i];
        __syncthreads();
      }
      double scale = 1.0;
      if (hist > 0) {
        const int slot = (head - 1 + ON_HIST) % ON_HIST;
        const double yy = on_dot(sh.Y + (size_t)slot * ng, sh.Y + (size_t)slot * ng, ng, sh);
        scale = yy > 0.0 ? 1.0 / (sh.rho[slot] * yy) : 1.0;
      } else {
        scale = gmax > 0.5 ? 0.5 / gmax : 1.0;  // first step: at most 0.5 rad in any angle
      }
      for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.d[i] *= scale;
      __syncthreads();
      for (int k = hist - 1; k >= 0; --k) {
        const int slot = (head - 1 - k + ON_HIST) % ON_HIST;
        const double yd = on_dot(sh.Y + (size_t)slot * ng, sh.d, ng, sh);
        // the product rounded on its own: the optimiser's path to the last digit rests on it
        const double c = sh.al[slot] - __dmul_rn(sh.rho[slot], yd);
        for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.d[i] += c * sh.S[(size_t)slot * ng + i];
        __syncthreads();
      }
      for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.d[i] = -sh.d[i];
      __syncthreads();
      double gd = on_dot(sh.g, sh.d, ng, sh);
      if (!(gd < 0.0)) {  // not a descent direction: restart from steepest descent
        hist = 0;
        const double sc = gmax > 0.5 ? 0.5 / gmax : 1.0;
        for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.d[i] = -sc * sh.g[i];
        __syncthreads();
        gd = on_dot(sh.g, sh.d, ng, sh);
      }
      // backtracking line search (Armijo, c1 = 1e-4)
      double t = 1.0, En = E;
      bool accepted = false;
      for (int ls = 0; ls < 40; ++ls) {
        for (int i = threadIdx.x; i < ng; i += ON_THREADS) sh.xn[i] = sh.x[i] + t * sh.d[i];
        __syncthreads();
        ok = on_evaluate(p, sh, sh.xn, sh.gn, &En);
        if (!ok) break;
        if (En <= E + 1e-4 * t * gd) {
          accepted = true;
          break;
        }
        t *= 0.5;
      }
      if (!accepted) {
        reason = 2;
        break;
      }
      // history update
      for (int i = threadIdx.x; i < ng; i += ON_THREADS) {
        sh.S[(size_t)head * ng + i] = sh.xn[i] - sh.x[i];
        sh.Y[(size_t)head * ng + i] = sh.gn[i] - sh.g[i];
      }
      __syncthreads();
      const double sy = on_dot(sh.S + (size_t)head * ng, sh.Y + (size_t)head * ng, ng, sh);
      if (sy > 0.0) {
        if (threadIdx.x == 0) sh.rho[head] = 1.0 / sy;
        head = (head + 1) % ON_HIST;
        hist = hist < ON_HIST ? hist + 1 : ON_HIST;
      }
      for (int i = threadIdx.x; i < ng; i += ON_THREADS) {
        sh.x[i] = sh.xn[i];
        sh.g[i] = sh.gn[i];
      }
      __syncthreads();
      const double dec = E - En;
      E = En;
      iters = it + 1;
      // Minima where an occupation reaches 0 or 1 sit on a kink of E(gamma) (the
      // sqrt(n) terms), where the gradient need not vanish: stop on the energy too.
      if (dec <= p.etol * fmax(1.0, fabs(E))) {
        reason = 3;
        break;
      }
    }
  }
  if (blockIdx.x != 0) return;
  // E depends on the angles through cos^2 and sin^2 only: an optimised gamma is
  // returned folded into [0, pi/2] (and its gradient with the matching sign).
  for (int i = threadIdx.x; i < ng; i += ON_THREADS) {
    double xi = sh.x[i], gi = sh.g[i];
    if (p.mode == 1) {
      const double c = cos(xi), s = sin(xi);
      xi = atan2(fabs(s), fabs(c));
      if (s * c < 0.0) gi = -gi;
    }
    p.gamma[i] = xi;
    p.grad_out[i] = gi;
  }
  if (threadIdx.x == 0) {
    p.E_out[0] = E;
    p.info_out[0] = iters;
    p.info_out[1] = p.mode == 1 ? reason : 0;
  }
}

// Features of each pairing subspace g for the learned warm start (one row of
// 3 + 4 N_g values): [H_ss, J_ss, mf_s, then per weak orbital w in rank order:
// H_ww, J_ww, K_sw, mf_w], with mf_p = sum_{q outside g} n0_q (2 J_pq - K_pq)
// the mean field of the other subspaces at the standard-guess occupations n0
// (strong 0.98, weak 0.02 / N_g).  Thread per (subspace, member).
__global__ void on_features_kernel(int NI, int Ng, int m, const int* subspace, const int* weak_rank, const double* J,
                                   const double* K, const double* Hd, float* X) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= NI * (Ng + 1)) return;
  const int g = t / (Ng + 1), k = t % (Ng + 1);
  int pp = -1, s = -1;
  for (int q = 0; q < m; ++q) {
    if (subspace[q] != g) continue;
    if (weak_rank[q] == k - 1) pp = q;
    if (weak_rank[q] < 0) s = q;
  }
  if (pp < 0 || s < 0) return;
  double mf = 0.0;
  for (int q = 0; q < m; ++q) {
    if (subspace[q] == g) continue;
    const double n0 = weak_rank[q] < 0 ? 0.98 : 0.02 / Ng;
    mf += n0 * (2.0 * J[(size_t)pp * m + q] - K[(size_t)pp * m + q]);
  }
  const int F = 3 + 4 * Ng;
  float* x = X + (size_t)g * F;
  if (k == 0) {
    x[0] = (float)Hd[pp];
    x[1] = (float)J[(size_t)pp * m + pp];
    x[2] = (float)mf;
  } else {
    float* y = x + 3 + 4 * (k - 1);
    y[0] = (float)Hd[pp];
    y[1] = (float)J[(size_t)pp * m + pp];
    y[2] = (float)K[(size_t)s * m + pp];
    y[3] = (float)mf;
  }
}

// Network outputs [N_I][N_g] -> gamma (strong angles, then the weak angles of each
// subspace), clipped to [clip, pi/2 - clip].
__global__ void on_unfold_kernel(const float* Y, int NI, int Ng, double clip, double* gamma) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= NI * Ng) return;
  const int g = t / Ng, j = t % Ng;
  double v = (double)Y[t];
  const double hi = 1.5707963267948966 - clip;
  v = v < clip ? clip : (v > hi ? hi : v);
  if (j == 0) gamma[g] = v;
  else gamma[NI + g * (Ng - 1) + j - 1] = v;
}

int onopt_features(donof_ri_ctx* ctx, float* d_X) {
  const int m = ctx->n_omega, nb = ctx->nbf, NI = ctx->n_strong, Ng = ctx->n_weak_per;
  int rc;
  if ((rc = launch_hc_public(ctx))) return rc;
  on_hdiag_kernel<<<ceil_div_u((long long)m * 32, 256), 256, 0, ctx->stream>>>(nb, m, ctx->d_C, ctx->d_HC,
                                                                               ctx->d_Hd);
  DONOF_LAUNCH_CHECK(ctx);
  on_features_kernel<<<ceil_div_u((long long)NI * (Ng + 1), 128), 128, 0, ctx->stream>>>(
      NI, Ng, m, ctx->d_subspace, ctx->d_weak_rank, ctx->d_J, ctx->d_K, ctx->d_Hd, d_X);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

int onopt_unfold(donof_ri_ctx* ctx, const float* d_Y, double clip, double* d_gamma) {
  const int NI = ctx->n_strong, Ng = ctx->n_weak_per;
  on_unfold_kernel<<<ceil_div_u((long long)NI * Ng, 128), 128, 0, ctx->stream>>>(d_Y, NI, Ng, clip, d_gamma);
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

// Runs the evaluation (mode 0) or the optimisation (mode 1) on the context's
// stream with gamma, E, grad and info in device memory.
int onopt_launch(donof_ri_ctx* ctx, double* d_gamma, double* d_E, double* d_grad, int* d_info, int mode,
                 int max_iter, double gtol, double etol) {
  const int m = ctx->n_omega, nb = ctx->nbf;
  const int ng = ctx->n_strong * ctx->n_weak_per;
  if (ctx->n_weak_per < 1 || ctx->n_weak_per > ON_MAX_WEAK) return DONOF_RI_E_UNSUPPORTED;
  int rc;
  if ((rc = launch_hc_public(ctx))) return rc;
  on_hdiag_kernel<<<ceil_div_u((long long)m * 32, 256), 256, 0, ctx->stream>>>(nb, m, ctx->d_C, ctx->d_HC,
                                                                               ctx->d_Hd);
  DONOF_LAUNCH_CHECK(ctx);
  OnParams p{};
  p.n_strong = ctx->n_strong;
  p.n_weak_per = ctx->n_weak_per;
  p.m = m;
  p.ng = ng;
  p.subspace = ctx->d_subspace;
  p.weak_rank = ctx->d_weak_rank;
  p.J = ctx->d_J;
  p.K = ctx->d_K;
  p.Hd = ctx->d_Hd;
  p.enuc = ctx->d_enuc;
  p.gamma = d_gamma;
  p.E_out = d_E;
  p.grad_out = d_grad;
  p.info_out = d_info;
  p.max_iter = max_iter;
  p.gtol = gtol;
  p.etol = etol;
  p.mode = mode;
  // one CTA per subspace, as far as the SMs go (a CTA needs an SM of its own at most)
  int dev = 0, sms = 0;
  DONOF_CUDA_TRY(cudaGetDevice(&dev));
  DONOF_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int Ng = p.n_weak_per, M = Ng + 1;
  const int grid = ctx->n_strong < sms ? ctx->n_strong : sms;
  p.nown = (ctx->n_strong + grid - 1) / grid;
  auto bytes = [&](int chunk) {
    return sizeof(double) * ((size_t)3 * m + (3 * M * M > ON_THREADS ? 3 * M * M : ON_THREADS) + 130 + 5 * (size_t)ng + 2 * (size_t)ON_HIST * ng + 2 * ON_HIST +
                             (size_t)p.nown * (3 * Ng + 2) + M + 4 * (size_t)M * chunk) +
           sizeof(int) * ((size_t)2 * chunk + (size_t)ctx->n_strong * M);
  };
  // the widest step of the row sums that fits beside the vectors
  for (p.chunk = 64; p.chunk > 4 && bytes(p.chunk) > SMEM_BLOCK_BYTES - 128;) p.chunk /= 2;
  const size_t smem = bytes(p.chunk);
  if (smem > SMEM_BLOCK_BYTES - 128) return DONOF_RI_E_UNSUPPORTED;
  DONOF_CUDA_TRY(allow_full_smem(on_opt_kernel));
  p.xch = ctx->d_on_xch;
  p.bar = (unsigned int*)(ctx->d_on_xch + 4 * (size_t)m + ng);
  p.status = ctx->d_status;
  DONOF_CUDA_TRY(cudaMemsetAsync(p.bar, 0, 2 * sizeof(unsigned int), ctx->stream));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(ON_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  DONOF_CUDA_TRY(cudaLaunchKernelEx(&cfg, on_opt_kernel, p));
  DONOF_LAUNCH_CHECK(ctx);
  return DONOF_RI_OK;
}

}  // namespace donof
