// The pieces of csrc/numeric.cuh run one by one, for tests/test_gpu_numeric.py.
#include "numeric.cuh"

using namespace donof;

// Column i: the running double-float sum of hi[k][i] + lo[k][i], k = 0 .. terms - 1 (n even).
__global__ void df_sums_kernel(const float* hi, const float* lo, int terms, int n, float* sh, float* sl) {
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  f32x2 s = 0, c = 0;
  for (int k = 0; k < terms; ++k) {
    const float *h = hi + (size_t)k * n + i, *l = lo + (size_t)k * n + i;
    df_add2(s, c, pack2(h[0], h[1]), pack2(l[0], l[1]));
  }
  unpack2(s, sh[i], sh[i + 1]);
  unpack2(c, sl[i], sl[i + 1]);
}

extern "C" int unit_df_sums(const float* hi, const float* lo, int terms, int n, float* sh, float* sl) {
  df_sums_kernel<<<(n / 2 + 127) / 128, 128>>>(hi, lo, terms, n, sh, sl);
  return (int)cudaDeviceSynchronize();
}

// q[i] = quotient(x[i], d[i], 1 / d[i]), ref[i] = x[i] / d[i].
__global__ void quotients_kernel(const double* x, const double* d, int n, double* q, double* ref) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  q[i] = quotient(x[i], d[i], 1.0 / d[i]);
  ref[i] = x[i] / d[i];
}

extern "C" int unit_quotients(const double* x, const double* d, int n, double* q, double* ref) {
  quotients_kernel<<<(n + 255) / 256, 256>>>(x, d, n, q, ref);
  return (int)cudaDeviceSynchronize();
}
