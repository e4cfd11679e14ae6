// The pairs j < i of n things in the order (1, 0), (2, 0), (2, 1), (3, 0), ...; pair t has
// t = i (i - 1) / 2 + j.  64-bit counts: 46342 nuclei already have more than 2^31 / 2 pairs.
// (Also compiled for the host, by the tests.)
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define DONOF_HD __host__ __device__ __forceinline__
#else
#define DONOF_HD inline
#endif

namespace donof {

DONOF_HD long long pair_count(int n) { return (long long)n * (n - 1) / 2; }

// i and j of pair t (0 <= t < 2^61): an FP32 root, then steps of one.
DONOF_HD void pair_at(long long t, int& i, int& j) {
  long long r = (long long)((1.0f + sqrtf(8.0f * (float)t + 1.0f)) * 0.5f);
  while (r * (r - 1) / 2 > t) --r;
  while (r * (r + 1) / 2 <= t) ++r;
  i = (int)r;
  j = (int)(t - r * (r - 1) / 2);
}

}  // namespace donof
