// FP32 normalized regular harmonics for P2M / L2P (see harmonics.cuh).
#pragma once
#include "common.cuh"

namespace fmm {

// Factors of the recurrences R~_n^m = f.x ((2n - 1) z R~_{n-1}^m - r^2 f.y R~_{n-2}^m):
// (rsqrt((n + m)(n - m)), sqrt((n + m - 1)(n - m - 1))) for n > m, and on the
// diagonal the factor from R~_{m-1}^{m-1} to R~_m^m.  Full warps compute them (the
// shared-memory pipe is what the sweeps' inner loops wait for: L2P of Taylor-Green
// 128^3 0.55 ms, 0.67 from a table); thread groups that share a leaf's columns read
// a table, [n (n + 1) / 2 + m].
__device__ inline float2 recurrence(int n, int m) {
  return n == m ? make_float2(sqrtf((2.f * m - 1.f) / (2.f * m)), 0.f)
                : make_float2(rsqrtf((float)((n + m) * (n - m))), sqrtf((float)((n + m - 1) * (n - m - 1))));
}
inline size_t recurrence_bytes(int p) { return (size_t)p * (p + 1) / 2 * sizeof(float2); }
__device__ inline void fill_recurrence(float2* f, int p, int t, int threads) {
  for (int e = t; e < p * p; e += threads) {
    const int n = e / p, m = e % p;
    if (m <= n && n > 0) f[n * (n + 1) / 2 + m] = recurrence(n, m);
  }
}

// Threads per group when n particles are spread over a CTA of `threads`, whose
// groups then share the columns of an expansion of degree p - 1 (short
// expansions stay whole: the groups' setup and sums cost what they save) ...
__device__ inline int column_width(int n, int p, int threads) {
  return n > 32 || p < 8 ? threads : (n <= 8 ? 8 : (n <= 16 ? 16 : 32));
}
// ... and the column of group grp of G in round i: rounds run back and forth.
__device__ inline int folded_column(int i, int grp, int G) { return i * G + ((i & 1) ? G - 1 - grp : grp); }

}  // namespace fmm
