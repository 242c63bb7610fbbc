// Statistics of the solution pass (cr_post.cu, cr_post_tc.cu): identities, the
// fixed-order combination over a CTA, and one entry's contribution.
#pragma once

#include "cr_common.cuh"

namespace cr {

__device__ __forceinline__ double stat_op(int q, double a, double b) {
  if (q == PS_MIN) return fmin(a, b);
  if (q == PS_MAX || q == PS_MAXABS) return fmax(a, b);
  return a + b;
}

__device__ __forceinline__ double stat_identity(int q) {
  if (q == PS_MIN) return INFINITY;
  if (q == PS_MAX) return -INFINITY;
  return 0.0;
}

// An entry w of W against the reference's wr; returns P(w).
__device__ __forceinline__ double stat_add(double (&s)[PS_N], double w, double wr, int nonneg) {
  if (w < 0.0) {
    s[PS_NNEG] += 1.0;
    s[PS_NEG2] = fma(w, w, s[PS_NEG2]);
  }
  s[PS_MIN] = fmin(s[PS_MIN], w);
  s[PS_MAX] = fmax(s[PS_MAX], w);
  s[PS_W2] = fma(w, w, s[PS_W2]);
  const double pw = (nonneg && w < 0.0) ? 0.0 : w;
  const double d = pw - wr;
  s[PS_REF2] = fma(wr, wr, s[PS_REF2]);
  s[PS_DIFF2] = fma(d, d, s[PS_DIFF2]);
  s[PS_MAXABS] = fmax(s[PS_MAXABS], fabs(d));
  return pw;
}

// fixed-order combination of per-thread statistics over the CTA; thread 0 writes out[0..PS_N)
template <int THREADS>
__device__ void block_stats(double (&v)[PS_N], double* out) {
  __shared__ double scr[THREADS / 32][PS_N];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int q = 0; q < PS_N; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] = stat_op(q, v[q], __shfl_down_sync(0xffffffffu, v[q], o));
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < PS_N; ++q) scr[wid][q] = v[q];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int q = 0; q < PS_N; ++q) {
      double a = scr[0][q];
      for (int w = 1; w < nw; ++w) a = stat_op(q, a, scr[w][q]);
      out[q] = a;
    }
}

}  // namespace cr
