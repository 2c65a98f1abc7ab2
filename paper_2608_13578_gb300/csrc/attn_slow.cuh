// One row of the intra-block attention (Sec. 3.3) and of its backward from the
// tensors themselves, one key at a time in order, N columns of the row.  The
// tiled kernels multiply whole tiles, where a masked key has weight 0: that
// turns a non-finite value of another token into 0 x inf = NaN.  They recompute
// a row that came out non-finite with these, so that a non-finite token reaches
// the rows that see it and no others.
#pragma once

#include "common.cuh"

namespace bcmt {

// The tensors of one attention call (rows of token (b, t) at b*T + t).
template <class E>
struct AttnPtrs {
  const E *Q, *K, *V, *O, *dO;
  long ld, ld_o;
  const float* lse;
  int T, H, dh, L;
  float scale;
};

template <class E>
__device__ float slow_dot(const E* x, const E* y, int dh) {
  float s = 0.f;
  for (int c = 0; c < dh; ++c) s = fmaf(to_f(x[c]), to_f(y[c]), s);
  return s;
}
template <int N, class E>
__device__ __forceinline__ void slow_axpy(float p, const E* x, float* acc) {
  for (int e = 0; e < N; ++e) acc[e] = fmaf(p, to_f(x[e]), acc[e]);
}

// O_t, columns c .. c+N-1 of head h.
template <int N, class E>
__device__ void slow_o(const AttnPtrs<E>& a, int b, int h, int t, int c, float* out) {
  const int bs = (t / a.L) * a.L, h0 = h * a.dh;
  const long r0 = (long)b * a.T;
  const E* q = a.Q + (r0 + t) * a.ld + h0;
  float mx = -INFINITY, sum = 0.f;
  for (int j = bs; j <= t; ++j)
    mx = fmaxf(mx, a.scale * slow_dot(q, a.K + (r0 + j) * a.ld + h0, a.dh));
  for (int e = 0; e < N; ++e) out[e] = 0.f;
  for (int j = bs; j <= t; ++j) {
    const float p = expf(a.scale * slow_dot(q, a.K + (r0 + j) * a.ld + h0, a.dh) - mx);
    sum += p;
    slow_axpy<N>(p, a.V + (r0 + j) * a.ld + h0 + c, out);
  }
  for (int e = 0; e < N; ++e) out[e] /= sum;
}

// P_tj, and P_tj (dO_t . v_j - dO_t . O_t) * scale.
template <class E>
__device__ float slow_ds(const AttnPtrs<E>& a, int b, int h, int t, int j, float* p) {
  const long rt = (long)b * a.T + t, rj = (long)b * a.T + j;
  const int c = h * a.dh;
  const E* g = a.dO + rt * a.ld_o + c;
  *p = expf(a.scale * slow_dot(a.Q + rt * a.ld + c, a.K + rj * a.ld + c, a.dh) -
            a.lse[((long)b * a.H + h) * a.T + t]);
  return *p * a.scale *
         (slow_dot(g, a.V + rj * a.ld + c, a.dh) - slow_dot(g, a.O + rt * a.ld_o + c, a.dh));
}
template <int N, class E>
__device__ void slow_dq(const AttnPtrs<E>& a, int b, int h, int t, int c, float* out) {
  for (int e = 0; e < N; ++e) out[e] = 0.f;
  for (int j = (t / a.L) * a.L; j <= t; ++j) {
    float p;
    const float ds = slow_ds(a, b, h, t, j, &p);
    slow_axpy<N>(ds, a.K + ((long)b * a.T + j) * a.ld + h * a.dh + c, out);
  }
}
template <int N, class E>
__device__ void slow_dkv(const AttnPtrs<E>& a, int b, int h, int j, int c, float* dk, float* dv) {
  const int be = min((j / a.L + 1) * a.L, a.T);
  for (int e = 0; e < N; ++e) dk[e] = dv[e] = 0.f;
  for (int t = j; t < be; ++t) {
    float p;
    const float ds = slow_ds(a, b, h, t, j, &p);
    slow_axpy<N>(ds, a.Q + ((long)b * a.T + t) * a.ld + h * a.dh + c, dk);
    slow_axpy<N>(p, a.dO + ((long)b * a.T + t) * a.ld_o + h * a.dh + c, dv);
  }
}
__device__ __forceinline__ bool is_finite(float v) { return fabsf(v) <= 3.402823466e38f; }

}  // namespace bcmt
