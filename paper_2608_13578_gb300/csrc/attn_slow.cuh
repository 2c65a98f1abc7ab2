// Single rows of the intra-block attention (Sec. 3.3) and of its backward from the
// tensors themselves, a warp per row.  The tiled kernels multiply whole tiles, where a
// masked key has weight 0: that turns a non-finite value of another token into
// 0 x inf = NaN.  They form the values that came out non-finite again with these, so
// that a non-finite token reaches the rows that see it and no others.
//
// A row takes 32 keys (or queries) at a time: their weights, a half warp reading a key's
// row, then each lane adds them, in order, to the four columns it holds.  It ends as soon
// as its result is known to be NaN: at a NaN weight, or when every sum is one.  Costs at
// B2 T2048 h4 L1024 with heads of 128, finite / one NaN key / all NaN, in ms: CUDA-core
// forward 0.36 / 0.51 / 0.40, backward 0.56 / 0.89 / 0.57, tcgen05 backward 0.10 / 5.0 /
// 0.13 (126 rows of the last tile walk the block).  Formed by the threads that held
// them, a row and four or eight columns at a time, the one key cost 13, 104 and 2185 ms.
#pragma once

#include "common.cuh"

namespace bcmt {

// The tensors of one attention call (rows of token (b, t) at b*T + t).
template <class E>
struct AttnPtrs {
  const E *Q, *K, *V, *O, *dO;
  long ld, ld_o;
  const float* lse;
  const float* Drow;  // dO . O of every token, or null
  int T, H, dh, L;
  float scale;
  int vec;  // rows of Q, K, V are aligned to eight elements (those of O and dO always are)
};

// Lane u < n: row u of A times row u of B (row strides lda, ldb; 0: one row).
template <class E>
__device__ __forceinline__ void slow_load8(const E* p, bool vec, float* v) {
  if (vec) {
    load8(p, v);
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = to_f(p[e]);
  }
}
template <class E>
__device__ float slow_dots(const E* A, long lda, const E* B, long ldb, int n, int dh, bool vec) {
  const int lane = threadIdx.x & 31, c = (lane & 15) * 8;
  float out = 0.f, y[8];
  if (ldb == 0 && c < dh) slow_load8(B + c, vec, y);
#pragma unroll 8
  for (int i = 0; i < 16; ++i) {
    const int u = 2 * i + (lane >> 4);
    float s = 0.f;
    if (u < n && c < dh) {
      float x[8];
      slow_load8(A + u * lda + c, vec, x);
      if (ldb != 0) slow_load8(B + u * ldb + c, vec, y);
#pragma unroll
      for (int e = 0; e < 8; ++e) s = fmaf(x[e], y[e], s);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float s0 = __shfl_sync(0xffffffffu, s, 0), s1 = __shfl_sync(0xffffffffu, s, 16);
    if (lane >> 1 == i) out = lane & 1 ? s1 : s0;
  }
  return out;
}
constexpr int kSlowWeights = 32;  // floats of shared memory a warp needs
// The columns lane + 32 i of a row.
struct SlowRow {
  float v[4];
  __device__ __forceinline__ void set(float x) { v[0] = v[1] = v[2] = v[3] = x; }
  // += p x
  template <class E>
  __device__ __forceinline__ void add(float p, const E* x, int dh) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = (threadIdx.x & 31) + 32 * i;
      if (c < dh) v[i] = fmaf(p, to_f(x[c]), v[i]);
    }
  }
  // every column of the row is NaN (whole warp)
  __device__ __forceinline__ bool lost(int dh) const {
    bool f = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) f = f && ((int)(threadIdx.x & 31) + 32 * i >= dh || v[i] != v[i]);
    return __all_sync(0xffffffffu, f);
  }
};
__device__ __forceinline__ float slow_nan() { return __int_as_float(0x7fffffff); }
__device__ __forceinline__ bool is_finite(float v) { return fabsf(v) <= 3.402823466e38f; }

// O_t of head h.
template <class E>
__device__ void slow_o(const AttnPtrs<E>& a, int b, int h, int t, float* w, SlowRow& o) {
  const int lane = threadIdx.x & 31, bs = (t / a.L) * a.L, n = t - bs + 1;
  const long c = h * a.dh, r0 = (long)b * a.T + bs;
  const E *q = a.Q + ((long)b * a.T + t) * a.ld + c, *k = a.K + r0 * a.ld + c,
          *v = a.V + r0 * a.ld + c;
  float mx = -INFINITY;
  o.set(slow_nan());
  for (int u0 = 0; u0 < n; u0 += 32) {
    const float s = a.scale * slow_dots(k + u0 * a.ld, a.ld, q, 0, n - u0, a.dh, a.vec);
    if (__any_sync(0xffffffffu, s != s)) return;
    if (u0 + lane < n) mx = fmaxf(mx, s);
  }
  mx = warp_max(mx);
  if (!is_finite(mx)) return;  // inf - inf
  o.set(0.f);
  float sum = 0.f;
  for (int u0 = 0; u0 < n && !o.lost(a.dh); u0 += 32) {
    w[lane] = expf(a.scale * slow_dots(k + u0 * a.ld, a.ld, q, 0, n - u0, a.dh, a.vec) - mx);
    __syncwarp();
#pragma unroll 16
    for (int j = 0; j < min(32, n - u0); ++j) {
      sum += w[j];
      o.add(w[j], v + (u0 + j) * a.ld, a.dh);
    }
    __syncwarp();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) o.v[i] /= sum;
}

// dQ_t = scale * sum_j P_tj (dO_t . v_j - dO_t . O_t) k_j
template <class E>
__device__ void slow_dq(const AttnPtrs<E>& a, int b, int h, int t, float* w, SlowRow& dq) {
  const int lane = threadIdx.x & 31, bs = (t / a.L) * a.L, n = t - bs + 1;
  const long c = h * a.dh, rt = (long)b * a.T + t, r0 = (long)b * a.T + bs;
  const E *q = a.Q + rt * a.ld + c, *g = a.dO + rt * a.ld_o + c, *k = a.K + r0 * a.ld + c,
          *v = a.V + r0 * a.ld + c;
  const float lse = a.lse[((long)b * a.H + h) * a.T + t];
  dq.set(slow_nan());
  if (lse != lse) return;  // so is every weight
  const float drow = __shfl_sync(0xffffffffu, slow_dots(g, 0, a.O + rt * a.ld_o + c, 0, 1, a.dh, true), 0);
  if (drow != drow) return;
  dq.set(0.f);
  for (int u0 = 0; u0 < n && !dq.lost(a.dh); u0 += 32) {
    const float p = expf(a.scale * slow_dots(k + u0 * a.ld, a.ld, q, 0, n - u0, a.dh, a.vec) - lse);
    const float dp = slow_dots(v + u0 * a.ld, a.ld, g, 0, n - u0, a.dh, a.vec);
    w[lane] = p * a.scale * (dp - drow);
    __syncwarp();
#pragma unroll 16
    for (int j = 0; j < min(32, n - u0); ++j) dq.add(w[j], k + (u0 + j) * a.ld, a.dh);
    __syncwarp();
  }
}

// Per key j, over the queries t of its block from j on:
// DV: dV_j = sum_t P_tj dO_t, else dK_j = scale * sum_t P_tj (dO_t . v_j - dO_t . O_t) q_t.
template <bool DV, class E>
__device__ void slow_dkv(const AttnPtrs<E>& a, int b, int h, int j, float* w, SlowRow& d) {
  const int lane = threadIdx.x & 31, n = min((j / a.L + 1) * a.L, a.T) - j;
  const long c = h * a.dh, r0 = (long)b * a.T + j, l0 = ((long)b * a.H + h) * a.T + j;
  const E *k = a.K + r0 * a.ld + c, *v = a.V + r0 * a.ld + c, *q = a.Q + r0 * a.ld + c,
          *g = a.dO + r0 * a.ld_o + c, *o = a.O + r0 * a.ld_o + c;
  // with its log-sum-exp all of a query's weights are NaN; with its dO . O, for dK
  bool nan = false;
  for (int u = lane; u < n; u += 32) {
    const float l = a.lse[l0 + u], dr = !DV && a.Drow ? a.Drow[l0 + u] : 0.f;
    nan = nan || l != l || dr != dr;
  }
  d.set(slow_nan());
  if (__any_sync(0xffffffffu, nan)) return;
  d.set(0.f);
  for (int u0 = 0; u0 < n && !d.lost(a.dh); u0 += 32) {
    const long l = l0 + min(u0 + lane, n - 1);
    float p = expf(a.scale * slow_dots(q + u0 * a.ld, a.ld, k, 0, n - u0, a.dh, a.vec) - a.lse[l]);
    if (!DV) {
      const float drow = a.Drow ? a.Drow[l]
                                : slow_dots(g + u0 * a.ld_o, a.ld_o, o + u0 * a.ld_o, a.ld_o, n - u0,
                                            a.dh, true);
      p *= a.scale * (slow_dots(g + u0 * a.ld_o, a.ld_o, v, 0, n - u0, a.dh, a.vec) - drow);
    }
    w[lane] = p;
    __syncwarp();
#pragma unroll 16
    for (int i = 0; i < min(32, n - u0); ++i)
      d.add(w[i], DV ? g + (u0 + i) * a.ld_o : q + (u0 + i) * a.ld, a.dh);
    __syncwarp();
  }
}

// Calls f(n, columns, scratch) by whole warps for every row n < N of which a thread of
// the CTA has marked a group of columns: mark(set) calls set(n, group), columns is the
// row's bit set of groups.  sm: free shared memory, N + 32 a warp floats.
template <int N, class M, class F>
__device__ __forceinline__ void slow_rows(float* sm, M&& mark, F&& f) {
  unsigned* set = reinterpret_cast<unsigned*>(sm);
  const int warp = threadIdx.x >> 5;
  for (int n = threadIdx.x; n < N; n += blockDim.x) set[n] = 0u;
  __syncthreads();
  mark([&](int n, int group) { atomicOr(&set[n], 1u << group); });
  __syncthreads();
  for (int n = warp; n < N; n += blockDim.x >> 5)
    if (set[n]) f(n, set[n], sm + N + warp * kSlowWeights);
}

}  // namespace bcmt
