// Incremental decoding: one new token per sequence per call, with the state
// that the forward of Sec. 3 implies for a causal stream (the paper trains
// only; this follows from Sec. 3.3-3.8).  Token t = pos of block i = pos / L,
// slot j = pos % L:
//   * attention over the keys of block i up to slot j (the block's K/V cache);
//   * H_t, then G_t = sigmoid(H_t W_g) and Y_t = H_t + G_t * C_i, where C_i is
//     P_{i-1} = M_{i-1} W_m (zero in block 0);
//   * the block summary accumulated online: running max m, denominator
//     sum exp(s - m) and numerator sum exp(s - m) H of the scores s = H w_p;
//   * at the last slot of a block, S_i = num / den, the memory recurrence
//     N_i = a N_{i-1} + S_i, Z_i = a Z_{i-1} + 1, M_i = N_i / Z_i, and the next
//     block's memory row C_{i+1} = M_i W_m.
// Values the full forward stores in the storage dtype (Q/K/V, Concat(heads),
// H, M) are rounded to it here too, so that a decoded token reproduces the
// forward's output row.  bf16 steps run as one launch (decode_cluster_kernel);
// fp32 steps, and bf16 shapes too large for it or faster so (staged_is_faster), as a
// launch per stage, whose vector-matrix products stream each weight once on CUDA cores.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace bcmt {

int g_decode_one_launch = 1;  // switchable only through bcmt_testing.h

namespace {
constexpr int kMaxL = 1024;

template <class T>
__device__ __forceinline__ float round_to(float v) {
  return to_f<T>(from_f<T>(v));
}
}  // namespace

// out[m, n] = sum_k A[m, k] W[k, n] (fp32 accumulate), A fp32 [M, K], W [K, N]
// row-major.  CTA: 32 columns (lane = column) x R rows of A; its 32 warps
// split K (warp g takes rows g, g+32, ...), each thread issuing all eight
// weight loads of a 256-row chunk before using them, and the warps' sums are
// added in warp order.  With round_out the result is rounded to TW.
template <class TW, int R>
__global__ void __launch_bounds__(1024)
    decode_gemv_kernel(const float* __restrict__ A, int M, int K, const TW* __restrict__ W, int N,
                       float* __restrict__ out, int round_out) {
  pdl_enter();
  A = after_wait(A);
  constexpr int KC = 256;  // K chunk staged in shared memory
  __shared__ float sA[R][KC];
  extern __shared__ float red[];  // [32 warps][R][33]
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
  const int n = blockIdx.x * 32 + lane;
  const int m0 = blockIdx.y * R;
  const int mc = min(R, M - m0);
  float acc[R];
#pragma unroll
  for (int m = 0; m < R; ++m) acc[m] = 0.f;
  for (int k0 = 0; k0 < K; k0 += KC) {
    for (int i = tid; i < R * KC; i += 1024) {
      const int m = i / KC, k = i - m * KC;
      sA[m][k] = (m < mc && k0 + k < K) ? A[(long)(m0 + m) * K + k0 + k] : 0.f;
    }
    __syncthreads();
    if (n < N) {
      const int kend = min(KC, K - k0);
      float wv[KC / 32];
#pragma unroll
      for (int u = 0; u < KC / 32; ++u) {
        const int kk = g + 32 * u;
        wv[u] = kk < kend ? to_f(W[(long)(k0 + kk) * N + n]) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < KC / 32; ++u) {
        const int kk = g + 32 * u;  // < KC; zero weight past kend
#pragma unroll
        for (int m = 0; m < R; ++m) acc[m] = fmaf(sA[m][kk], wv[u], acc[m]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int m = 0; m < R; ++m) red[(g * R + m) * 33 + lane] = acc[m];
  __syncthreads();
  for (int i = tid; i < R * 32; i += 1024) {
    const int m = i / 32, c = i - m * 32;
    const int col = blockIdx.x * 32 + c;
    if (m < mc && col < N) {
      float t = 0.f;
      for (int q = 0; q < 32; ++q) t += red[(q * R + m) * 33 + c];
      out[(long)(m0 + m) * N + col] = round_out ? round_to<TW>(t) : t;
    }
  }
}

// One CTA per (head h, sequence b): stores k, v of the new token in the
// block's cache slot j, then attends the (rounded) query over slots 0..j.
template <class T>
__global__ void __launch_bounds__(128)
    decode_attn_kernel(const float* __restrict__ qkv, T* __restrict__ Kc, T* __restrict__ Vc,
                       float* __restrict__ hhat, int D, int dh, int L, int j, float scale) {
  pdl_enter();
  qkv = after_wait(qkv);
  Kc = after_wait(Kc);
  Vc = after_wait(Vc);
  __shared__ float q[128];
  __shared__ float p[kMaxL];
  __shared__ float red[2][4];
  const int h = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const float* row = qkv + (long)b * 3 * D;
  const long cache = (long)b * L * D;
  if (tid >= dh) q[tid] = 0.f;  // channels past dh multiply zero-filled key values
  for (int c = tid; c < dh; c += 128) {
    const int col = h * dh + c;
    q[c] = round_to<T>(row[col]);
    Kc[cache + (long)j * D + col] = from_f<T>(row[D + col]);
    Vc[cache + (long)j * D + col] = from_f<T>(row[2 * D + col]);
  }
  __syncthreads();
  float mx = -INFINITY;
  for (int u = tid; u <= j; u += 128) {
    // key u's row, 32 channels at a time: the four 16-byte loads go out together
    const T* kr = Kc + cache + (long)u * D + h * dh;
    float s = 0.f;
    for (int c0 = 0; c0 < dh; c0 += 32) {
      float kv[32];
#pragma unroll
      for (int q8 = 0; q8 < 4; ++q8) {
        if (c0 + 8 * q8 < dh) {
          load8(kr + c0 + 8 * q8, kv + 8 * q8);
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) kv[8 * q8 + e] = 0.f;
        }
      }
#pragma unroll
      for (int e = 0; e < 32; ++e) s = fmaf(q[min(c0 + e, 127)], kv[e], s);
    }
    s *= scale;
    p[u] = s;
    mx = fmaxf(mx, s);
  }
  mx = warp_max(mx);
  if (lane == 0) red[0][warp] = mx;
  __syncthreads();
  mx = fmaxf(fmaxf(red[0][0], red[0][1]), fmaxf(red[0][2], red[0][3]));
  float sum = 0.f;
  for (int u = tid; u <= j; u += 128) {
    const float e = expf(p[u] - mx);
    p[u] = e;
    sum += e;
  }
  sum = warp_sum(sum);
  if (lane == 0) red[1][warp] = sum;
  __syncthreads();
  sum = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]);
  const float inv = 1.0f / sum;
  for (int c = tid; c < dh; c += 128) {
    const T* vc = Vc + cache + h * dh + c;
    float o = 0.f;
#pragma unroll 8
    for (int u = 0; u <= j; ++u) o = fmaf(p[u], to_f(vc[(long)u * D]), o);
    hhat[(long)b * D + h * dh + c] = round_to<T>(o * inv);
  }
}

// One CTA per sequence b.  H (already rounded), U = H W_g (fp32) -> Y; the
// online block summary; at the block's last slot the summary, the memory
// recurrence and the rounded M for the next block's projection.
template <class T>
__global__ void __launch_bounds__(256)
    decode_post_kernel(const float* __restrict__ Hr, const float* __restrict__ U,
                       const T* __restrict__ w_p, const float* __restrict__ decay,
                       float* __restrict__ Cm, float* __restrict__ pm, float* __restrict__ pden,
                       float* __restrict__ pnum, float* __restrict__ Nn, float* __restrict__ Zz,
                       float* __restrict__ Mr, T* __restrict__ y, int D, int j, int last,
                       int honly) {
  pdl_enter();
  Hr = after_wait(Hr);
  U = after_wait(U);
  Cm = after_wait(Cm);
  pm = after_wait(pm);
  pden = after_wait(pden);
  pnum = after_wait(pnum);
  Nn = after_wait(Nn);
  Zz = after_wait(Zz);
  __shared__ float red[8];
  const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* h = Hr + (long)b * D;
  if (honly) {
    for (int c = tid; c < D; c += 256) y[(long)b * D + c] = from_f<T>(h[c]);
    return;
  }
  float s = 0.f;
  for (int c = tid; c < D; c += 256) s = fmaf(h[c], to_f(w_p[c]), s);
  s = warp_sum(s);
  if (lane == 0) red[warp] = s;
  __syncthreads();
  s = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) s += red[w];
  // online softmax of the block's scores (slot 0 starts a new block)
  const float m_old = j == 0 ? s : pm[b];
  const float m_new = fmaxf(m_old, s);
  const float f_old = j == 0 ? 0.f : expf(m_old - m_new);
  const float e = expf(s - m_new);
  const float den = (j == 0 ? 0.f : pden[b]) * f_old + e;
  for (int c = tid; c < D; c += 256) {
    const long o = (long)b * D + c;
    y[o] = from_f<T>(fmaf(sigmoidf_(U[o]), Cm[o], h[c]));
    const float num = (j == 0 ? 0.f : pnum[o]) * f_old + e * h[c];
    if (last) {
      const float a = decay[c];
      const float n = fmaf(a, Nn[o], num / den);
      const float z = fmaf(a, Zz[o], 1.0f);
      Nn[o] = n;
      Zz[o] = z;
      Mr[o] = round_to<T>(n / z);
    } else {
      pnum[o] = num;
    }
  }
  __syncthreads();  // every thread has read pm[b] and pden[b]
  if (tid == 0 && !last) {
    pm[b] = m_new;
    pden[b] = den;
  }
}

// ------------------------------------------------ one launch per token (bf16)
// A whole step of up to 16 sequences in one thread-block cluster.  The stages are
// matrix-vector products over the same weights, each too short to be worth a
// launch (two to three microseconds of start-up, six of them a token), and a
// cluster's barrier costs a fraction of that.  CTA c of the cluster
//   1. multiplies the token rows by the q, k, v columns of its heads (of its part
//      of a head's columns when there are few heads), appends k and v to the
//      cache, attends over the block's cached keys,
//   2. multiplies the heads' outputs by its columns of W_O,
//   3. multiplies H by its columns of W_g, injects the memory, updates the block
//      summary and at the block's last slot the memory recurrence,
//   4. there also multiplies M by its columns of W_m.
// A stage's rows go straight into every CTA's shared memory (distributed shared
// memory stores), a cluster barrier follows.  What a stage reads beside them does
// not depend on this token's earlier stages and is fetched ahead: the weights of
// the next product into registers before the barrier, the cached keys and values,
// w_p and the running sums at the start.  Bound: the weights' way from L2 into
// the cluster's 16 SMs (64 B per cycle each) and the chain of barriers; sequences
// are spread over up to kDecClusters clusters, each of which streams all weights.
// A token took (queued calls, launch per stage, then this): B = 1, D = 512, h = 8,
// L = 64 28.8 and 16.6 us (the host's part by then); B = 16, D = 1024, h = 16,
// L = 128 66.5 and 23.5 us.
//
// Products: mma.sync m16n8k16 with the weights as the 16-row operand (columns of W)
// and the sequences as the 8 columns of the other, so that a few sequences waste
// half as much as rows would (the instruction takes about 17 cycles of an SM
// quarter here whatever it carries).  A chunk is 64 columns of W (eight pieces of
// eight); the 16 warps share the chunks and split K, each taking every nks-th
// 16-deep step.  A load instruction reads four rows, eight consecutive lanes the
// 128 bytes of one (lane l: piece l % 8, row 4 (l / 8) + i; with the lanes of a row
// spread over the warp, as the fragments want them, an SM draws 23 bytes per cycle
// from L2 instead of 59), four steps ahead; sixteen shuffles then hand lane l the
// piece l / 4 of rows 4 (l % 4) + i, two rows' values are interleaved into the
// fragments: tile e is column e of the pieces in its upper eight rows and column
// e + 4 in its lower.  Weights never touch shared memory; the warps' partial sums
// are added in a fixed order.  One copy of this code serves every product.
constexpr int kDecThreads = 512;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecClusters = 4;
constexpr int kDecRows = 16;       // sequences per cluster (mma rows)
constexpr int kDecSmem = 200 * 1024;
constexpr int kDecStage = 96 * 1024;  // at most this much of the cache is staged

struct DecodeClusterArgs {
  const bf16 *x, *w_qkv, *w_o, *w_p, *w_m, *w_g;
  const float* decay;
  bf16* y;
  bf16 *Kc, *Vc;
  float *pm, *pden, *pnum, *N, *Z, *C;
  int B, D, heads, dh, L, j, honly, last;
  int spc;    // sequences per cluster
  int parts;  // CTAs that share a head's columns
  int stage;  // the cached keys and values go through shared memory
  float scale;
  // divisions done by the host: log2(parts), and reciprocals for small quotients
  // (DecDiv) by the chunks of a q, k, v slot and of the CTA's columns, by a part's
  // pieces, by the warps of a sequence (nw) and by the columns' pieces
  int lparts, nch_q, nch_c, nks_q, nks_c, nw, inv_q, inv_c, inv_per, inv_nw, inv_cols;
  struct DecodeClusterSmem {
    int slots, pw, cols, arows;
    int a[2], red, qkv, sc, out, wp, kv, bytes;  // byte offsets
  } sm;
};
using DecodeClusterSmem = DecodeClusterArgs::DecodeClusterSmem;
// x / d as (x * dec_inv(d)) >> 16, exact for x < 1024 and d <= 64 (x (d - 1) < 65536)
__host__ __device__ constexpr int dec_inv(int d) { return (65536 + d - 1) / d; }
__device__ __forceinline__ int dec_div(int x, int inv) { return (x * inv) >> 16; }

__device__ __forceinline__ uint4 ld_weight16(const void* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ void dec_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctas() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void st_cluster16(uint32_t addr, uint4 v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ void st_cluster_f(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void mma_16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One product of the cluster's rows, `groups` pieces of eight columns: this
// thread's share.
struct DecJob {
  const bf16* w;  // row 4 (lane / 8) of the thread's piece
  long ld;
  int s0, nks, steps;  // K steps s0, s0 + nks, ...
  int groups, chunk;
  bool on;
};
constexpr int kDecU = 4;  // K steps held at a time
// One step's weights of the thread.
__device__ __forceinline__ void dec_step_fetch(const DecJob& t, int s, uint4* w) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    w[r] = make_uint4(0u, 0u, 0u, 0u);
    if (t.on && s < t.steps)
      w[r] = ld_weight16(t.w + (long)(16 * s + r) * t.ld);
  }
}
__device__ __forceinline__ void dec_permute(const uint4& v, int src, uint32_t* r) {
  r[0] = __shfl_sync(0xffffffffu, v.x, src);
  r[1] = __shfl_sync(0xffffffffu, v.y, src);
  r[2] = __shfl_sync(0xffffffffu, v.z, src);
  r[3] = __shfl_sync(0xffffffffu, v.w, src);
}
// The product of NT * 8 sequences, the first kDecU steps already in w: the warps'
// partial sums in red[part][row][8 g + e], row < rows.
template <int NT>
__device__ __forceinline__ void dec_run(const DecJob& t, uint4 (*w)[4], const bf16* A, int lda,
                                        int rows, float* red) {
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3, src = 8 * c + g;
  float acc[NT][4][4];
#pragma unroll
  for (int m = 0; m < NT; ++m)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[m][e][0] = acc[m][e][1] = acc[m][e][2] = acc[m][e][3] = 0.f;
  for (int f = t.s0; f < t.steps; f += kDecU * t.nks) {
#pragma unroll
    for (int u = 0; u < kDecU; ++u) {
      const int s = f + u * t.nks;
      if (s < t.steps) {
        uint2 x[NT];  // sequence l / 4 (+8), rows 4 (l % 4) .. +3 of the step
#pragma unroll
        for (int m = 0; m < NT; ++m)
          x[m] = *reinterpret_cast<const uint2*>(A + (g + 8 * m) * lda + 16 * s + 4 * c);
        uint32_t r0[4], r1[4], r2[4], r3[4];
        dec_permute(w[u][0], src, r0);
        dec_permute(w[u][1], src, r1);
        dec_permute(w[u][2], src, r2);
        dec_permute(w[u][3], src, r3);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t sel = (e & 1) ? 0x7632u : 0x5410u;
          const int h = e >> 1;
          const uint32_t fr[4] = {__byte_perm(r0[h], r1[h], sel), __byte_perm(r0[h + 2], r1[h + 2], sel),
                                  __byte_perm(r2[h], r3[h], sel), __byte_perm(r2[h + 2], r3[h + 2], sel)};
#pragma unroll
          for (int m = 0; m < NT; ++m) mma_16816(acc[m][e], fr, x[m].x, x[m].y);
        }
      }
      dec_step_fetch(t, s + kDecU * t.nks, w[u]);
    }
  }
  // tile e: column e (rows 0-7: element 0, 1) or e + 4 (rows 8-15: 2, 3) of group
  // l / 4, sequences 2 (l % 4) + {0, 1}
  const int gi = t.chunk * 8 + g, wide = 8 * t.groups;
  if (t.steps > 0 && gi < t.groups) {
#pragma unroll
    for (int m = 0; m < NT; ++m)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int row = 8 * m + 2 * c + q;
        if (row < rows) {
          float* p = red + (t.s0 * rows + row) * wide + 8 * gi;
          *reinterpret_cast<float4*>(p) =
              make_float4(acc[m][0][q], acc[m][1][q], acc[m][2][q], acc[m][3][q]);
          *reinterpret_cast<float4*>(p + 4) =
              make_float4(acc[m][0][2 + q], acc[m][1][2 + q], acc[m][2][2 + q], acc[m][3][2 + q]);
        }
      }
  }
}
// q . k over pw columns (two chains).
__device__ __forceinline__ float dec_dot(const float* q, const bf16* k, int pw) {
  float d0 = 0.f, d1 = 0.f;
#pragma unroll 4
  for (int c = 0; c < pw; c += 8) {
    float v[8];
    load8(k + c, v);
    const float4 a = *reinterpret_cast<const float4*>(q + c);
    const float4 b = *reinterpret_cast<const float4*>(q + c + 4);
    d0 = fmaf(a.x, v[0], d0);
    d1 = fmaf(a.y, v[1], d1);
    d0 = fmaf(a.z, v[2], d0);
    d1 = fmaf(a.w, v[3], d1);
    d0 = fmaf(b.x, v[4], d0);
    d1 = fmaf(b.y, v[5], d1);
    d0 = fmaf(b.z, v[6], d0);
    d1 = fmaf(b.w, v[7], d1);
  }
  return d0 + d1;
}
// o += sum over cnt keys of p[u] v[u * ld + c], at columns ca, ca + 1 and cb, cb + 1.
__device__ __forceinline__ void dec_pv(const float* p, const bf16* v, long ld, int cnt, int ca,
                                       int cb, float2& oa, float2& ob) {
#pragma unroll 8
  for (int u = 0; u < cnt; ++u) {
    const float e = p[u];
    const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(v + u * ld + ca));
    const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(v + u * ld + cb));
    oa.x = fmaf(e, x.x, oa.x);
    oa.y = fmaf(e, x.y, oa.y);
    ob.x = fmaf(e, y.x, ob.x);
    ob.y = fmaf(e, y.y, ob.y);
  }
}
// Calls f(row, column, sum) for every output (128 threads a row), the partial sums
// added in order.
template <class F>
__device__ __forceinline__ void dec_sums(const float* red, int parts, int rows, int wide, F&& f) {
  for (int b = threadIdx.x >> 7; b < rows; b += kDecThreads / 128)
    for (int c = threadIdx.x & 127; c < wide; c += 128) {
      float v = 0.f;
#pragma unroll 8
      for (int k = 0; k < parts; ++k) v += red[(k * rows + b) * wide + c];
      f(b, c, v);
    }
}

// Shared memory of a step.
static DecodeClusterSmem dec_smem(int D, int heads, int dh, int L, int parts, int spc, int ctas,
                                  int stage) {
  DecodeClusterSmem s;
  s.slots = (heads * parts + ctas - 1) / ctas;
  s.pw = dh / parts;
  s.cols = (D / 8 + ctas - 1) / ctas * 8;
  s.arows = spc <= 8 ? 8 : 16;
  const int a = s.arows * (D + 8) * 2;
  s.a[0] = 0;                                    // x, then H
  s.a[1] = a;                                    // Concat(heads), then M
  s.red = 2 * a;                                 // partial sums; the attention's
  s.qkv = s.red + std::max(spc * kDecWarps * 64, kDecWarps * (s.pw + 4)) * 4;
  s.sc = s.qkv + s.slots * spc * 3 * s.pw * 4;   // scores, per part
  s.out = s.sc + ((parts * s.slots * spc * L + 3) & ~3) * 4;  // a product's columns
  s.wp = s.out + (spc * s.cols + kDecWarps * kDecRows) * 4;   // and the pooling scores; w_p
  s.kv = s.wp + D * 2;                           // keys, then values
  s.bytes = s.kv + (stage ? 2 * s.slots * spc * L * (s.pw + 8) * 2 : 0);
  return s;
}

template <int NT>
__global__ void __launch_bounds__(kDecThreads, 1)
    decode_cluster_kernel(const __grid_constant__ DecodeClusterArgs a) {
  extern __shared__ __align__(16) uint8_t dsm[];
  const int rank = (int)tc::cluster_rank(), ctas = (int)cluster_ctas();
  const DecodeClusterSmem& lay = a.sm;
  bf16* Ax = reinterpret_cast<bf16*>(dsm + lay.a[0]);
  bf16* Ah = reinterpret_cast<bf16*>(dsm + lay.a[1]);
  float* red = reinterpret_cast<float*>(dsm + lay.red);
  float* qkv = reinterpret_cast<float*>(dsm + lay.qkv);
  float* sc = reinterpret_cast<float*>(dsm + lay.sc);
  float* out = reinterpret_cast<float*>(dsm + lay.out);
  float* sr = out + a.spc * lay.cols;  // [16 warps][16]: shares of the pooling scores
  bf16* wps = reinterpret_cast<bf16*>(dsm + lay.wp);
  bf16* Ks = reinterpret_cast<bf16*>(dsm + lay.kv);
  bf16* Vs = Ks + (size_t)lay.slots * a.spc * a.L * (lay.pw + 8);
  const int D = a.D, lda = D + 8, dh = a.dh, pw = lay.pw, n = a.j + 1;
  const int b0 = (int)cluster_id() * a.spc, rows = min(a.spc, a.B - b0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int units = a.heads * a.parts;
  int nslots = 0;
  while (rank + nslots * ctas < units) ++nslots;
  const int first = rank * lay.cols, cols = max(0, min(lay.cols, D - first));
  const int inv_mine = cols == lay.cols || cols == 0 ? a.inv_cols : dec_inv(cols / 8);
  auto unit_col = [&](int s) {
    const int unit = rank + s * ctas;
    return (unit >> a.lparts) * dh + (unit & (a.parts - 1)) * pw;
  };
  // product p of this CTA: its q, k, v slots, then W_O, W_g, W_m
  auto job = [&](int p) {
    DecJob t;
    const bool q = p < nslots;
    const int nch = q ? a.nch_q : a.nch_c;
    t.s0 = dec_div(warp, q ? a.inv_q : a.inv_c);
    t.chunk = warp - t.s0 * nch;
    t.nks = q ? a.nks_q : a.nks_c;
    t.steps = t.s0 < t.nks ? D / 16 : 0;
    t.groups = q ? 3 * pw / 8 : cols / 8;
    const int g = t.chunk * 8 + (lane & 7);
    t.on = g < t.groups;
    const bf16* W = q ? a.w_qkv : p == nslots ? a.w_o : p == nslots + 1 ? a.w_g : a.w_m;
    t.ld = q ? 3 * D : D;
    int col = first + 8 * g;
    if (q) {
      const int m = dec_div(g, a.inv_per);  // q, k or v
      col = m * D + unit_col(p) + 8 * (g - m * (pw / 8));
    }
    t.w = W + (t.on ? col : 0) + (long)(4 * (lane >> 3)) * t.ld;
    return t;
  };
  // 8 per columns per row of `src` (rows ldsrc floats apart; inv: 1 / per) as bf16
  // into the rows of every CTA's `A`, from column col: a warp per CTA
  auto push = [&](bf16* A, const float* src, int ldsrc, int per, int inv, int col) {
    for (int i = lane; i < rows * per; i += 32) {
      const int b = dec_div(i, inv), c = 8 * (i - b * per);
      const float4 lo = *reinterpret_cast<const float4*>(src + b * ldsrc + c);
      const float4 hi = *reinterpret_cast<const float4*>(src + b * ldsrc + c + 4);
      const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
      uint4 u;
      uint32_t* w = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
        w[e] = *reinterpret_cast<const uint32_t*>(&h);
      }
      const uint32_t to = tc::smem_u32(A + b * lda + col + c);
      for (int cta = warp; cta < ctas; cta += kDecWarps)
        st_cluster16(tc::mapa(to, (uint32_t)cta), u);
    }
  };

  // rows past the cluster's sequences stay zero
  for (int i = tid; i < 2 * lay.arows * lda / 8; i += kDecThreads)
    reinterpret_cast<uint4*>(Ax)[i] = make_uint4(0u, 0u, 0u, 0u);
  tc::cluster_sync();  // every CTA is there, its rows are cleared
  pdl_enter();

  // ---- everything that does not wait for this token's own stages
  for (int b = warp; b < rows; b += kDecWarps)
    for (int c = 8 * lane; c < D; c += 256)
      dec_cp16(Ax + b * lda + c, a.x + (long)(b0 + b) * D + c);
  asm volatile("cp.async.commit_group;" ::: "memory");
  uint4 w[kDecU][4];
  DecJob t = job(0);
#pragma unroll
  for (int u = 0; u < kDecU; ++u) dec_step_fetch(t, t.s0 + u * t.nks, w[u]);
  if (a.stage) {  // a warp per cached row: lanes 0-15 its key, 16-31 its value
    const int c = (lane & 15) * 8;
    for (int s = 0; s < nslots; ++s)
      for (int b = 0; b < rows; ++b)
        for (int u = warp; u < a.j; u += kDecWarps)
          if (c < pw)
            dec_cp16((lane < 16 ? Ks : Vs) + ((s * a.spc + b) * a.L + u) * (pw + 8) + c,
                     (lane < 16 ? a.Kc : a.Vc) + ((long)(b0 + b) * a.L + u) * D + unit_col(s) + c);
  }
  if (!a.honly)
    for (int i = tid; i < D / 8; i += kDecThreads) dec_cp16(wps + 8 * i, a.w_p + 8 * i);
  asm volatile("cp.async.commit_group;" ::: "memory");
  // the running sums of the thread's first output element
  const int rd = (a.j + 1) & 1, wr = a.j & 1;  // the pair of the last slot, of this one
  float st_C = 0.f, st_num = 0.f, st_N = 0.f, st_Z = 0.f, st_a = 0.f, st_m = 0.f, st_den = 0.f;
  auto state = [&](int b, int col) {
    const long o = (long)(b0 + b) * D + col;
    st_C = a.C[o];
    if (a.j > 0) {
      st_num = a.pnum[o];
      st_m = a.pm[rd * a.B + b0 + b];
      st_den = a.pden[rd * a.B + b0 + b];
    }
    if (a.last) {
      st_N = a.N[o];
      st_Z = a.Z[o];
      st_a = a.decay[col];
    }
  };
  if (!a.honly && (tid >> 7) < rows && (tid & 127) < cols) state(tid >> 7, first + (tid & 127));
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();  // x is there

  const int nprod = nslots + (a.honly ? 1 : a.last ? 3 : 2);
  for (int p = 0; p < nprod; ++p) {
    const int stage = p - nslots;  // < 0: q, k, v of slot p; 0: W_O; 1: W_g; 2: W_m
    if (stage == 0) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      if (a.parts > 1 && nslots == 0) tc::cluster_sync();  // the others' between parts
      tc::cluster_sync();  // every head's output is in Ah
    }
    if (stage == 1) {  // the pooling scores H w_p, a share of the columns per warp
      for (int bq = 0; bq < rows; bq += 4) {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        for (int c = 2 * tid; c < D; c += 2 * kDecThreads) {
          const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(wps + c));
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // (rows past the sequences are zero)
            const float2 h = __bfloat1622float2(
                *reinterpret_cast<const __nv_bfloat162*>(Ax + (bq + q) * lda + c));
            s[q] = fmaf(h.x, v.x, s[q]);
            s[q] = fmaf(h.y, v.y, s[q]);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] = warp_sum(s[q]);
        if (lane == 0)
          *reinterpret_cast<float4*>(sr + warp * kDecRows + bq) = make_float4(s[0], s[1], s[2], s[3]);
      }
    }
    const int sums = t.nks, wide = 8 * t.groups;
    dec_run<NT>(t, w, stage < 0 || stage == 1 ? Ax : Ah, lda, rows, red);
    if (p + 1 < nprod) {  // the next product's weights, ahead of this stage's barriers
      t = job(p + 1);
#pragma unroll
      for (int u = 0; u < kDecU; ++u) dec_step_fetch(t, t.s0 + u * t.nks, w[u]);
    }
    if (p == 0 && nslots > 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (stage < 0) {
      const int s = p, c0 = unit_col(s);
      float* dst = qkv + s * a.spc * 3 * pw;
      // q, k, v rounded to bf16; k and v to the cache's slot j
      dec_sums(red, sums, rows, wide, [&](int b, int c, float v) {
        const bf16 h = __float2bfloat16_rn(v);
        dst[b * 3 * pw + c] = __bfloat162float(h);
        const long o = ((long)(b0 + b) * a.L + a.j) * D + c0;
        if (c >= 2 * pw)
          a.Vc[o + c - 2 * pw] = h;
        else if (c >= pw)
          a.Kc[o + c - pw] = h;
      });
      __syncthreads();
      // attention: nw warps per sequence; pass k of warp wi takes the 32 keys from
      // 32 (k nw + wi), a lane per key for the scores and the softmax, then two of
      // the columns per lane (and two more, 64 on) for P V
      const int nw = a.nw, b = dec_div(warp, a.inv_nw), wi = warp - b * nw;
      const bool in = b < rows;
      const int part = (rank + s * ctas) & (a.parts - 1), step = lay.slots * a.spc * a.L;
      float* pr = sc + (s * a.spc + b) * a.L;
      const float* q = dst + b * 3 * pw;
      const long row0 = (long)(b0 + b) * a.L * D + c0;
      const int srow = (s * a.spc + b) * a.L;
      if (in) {
        auto score = [&](int u, float d) {
          float* to = pr + part * step + u;
          if (a.parts == 1)
            *to = d;
          else  // to every part's row of this part's shares
            for (int k = 0; k < a.parts; ++k)
              st_cluster_f(tc::mapa(tc::smem_u32(to), (uint32_t)(rank - part + k)), d);
        };
        for (int u0 = 32 * wi; u0 < n; u0 += 32 * nw) {
          const int u = u0 + lane;
          if (u < a.j)
            score(u, a.stage ? dec_dot(q, Ks + (srow + u) * (pw + 8), pw)
                             : dec_dot(q, a.Kc + row0 + (long)u * D, pw));
          if (a.j - u0 < 32 && a.j >= u0) {  // the new token's own key: lanes over columns
            float d = 0.f;
            for (int c = lane; c < pw; c += 32) d = fmaf(q[c], q[pw + c], d);
            d = warp_sum(d);
            if (lane == 0) score(a.j, d);
          }
        }
        __syncwarp();
      }
      if (a.parts > 1) tc::cluster_sync();  // (one slot per CTA then)
      float* mine = red + warp * (pw + 4);  // o, maximum, sum of the warp's keys
      if (in) {
        float mx = -INFINITY, sum = 0.f;
        for (int u = 32 * wi + lane; u < n; u += 32 * nw) {
          float v = pr[u];
          for (int k = 1; k < a.parts; ++k) v += pr[k * step + u];
          v *= a.scale;
          pr[u] = v;
          mx = fmaxf(mx, v);
        }
        mx = warp_max(mx);
        for (int u = 32 * wi + lane; u < n; u += 32 * nw) {
          const float e = expf(pr[u] - mx);
          pr[u] = e;
          sum += e;
        }
        sum = warp_sum(sum);
        __syncwarp();
        // a lane's two columns (and two more, 64 on): lanes past the part's width
        // repeat its last two
        const int ca = min(2 * lane, pw - 2), cb = min(64 + 2 * lane, pw - 2);
        float2 oa = make_float2(0.f, 0.f), ob = make_float2(0.f, 0.f);
        for (int u0 = 32 * wi; u0 < n; u0 += 32 * nw) {
          const int cnt = min(32, a.j - u0);  // cached keys of the pass
          if (a.stage)
            dec_pv(pr + u0, Vs + (srow + u0) * (pw + 8), pw + 8, cnt, ca, cb, oa, ob);
          else
            dec_pv(pr + u0, a.Vc + row0 + (long)u0 * D, D, cnt, ca, cb, oa, ob);
          if (a.j - u0 < 32 && a.j >= u0) {  // the new token's value
            const float e = pr[a.j];
            oa.x = fmaf(e, q[2 * pw + ca], oa.x);
            oa.y = fmaf(e, q[2 * pw + ca + 1], oa.y);
            ob.x = fmaf(e, q[2 * pw + cb], ob.x);
            ob.y = fmaf(e, q[2 * pw + cb + 1], ob.y);
          }
        }
        if (2 * lane < pw) *reinterpret_cast<float2*>(mine + 2 * lane) = oa;
        if (64 + 2 * lane < pw) *reinterpret_cast<float2*>(mine + 64 + 2 * lane) = ob;
        if (lane == 0) {
          mine[pw] = mx;
          mine[pw + 1] = sum;
        }
      }
      __syncthreads();
      // the warps of a sequence, in order (a warp without keys has weight 0)
      for (int bb = tid >> 7; bb < rows; bb += kDecThreads / 128) {
        const int c = tid & 127;
        if (c < pw) {
          const float* pw0 = red + bb * nw * (pw + 4);
          float m = -INFINITY, sum = 0.f, o = 0.f;
          for (int k = 0; k < nw; ++k) m = fmaxf(m, pw0[k * (pw + 4) + pw]);
          for (int k = 0; k < nw; ++k) {
            const float f = expf(pw0[k * (pw + 4) + pw] - m);
            sum = fmaf(f, pw0[k * (pw + 4) + pw + 1], sum);
            o = fmaf(f, pw0[k * (pw + 4) + c], o);
          }
          dst[bb * 3 * pw + c] = o / sum;
        }
      }
      __syncthreads();
      push(Ah, dst, 3 * pw, pw / 8, a.inv_per, c0);
    } else if (stage == 0) {
      if (a.honly) {
        dec_sums(red, sums, rows, wide, [&](int b, int c, float v) {
          a.y[(long)(b0 + b) * D + first + c] = __float2bfloat16_rn(v);
        });
      } else {
        dec_sums(red, sums, rows, wide, [&](int b, int c, float v) { out[b * lay.cols + c] = v; });
        __syncthreads();
        push(Ax, out, lay.cols, cols / 8, inv_mine, first);
        tc::cluster_sync();
      }
    } else if (stage == 1) {
      dec_sums(red, sums, rows, wide, [&](int b, int c, float u) {
        const int col = first + c;
        const long o = (long)(b0 + b) * D + col;
        if (b >= kDecThreads / 128 || c >= 128) state(b, col);  // else fetched at the start
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < kDecWarps; ++k) s += sr[k * kDecRows + b];
        const float m_old = a.j == 0 ? s : st_m;
        const float m_new = fmaxf(m_old, s);
        const float f_old = a.j == 0 ? 0.f : expf(m_old - m_new);
        const float e = expf(s - m_new);
        const float den = st_den * f_old + e;
        const float h = __bfloat162float(Ax[b * lda + col]);
        a.y[o] = __float2bfloat16_rn(fmaf(sigmoidf_(u), st_C, h));
        const float num = st_num * f_old + e * h;
        if (a.last) {
          const float nn = fmaf(st_a, st_N, num / den);
          const float z = fmaf(st_a, st_Z, 1.0f);
          a.N[o] = nn;
          a.Z[o] = z;
          out[b * lay.cols + c] = nn / z;
        } else {
          a.pnum[o] = num;
          if (col == 0) {
            a.pm[wr * a.B + b0 + b] = m_new;
            a.pden[wr * a.B + b0 + b] = den;
          }
        }
      });
      if (a.last) {
        __syncthreads();
        push(Ah, out, lay.cols, cols / 8, inv_mine, first);
        tc::cluster_sync();
      }
    } else {  // the next block's memory row
      dec_sums(red, sums, rows, wide, [&](int b, int c, float v) {
        a.C[(long)(b0 + b) * D + first + c] = v;
      });
    }
    __syncthreads();  // red is free
  }
}

// ---------------------------------------------------------------- host side
namespace {
template <class TW, int R>
cudaError_t gemv_r(const Launch& lc, const float* A, int M, int K, const void* W, int N, float* out,
                   bool round_out) {
  const int smem = 32 * R * 33 * (int)sizeof(float);
  static std::atomic<unsigned long long> opted{0};
  if (smem > 48 * 1024) {
    if (cudaError_t e = smem_opt_in(decode_gemv_kernel<TW, R>, smem, &opted); e != cudaSuccess)
      return e;
  }
  dim3 grid((N + 31) / 32, (M + R - 1) / R);
  cudaError_t e = launch_k(decode_gemv_kernel<TW, R>, grid, dim3(1024), smem, lc.stream, A, M, K,
                           (const TW*)W, N, out, round_out ? 1 : 0);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <class TW>
cudaError_t gemv(const Launch& lc, const float* A, int M, int K, const void* W, int N, float* out,
                 bool round_out) {
  if (M == 1) return gemv_r<TW, 1>(lc, A, M, K, W, N, out, round_out);
  if (M <= 4) return gemv_r<TW, 4>(lc, A, M, K, W, N, out, round_out);
  return gemv_r<TW, 16>(lc, A, M, K, W, N, out, round_out);
}

template <class T>
cudaError_t step_typed(const Launch& lc, const DecodeArgs& a) {
  const int B = a.B, D = a.D, j = a.j;
  cudaError_t e;
  if ((e = gemv<T>(lc, a.s.xf, B, D, a.w_qkv, 3 * D, a.s.qkv, false)) != cudaSuccess) return e;
  e = launch_k(decode_attn_kernel<T>, dim3(a.H, B), dim3(128), 0, lc.stream, (const float*)a.s.qkv,
               (T*)a.s.Kc, (T*)a.s.Vc, a.s.hhat, D, a.dh, a.L, j, 1.0f / sqrtf((float)a.dh));
  if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = gemv<T>(lc, a.s.hhat, B, D, a.w_o, D, a.s.H, true)) != cudaSuccess) return e;
  if (!a.honly && (e = gemv<T>(lc, a.s.H, B, D, a.w_g, D, a.s.U, false)) != cudaSuccess) return e;
  const int last = (j == a.L - 1) ? 1 : 0;
  e = launch_k(decode_post_kernel<T>, dim3(B), dim3(256), 0, lc.stream, (const float*)a.s.H,
               (const float*)a.s.U, (const T*)a.w_p, a.decay, a.s.C, a.s.pm, a.s.pden, a.s.pnum,
               a.s.N, a.s.Z, a.s.Mr, (T*)a.y, D, j, last, a.honly ? 1 : 0);
  if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
  // the next block's memory row C_{i+1} = M_i W_m
  if (last && !a.honly) return gemv<T>(lc, a.s.Mr, B, D, a.w_m, D, a.s.C, false);
  return cudaSuccess;
}
}  // namespace


// The token's input row is taken as fp32 by the first product; copy (and
// widen) x_t into the state's fp32 row.
template <class T>
__global__ void __launch_bounds__(256) decode_widen_kernel(const T* __restrict__ x, float* out,
                                                           long n) {
  pdl_enter();
  x = after_wait(x);
  for (long i = blockIdx.x * 256L + threadIdx.x; i < n; i += (long)gridDim.x * 256)
    out[i] = to_f(x[i]);
}

static cudaError_t decode_widen(const Launch& lc, int dtype, const void* x, float* out, long n) {
  const int blocks = (int)std::min<long>((n + 255) / 256, 1024);
  cudaError_t e = dtype == 0 ? launch_k(decode_widen_kernel<float>, dim3(blocks), dim3(256), 0,
                                        lc.stream, (const float*)x, out, n)
                             : launch_k(decode_widen_kernel<bf16>, dim3(blocks), dim3(256), 0,
                                        lc.stream, (const bf16*)x, out, n);
  return e != cudaSuccess ? e : cudaGetLastError();
}

namespace {
// CTAs per cluster and clusters at a time that this device runs the one-launch
// step with (16 CTAs where a GPC has them, else the portable 8; 0: neither),
// looked up once per device.
struct DecodeFit {
  int ctas, clusters;
};
template <int NT>
DecodeFit decode_fit() {
  static std::atomic<int> known[64];  // 0: not yet, else 1 + 64 * ctas + clusters
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return {0, 0};
  int v = known[dev].load();
  if (!v) {
    DecodeFit f{0, 0};
    if (cudaFuncSetAttribute(decode_cluster_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kDecSmem) == cudaSuccess &&
        cudaFuncSetAttribute(decode_cluster_kernel<NT>,
                             cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      for (int ctas = 16; ctas >= 8 && !f.ctas; ctas /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(kDecThreads);
        cfg.dynamicSmemBytes = kDecSmem;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = ctas;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, decode_cluster_kernel<NT>, &cfg) == cudaSuccess && n > 0)
          f = {ctas, std::min(n, 63)};
      }
    }
    cudaGetLastError();  // an attribute this device refuses is no launch error
    v = 1 + 64 * f.ctas + f.clusters;
    known[dev].store(v);
  }
  return {(v - 1) / 64, (v - 1) % 64};
}

// Sizes that fit one launch and are faster as a launch per stage, which has all SMs at
// work (us a token, staged and one launch, in the last quarter of a block):
//   one sequence of a wide layer, whose weights one cluster's SMs have to bring alone:
//     D = 1280 27 and 37 (L 16), 31 and 37 (L 64), 46 and 42 (L 256); 2048 43 and 51, 47 and
//     51, 63 and 56; from two sequences on the other way round (D = 1280 41 and 37, L 16);
//   many sequences of a narrow layer, sixteen to a cluster: B = 64, D = 64 23 and 24 (L 16),
//     44 and 40 (L 256); D = 256 24 and 27, 46 and 43; at B = 48 24 and 23 (D = 256, L 16), at
//     D = 384 37 and 28;
//   more sequences than the clusters that run at a time hold (seven, 112 sequences):
//     B = 128, D = 128 24 and 50 (L 16), D = 512 52 and 57, D = 640 100 and 66.
bool staged_is_faster(const DecodeArgs& a, int clusters) {
  if (a.B == 1) return a.D > 1024 && a.L < 256;
  if (a.B > kDecRows * clusters) return a.D < 640;
  return a.B > 48 && a.D < 384 && a.L < 256;
}

// The whole step in one launch; cudaErrorNotSupported for shapes whose rows do
// not fit a CTA's shared memory, and for those above.
template <int NT>
cudaError_t step_cluster(const Launch& lc, const DecodeArgs& a) {
  const DecodeFit fit = decode_fit<NT>();
  if (!fit.ctas) return cudaErrorNotSupported;
  if (g_decode_one_launch == 1 && staged_is_faster(a, fit.clusters)) return cudaErrorNotSupported;
  // sequences per cluster: over up to kDecClusters clusters, at most kDecRows each
  int ncl = std::min(a.B, std::min(fit.clusters, kDecClusters));
  if (a.B > ncl * kDecRows) ncl = (a.B + kDecRows - 1) / kDecRows;
  const int spc = (a.B + ncl - 1) / ncl;
  if (NT == 1 && spc > 8) return step_cluster<2>(lc, a);
  // fewer heads than CTAs: parts of eight columns or more share a head
  int parts = 1;
  while (a.H * parts * 2 <= fit.ctas && a.dh % (parts * 16) == 0) parts *= 2;
  DecodeClusterSmem sm = dec_smem(a.D, a.H, a.dh, a.L, parts, spc, fit.ctas, 1);
  const bool stage = sm.bytes <= kDecSmem && sm.bytes - sm.kv <= kDecStage;
  if (!stage) sm = dec_smem(a.D, a.H, a.dh, a.L, parts, spc, fit.ctas, 0);
  // (the product's column chunks also have to leave every warp a share of K)
  if (sm.bytes > kDecSmem || sm.cols > 64 * kDecWarps) return cudaErrorNotSupported;
  DecodeClusterArgs k;
  k.x = (const bf16*)a.x_t;
  k.w_qkv = (const bf16*)a.w_qkv;
  k.w_o = (const bf16*)a.w_o;
  k.w_p = (const bf16*)a.w_p;
  k.w_m = (const bf16*)a.w_m;
  k.w_g = (const bf16*)a.w_g;
  k.decay = a.decay;
  k.y = (bf16*)a.y;
  k.Kc = (bf16*)a.s.Kc;
  k.Vc = (bf16*)a.s.Vc;
  k.pm = a.s.pm;
  k.pden = a.s.pden;
  k.pnum = a.s.pnum;
  k.N = a.s.N;
  k.Z = a.s.Z;
  k.C = a.s.C;
  k.B = a.B;
  k.D = a.D;
  k.heads = a.H;
  k.dh = a.dh;
  k.L = a.L;
  k.j = a.j;
  k.honly = a.honly ? 1 : 0;
  k.last = a.j == a.L - 1 ? 1 : 0;
  k.spc = spc;
  k.parts = parts;
  k.stage = stage ? 1 : 0;
  k.sm = sm;
  for (k.lparts = 0; (1 << k.lparts) < parts;) ++k.lparts;
  k.nch_q = (3 * sm.pw / 8 + 7) / 8;
  k.nch_c = (sm.cols / 8 + 7) / 8;
  k.nks_q = kDecWarps / k.nch_q;
  k.nks_c = kDecWarps / k.nch_c;
  k.nw = kDecWarps / spc;
  k.inv_q = dec_inv(k.nch_q);
  k.inv_c = dec_inv(k.nch_c);
  k.inv_per = dec_inv(sm.pw / 8);
  k.inv_nw = dec_inv(k.nw);
  k.inv_cols = dec_inv(sm.cols / 8);
  k.scale = 1.0f / sqrtf((float)a.dh);
  cudaError_t e = launch_k_cluster(decode_cluster_kernel<NT>, dim3((a.B + spc - 1) / spc * fit.ctas),
                                   dim3(kDecThreads), sm.bytes, lc.stream, fit.ctas, k);
  return e != cudaSuccess ? e : cudaGetLastError();
}
}  // namespace

// bf16: one launch (step_cluster) where the shape fits it; fp32 (whose products
// are fp32 multiply-adds) and the rest: a launch per stage.
cudaError_t decode_step(const Launch& lc, int dtype, const DecodeArgs& a) {
  if (a.L > kMaxL || a.dh > 128) return cudaErrorInvalidValue;
  if (dtype == 1 && g_decode_one_launch != 0) {
    const cudaError_t e = step_cluster<1>(lc, a);
    if (e != cudaErrorNotSupported) return e;
  }
  const cudaError_t e = decode_widen(lc, dtype, a.x_t, a.s.xf, (long)a.B * a.D);
  if (e != cudaSuccess) return e;
  return dtype == 0 ? step_typed<float>(lc, a) : step_typed<bf16>(lc, a);
}

}  // namespace bcmt
