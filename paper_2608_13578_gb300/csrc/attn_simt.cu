// Intra-block causal multi-head attention on CUDA cores (Sec. 3.3): forward and
// backward of fp32 tensors (true fp32 arithmetic throughout), the forward of
// the bf16 shapes that attn_tc.cu and attn_flash.cu do not take, the backward
// that allocates nothing, and every bf16 shape when the tensor-core kernels are
// switched off.
//
// One CTA of 256 threads (16 x 16) per 64-token tile of one head.  For L <= 64 a
// tile holds the 64 / L whole blocks that fit and is its own key tile; for
// L > 64 it is up to 64 rows of one block and walks the block's tiles.  Tiles lie
// in shared memory as fp32 rows padded by 4 (the 8 rows that a quarter-warp's
// 16-byte loads touch fall in distinct banks).  A thread holds a 4 x 4 block of
// scores (rows 4 ty .. +3, columns tx + 16 j): 64 multiply-adds for every eight
// 16-byte loads.  In the products over keys or queries it holds four columns
// (twice four for heads above 64) of one, two or four rows, so that all threads
// have outputs at every head width, and skips what the causal mask hides from
// its rows.  Long walks start first: in tile order the last wave held half of them
// (16 % of the SMs' time at L 128).  Bound: no single unit (issue 0.55 a cycle, FMA
// 32 %, shared memory 44 %); two or three CTAs of eight warps hide little of the
// loads, barriers and exponentials between the products.  Forward: three CTAs per
// SM for heads up to 64 (80 registers), two above (shared memory).  Before, one warp
// per query row read every key row from L2; times before and now: B8 T1024 D512 h8
// L64 fp32 forward 516 and 48 us, backward 2002 and 92 us; B4 T2048 D1024 h8 L128
// bf16 forward 1997 and 126 us; B4 T1000 D768 h8 L48 bf16 forward 306 and 63 us.
// Deterministic: every sum runs in a fixed order.
#include <limits.h>

#include <algorithm>

#include "attn_slow.cuh"
#include "common.cuh"
#include "internal.h"

namespace bcmt {

namespace {
constexpr int kMaxL = 1024;   // longest block
constexpr int kMaxDh = 128;   // widest head
constexpr int kTile = 64;
constexpr int kThreads = 256;
constexpr int kPld = kTile + 4;  // row stride of a score tile

template <class E>
struct SimtArgs {
  AttnPtrs<E> x;
  E *Out, *dQ, *dK, *dV;
  long ld_d;
  float *lse, *Drow;
  int rows;  // L <= 64: rows per tile (whole blocks)
  int tpb;   // L > 64: tiles per block
  int nb, B; // tiles (L <= 64) or blocks of a sequence, sequences
  int vec;   // rows of every tensor are aligned to four elements
};

struct TileAt {
  int t0, rows, kstart, j, h, b;
};
// Blocks first, heads of one block as neighbours; tiles of a long block by the key
// (or query) tiles they walk, the longest walks of the whole grid first, so that
// the last CTAs to run are short ones (DESC: tile j walks j + 1 of them).
template <bool DESC, class E>
__device__ __forceinline__ TileAt tile_at(const SimtArgs<E>& a) {
  TileAt t;
  int x = blockIdx.x / a.x.H;
  t.h = blockIdx.x - x * a.x.H;
  const int n = x / a.nb;
  x -= n * a.nb;
  const int jj = n / a.B;
  t.b = n - jj * a.B;
  if (a.x.L <= kTile) {
    t.t0 = t.kstart = x * a.rows;
    t.j = 0;
    t.rows = min(a.rows, a.x.T - t.t0);
  } else {
    t.j = DESC ? a.tpb - 1 - jj : jj;
    t.kstart = x * a.x.L;
    t.t0 = t.kstart + t.j * kTile;
    t.rows = min(min(kTile, a.x.L - t.j * kTile), a.x.T - t.t0);
  }
  return t;
}

// The 16-key groups [j0, j0 + n) of a score tile that any of the warp's eight rows
// sees.  Heads up to 64 (CB = 1) form all four: there the shorter loops do not make
// up for four copies of the code (B8 T1024 D512 h8 L64 fp32 forward 46 us, 51 with
// them; backward 90 and 95), above they do (heads of 96, L 48: 169 -> 153 us for 16 x
// 1000 tokens; heads of 128, L 128, 113 -> 109 us for 4 x 2048).
struct Groups {
  int j0, n;
};
template <int CB>
__device__ __forceinline__ Groups groups_seen(bool diag, int rows, int L) {
  const int r0 = 8 * (threadIdx.x >> 5);
  if (CB == 1) return {0, 4};
  if (r0 >= rows) return {0, 0};
  if (!diag) return {0, 4};
  const int j0 = L <= kTile ? (r0 / L) * L / 16 : 0;
  return {j0, min(r0 + 7, rows - 1) / 16 + 1 - j0};
}
// f(N) for n groups, N a compile-time count.
template <int CB, class F>
__device__ __forceinline__ void with_groups(int n, F&& f) {
  using std::integral_constant;
  if (CB == 1 || n == 4) f(integral_constant<int, 4>());
  else if (n == 3) f(integral_constant<int, 3>());
  else if (n == 2) f(integral_constant<int, 2>());
  else if (n == 1) f(integral_constant<int, 1>());
}

// Rows [0, rows) x dh columns of a head into a tile, the other rows zero; a
// thread's loads of four rows go out together.
template <class E>
__device__ __forceinline__ void fill(float* dst, int ldh, const E* src, long ld, int rows, int dh,
                                     bool vec) {
  const int r0 = threadIdx.x >> 4;
  for (int c = (threadIdx.x & 15) * 4; c < dh; c += 64) {
    float v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + 16 * u;
#pragma unroll
      for (int e = 0; e < 4; ++e) v[u][e] = 0.f;
      if (r < rows) {
        const E* p = src + (long)r * ld + c;
        if (vec) {
          load4(p, v[u]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) v[u][e] = to_f(p[e]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      *reinterpret_cast<float4*>(dst + (r0 + 16 * u) * ldh + c) =
          make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
  }
}
template <class E>
__device__ __forceinline__ void put4(E* p, const float* v, bool vec) {
  if (vec) {
    store4(p, v);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) p[e] = from_f<E>(v[e]);
  }
}

// s[i][j] = A[4 ty + i] . B[tx + 16 j], j < N, over dh columns, each a single chain
// in column order.
template <int N>
__device__ __forceinline__ void scores_in_order(const float* A, const float* B, int ldh, int dh,
                                                float (*s)[4]) {
  const float* pa = A + 4 * (threadIdx.x >> 4) * ldh;
  const float* pb = B + (threadIdx.x & 15) * ldh;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) s[i][j] = 0.f;
#pragma unroll 2
  for (int k = 0; k < dh; k += 4) {
    float4 x[4], y[N];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4*>(pa + i * ldh + k);
#pragma unroll
    for (int j = 0; j < N; ++j) y[j] = *reinterpret_cast<const float4*>(pb + 16 * j * ldh + k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) {
        s[i][j] = fmaf(x[i].x, y[j].x, s[i][j]);
        s[i][j] = fmaf(x[i].y, y[j].y, s[i][j]);
        s[i][j] = fmaf(x[i].z, y[j].z, s[i][j]);
        s[i][j] = fmaf(x[i].w, y[j].w, s[i][j]);
      }
  }
}

// The same with two chains per score (even and odd columns), as packed pairs.
template <int N>
__device__ __forceinline__ void scores(const float* A, const float* B, int ldh, int dh,
                                       float (*s)[4]) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  float2 acc[4][N];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const float* pa = A + (4 * ty) * ldh;
  const float* pb = B + tx * ldh;
#pragma unroll 2
  for (int k = 0; k < dh; k += 4) {
    float4 x[4], y[N];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4*>(pa + i * ldh + k);
#pragma unroll
    for (int j = 0; j < N; ++j) y[j] = *reinterpret_cast<const float4*>(pb + 16 * j * ldh + k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) {
        acc[i][j] = __ffma2_rn(make_float2(x[i].x, x[i].y), make_float2(y[j].x, y[j].y), acc[i][j]);
        acc[i][j] = __ffma2_rn(make_float2(x[i].z, x[i].w), make_float2(y[j].z, y[j].w), acc[i][j]);
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) s[i][j] = acc[i][j].x + acc[i][j].y;
}

// The thread's outputs: column group threadIdx.x % C4 (four columns, CB times 64
// apart) of RT consecutive rows; 64 rows x C4 groups over 256 threads.
template <int C4, int CB>
struct Cols {
  static constexpr int RT = C4 / 4;
  __device__ __forceinline__ static int col() { return (threadIdx.x & (C4 - 1)) * 4; }
  __device__ __forceinline__ static int row() { return (threadIdx.x / C4) * RT; }
};

// acc[i] += sum over keys j in [lo, hi), in order, of P[row + i][j] B[j - b0], four
// keys at a time: the range is widened to multiples of four, where P is 0 (hidden
// keys) and B has its zero rows.
template <int C4, int CB>
__device__ __forceinline__ void rows_times(const float* P, int ldp, const float* B, int ldh, int dh,
                                           int lo, int hi, int b0, float (*acc)[CB][4]) {
  using C = Cols<C4, CB>;
  const float* p = P + C::row() * ldp;
  const int c = C::col();
  if (c >= dh) return;
#pragma unroll 2
  for (int j = lo & ~3; j < hi; j += 4) {
    float w[C::RT][4];
#pragma unroll
    for (int i = 0; i < C::RT; ++i) {
      const float4 x = *reinterpret_cast<const float4*>(p + i * ldp + j);
      w[i][0] = x.x; w[i][1] = x.y; w[i][2] = x.z; w[i][3] = x.w;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int m = 0; m < CB; ++m)
        if (m == 0 || c + 64 * m < dh) {
          const float4 v = *reinterpret_cast<const float4*>(B + (j + q - b0) * ldh + c + 64 * m);
#pragma unroll
          for (int i = 0; i < C::RT; ++i) {
            acc[i][m][0] = fmaf(w[i][q], v.x, acc[i][m][0]);
            acc[i][m][1] = fmaf(w[i][q], v.y, acc[i][m][1]);
            acc[i][m][2] = fmaf(w[i][q], v.z, acc[i][m][2]);
            acc[i][m][3] = fmaf(w[i][q], v.w, acc[i][m][3]);
          }
        }
  }
}
// acc[i] += sum over queries r in [lo, hi) of P[r][row + i] B[r].
template <int C4, int CB>
__device__ __forceinline__ void cols_times(const float* P, const float* B, int ldh, int dh, int lo,
                                           int hi, float (*acc)[CB][4]) {
  using C = Cols<C4, CB>;
  const float* p = P + C::row();
  const int c = C::col();
  if (c >= dh) return;
#pragma unroll 4
  for (int r = lo; r < hi; ++r) {
    float w[C::RT];
    if (C::RT == 4) {
      const float4 x = *reinterpret_cast<const float4*>(p + r * kPld);
      w[0] = x.x; w[C::RT > 1 ? 1 : 0] = x.y; w[C::RT > 2 ? 2 : 0] = x.z; w[C::RT > 3 ? 3 : 0] = x.w;
    } else {
#pragma unroll
      for (int i = 0; i < C::RT; ++i) w[i] = p[r * kPld + i];
    }
#pragma unroll
    for (int m = 0; m < CB; ++m)
      if (m == 0 || c + 64 * m < dh) {
        const float4 v = *reinterpret_cast<const float4*>(B + r * ldh + c + 64 * m);
#pragma unroll
        for (int i = 0; i < C::RT; ++i) {
          acc[i][m][0] = fmaf(w[i], v.x, acc[i][m][0]);
          acc[i][m][1] = fmaf(w[i], v.y, acc[i][m][1]);
          acc[i][m][2] = fmaf(w[i], v.z, acc[i][m][2]);
          acc[i][m][3] = fmaf(w[i], v.w, acc[i][m][3]);
        }
      }
  }
}
template <int RT, int CB>
__device__ __forceinline__ void zero(float (*acc)[CB][4]) {
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int m = 0; m < CB; ++m)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][m][e] = 0.f;
}
__device__ __forceinline__ bool finite4(const float* v) {
  return is_finite(v[0]) && is_finite(v[1]) && is_finite(v[2]) && is_finite(v[3]);
}
// sum over the 16 threads of a row group
__device__ __forceinline__ float sum16(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float max16(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// First row of the block that row r of a tile belongs to (0 for L > 64: the
// tile's whole walk is one block).
__device__ __forceinline__ int block_row(int r, int L) { return L <= kTile ? (r / L) * L : 0; }
__device__ __forceinline__ int block_end(int r, int L) {
  return L <= kTile ? min((r / L) * L + L, kTile) : kTile;
}
}  // namespace

namespace {
// The groups of four columns that came out non-finite, formed again row by row; bit
// i * CB + m of bad: the thread's row i, column block m.
template <int C4, int CB, class S>
__device__ __forceinline__ void mark_bad(S&& set, int row0, unsigned bad) {
  using C = Cols<C4, CB>;
  for (int n = 0; n < C::RT * CB; ++n)
    if (bad >> n & 1u) set(row0 + C::row() + n / CB, C::col() / 4 + 16 * (n % CB));
}
template <class E>
__device__ __forceinline__ void put_groups(E* p, const SlowRow& r, unsigned groups, int dh) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int c = (threadIdx.x & 31) + 32 * i;
    if (c < dh && (groups >> (c / 4) & 1u)) p[c] = from_f<E>(r.v[i]);
  }
}
template <class E, int C4, int CB>
__device__ __noinline__ void redo_o(const SimtArgs<E>& a, TileAt tt, float* sm, unsigned bad) {
  E* out = a.Out + ((long)tt.b * a.x.T + tt.t0) * a.x.ld_o + tt.h * a.x.dh;
  slow_rows<kTile>(sm, [&](auto set) { mark_bad<C4, CB>(set, 0, bad); },
                   [&](int r, unsigned groups, float* w) {
    SlowRow o;
    slow_o(a.x, tt.b, tt.h, tt.t0 + r, w, o);
    put_groups(out + r * a.x.ld_o, o, groups, a.x.dh);
  });
}
template <class E, int C4, int CB>
__device__ __noinline__ void redo_dq(const SimtArgs<E>& a, TileAt tt, float* sm, unsigned bad) {
  E* out = a.dQ + ((long)tt.b * a.x.T + tt.t0) * a.ld_d + tt.h * a.x.dh;
  slow_rows<kTile>(sm, [&](auto set) { mark_bad<C4, CB>(set, 0, bad); },
                   [&](int r, unsigned groups, float* w) {
    SlowRow dq;
    slow_dq(a.x, tt.b, tt.h, tt.t0 + r, w, dq);
    put_groups(out + r * a.ld_d, dq, groups, a.x.dh);
  });
}
template <class E, int C4, int CB>
__device__ __noinline__ void redo_dkv(const SimtArgs<E>& a, TileAt tt, float* sm,
                                      unsigned badk, unsigned badv) {
  const long o = ((long)tt.b * a.x.T + tt.t0) * a.ld_d + tt.h * a.x.dh;
  slow_rows<2 * kTile>(sm, [&](auto set) {
    mark_bad<C4, CB>(set, 0, badk);
    mark_bad<C4, CB>(set, kTile, badv);
  }, [&](int n, unsigned groups, float* w) {
    const int r = n & (kTile - 1);
    SlowRow d;
    if (n < kTile)
      slow_dkv<false>(a.x, tt.b, tt.h, tt.t0 + r, w, d);
    else
      slow_dkv<true>(a.x, tt.b, tt.h, tt.t0 + r, w, d);
    put_groups((n < kTile ? a.dK : a.dV) + o + r * a.ld_d, d, groups, a.x.dh);
  });
}
}  // namespace

// O[t] = sum_j softmax_j(q_t . k_j * scale) v_j over keys j in [blockstart(t), t].
//
// The arithmetic and its order are those of one query at a time -- a score is
// one chain of fused multiply-adds over the columns, the largest score of the
// whole row is subtracted before any exponential, the sum runs in 32 interleaved
// partials joined by a butterfly, the output is one chain over the keys -- so
// the result does not depend on the tiling.  (A bf16 layer rounds O, H and the
// gate to bf16 in turn: a last-bit difference here would move every later
// rounding, the fp32 decay gradient among the results.)  Hence two phases: all
// of the row's scores, kept in shared memory for up to kKeep key tiles (beyond
// that they are formed twice), then exponentials, sum and output.  share: K and V
// take turns in one buffer, where that makes room for a second CTA on the SM.
constexpr int kKeep = 4;
template <class E, int C4, int CB>
__global__ void __launch_bounds__(kThreads, CB == 1 ? 3 : 2)
    attn_fwd_simt_kernel(const __grid_constant__ SimtArgs<E> a, int ldp, int share) {
  pdl_enter();
  using C = Cols<C4, CB>;
  extern __shared__ __align__(16) float sm[];
  const int dh = a.x.dh, ldh = dh + 4;
  float *Qs = sm, *Ks = Qs + kTile * ldh, *Vs = share ? Ks : Ks + kTile * ldh,
        *Ps = Vs + kTile * ldh, *inv = Ps + kTile * ldp;  // inv: [64]
  const int tid = threadIdx.x, ty = threadIdx.x >> 4, tx = tid & 15;
  const TileAt tt = tile_at<true>(a);
  const int h = tt.h, b = tt.b;
  if (tt.rows <= 0) return;
  const long row0 = (long)b * a.x.T;
  const int c0 = h * dh;
  const bool keep = ldp > kPld || tt.j == 0;
  auto keys = [&](int kt) { return kt == tt.j ? tt.rows : kTile; };
  auto load_tile = [&](float* dst, const E* src, int kt) {
    fill(dst, ldh, src + (row0 + tt.kstart + kt * kTile) * a.x.ld + c0, a.x.ld, keys(kt), dh, a.vec);
  };
  // the thread's scaled scores of N groups of key tile kt (hidden keys -inf)
  auto tile_scores = [&](auto n, int j0, int kt, float (*s)[4]) {
    constexpr int N = decltype(n)::value;
    scores_in_order<N>(Qs, Ks + 16 * j0 * ldh, ldh, dh, s);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = 4 * ty + i, rbs = block_row(r, a.x.L);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int k = tx + 16 * (j0 + j);
        s[i][j] = (kt < tt.j || (k >= rbs && k <= r)) ? __fmul_rn(s[i][j], a.x.scale) : -INFINITY;
      }
    }
  };
  fill(Qs, ldh, a.x.Q + (row0 + tt.t0) * a.x.ld + c0, a.x.ld, tt.rows, dh, a.vec);
  if (!share) load_tile(Vs, a.x.V, 0);
  float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
  for (int kt = 0; kt <= tt.j; ++kt) {
    if (kt > 0) __syncthreads();
    load_tile(Ks, a.x.K, kt);
    __syncthreads();
    const Groups g = groups_seen<CB>(kt == tt.j, tt.rows, a.x.L);
    with_groups<CB>(g.n, [&](auto n) {
      float s[4][4];
      tile_scores(n, g.j0, kt, s);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < decltype(n)::value; ++j) {
          mx[i] = fmaxf(mx[i], s[i][j]);
          if (keep) Ps[(4 * ty + i) * ldp + kt * kTile + tx + 16 * (g.j0 + j)] = s[i][j];
        }
    });
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) mx[i] = max16(mx[i]);

  // exponentials of key tile kt into columns p0 .. of Ps (groups that no row of the
  // warp sees are neither written nor read)
  auto exps = [&](int kt, int p0) {
    const Groups g = groups_seen<CB>(kt == tt.j, tt.rows, a.x.L);
    with_groups<CB>(g.n, [&](auto n) {
      float s[4][4];
      if (!keep) tile_scores(n, g.j0, kt, s);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < decltype(n)::value; ++j) {
          float* p = Ps + (4 * ty + i) * ldp + p0 + tx + 16 * (g.j0 + j);
          *p = expf((keep ? *p : s[i][j]) - mx[i]);
        }
    });
  };
  if (keep)
    for (int kt = 0; kt <= tt.j; ++kt) exps(kt, kt * kTile);
  float acc[C::RT][CB][4], part[8];
  zero<C::RT, CB>(acc);
#pragma unroll
  for (int u = 0; u < 8; ++u) part[u] = 0.f;
  const int warp = tid >> 5, lane = tid & 31;
  for (int kt = 0; kt <= tt.j; ++kt) {
    const int p0 = keep ? kt * kTile : 0;
    __syncthreads();  // keep: the probabilities are written; else the last tile is used up
    if (!keep) {
      load_tile(Ks, a.x.K, kt);
      if (!share) load_tile(Vs, a.x.V, kt);
      __syncthreads();
      exps(kt, 0);
      __syncthreads();
      if (share) {
        load_tile(Vs, a.x.V, kt);
        __syncthreads();
      }
    } else if (share || kt > 0) {
      load_tile(Vs, a.x.V, kt);
      __syncthreads();
    }
    // partial sums of the warp's eight rows, lane = key index in the block mod 32
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int r = 8 * warp + u, rbs = block_row(r, a.x.L);
      const int n = r >= tt.rows ? 0 : kt < tt.j ? kTile : r + 1 - rbs;  // visible keys of this tile
      for (int j = lane; j < n; j += 32) part[u] += Ps[r * ldp + p0 + rbs + j];
    }
    rows_times<C4, CB>(Ps, ldp, Vs, ldh, dh, p0 + (kt < tt.j ? 0 : block_row(C::row(), a.x.L)),
                       p0 + (C::row() >= tt.rows ? 0 : kt < tt.j ? kTile : min(C::row() + C::RT, tt.rows)),
                       p0, acc);
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    part[u] = warp_sum(part[u]);
    if (lane == u) inv[8 * warp + u] = part[u];
  }
  __syncthreads();
  if (tx < 4 && 4 * ty + tx < tt.rows) {
    const int r = 4 * ty + tx;
    const float m = tx == 0 ? mx[0] : tx == 1 ? mx[1] : tx == 2 ? mx[2] : mx[3];
    a.lse[((long)b * a.x.H + h) * a.x.T + tt.t0 + r] = m + logf(inv[r]);
  }
  const int c = C::col();
  unsigned bad = 0u;
#pragma unroll
  for (int i = 0; i < C::RT; ++i) {
    const int r = C::row() + i, t = tt.t0 + r;
    if (r >= tt.rows) break;
    const float in = 1.0f / inv[r];
#pragma unroll
    for (int m = 0; m < CB; ++m)
      if (c + 64 * m < dh) {
        float* v = acc[i][m];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] *= in;
        if (!finite4(v)) bad |= 1u << (i * CB + m);
        put4(a.Out + (row0 + t) * a.x.ld_o + c0 + c + 64 * m, v, true);
      }
  }
  if (__syncthreads_or(bad)) redo_o<E, C4, CB>(a, tt, sm, bad);
}

namespace {
// Drow of the thread's four rows, from the tensors: the 16 threads of a row
// group share a row's columns.
template <class E>
__device__ __forceinline__ void drow4(const SimtArgs<E>& a, int b, int h, int t0, int rows,
                                      float* d) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = 4 * ty + i;
    float s = 0.f;
    if (r < rows) {
      const long o = ((long)b * a.x.T + t0 + r) * a.x.ld_o + h * a.x.dh;
      for (int c = 4 * tx; c < a.x.dh; c += 64) {
        float u[4], v[4];
        load4(a.x.dO + o + c, u);
        load4(a.x.O + o + c, v);
#pragma unroll
        for (int e = 0; e < 4; ++e) s = fmaf(u[e], v[e], s);
      }
    }
    d[i] = sum16(s);
  }
}
// P and dS = P (dP - Drow) scale of the thread's rows into score tiles (P may be
// null), rows past `rows` and hidden keys 0; groups that no row of the warp sees are
// neither written nor read.
template <int CB, class E>
__device__ __forceinline__ void p_ds(const SimtArgs<E>& a, const float* Qs, const float* Ks,
                                     const float* Gs, const float* Vs, int ldh, bool diag, int rows,
                                     const float* lse, const float* drow, float* P, float* S) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  const Groups g = groups_seen<CB>(diag, rows, a.x.L);
  with_groups<CB>(g.n, [&](auto n) {
    constexpr int N = decltype(n)::value;
    float p[4][4], ds[4][4];
    scores<N>(Qs, Ks + 16 * g.j0 * ldh, ldh, a.x.dh, p);
    scores<N>(Gs, Vs + 16 * g.j0 * ldh, ldh, a.x.dh, ds);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = 4 * ty + i, rbs = block_row(r, a.x.L);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int k = tx + 16 * (g.j0 + j);
        const bool vis = r < rows && (!diag || (k >= rbs && k <= r));
        p[i][j] = vis ? expf(p[i][j] * a.x.scale - lse[i]) : 0.f;
        ds[i][j] = vis ? p[i][j] * (ds[i][j] - drow[i]) * a.x.scale : 0.f;
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int o = (4 * ty + i) * kPld + tx + 16 * (g.j0 + j);
        if (P) P[o] = p[i][j];
        S[o] = ds[i][j];
      }
  });
}
template <class E>
__device__ __forceinline__ void rows_lse(const SimtArgs<E>& a, int b, int h, int t0, int rows,
                                         const float* src, float* v) {
  const int ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    v[i] = 4 * ty + i < rows ? src[((long)b * a.x.H + h) * a.x.T + t0 + 4 * ty + i] : 0.f;
}
// Stores the thread's dQ; the groups that are not finite (as `bad` above).
template <class E, int C4, int CB>
__device__ __forceinline__ unsigned store_dq(const SimtArgs<E>& a, const TileAt& tt, int b, int h,
                                             float (*acc)[CB][4]) {
  using C = Cols<C4, CB>;
  const int c = C::col();
  unsigned bad = 0u;
#pragma unroll
  for (int i = 0; i < C::RT; ++i) {
    const int r = C::row() + i, t = tt.t0 + r;
    if (r >= tt.rows) break;
#pragma unroll
    for (int m = 0; m < CB; ++m)
      if (c + 64 * m < a.x.dh) {
        if (!finite4(acc[i][m])) bad |= 1u << (i * CB + m);
        put4(a.dQ + ((long)b * a.x.T + t) * a.ld_d + h * a.x.dh + c + 64 * m, acc[i][m], a.vec);
      }
  }
  return bad;
}
}  // namespace

// L > 64, per query tile: Drow_t = dO_t . O_t, and
// dQ_t = scale * sum_j P_tj (dO_t . v_j - Drow_t) k_j over the block's key tiles.
template <class E, int C4, int CB>
__global__ void __launch_bounds__(kThreads, CB == 1 ? 2 : 1)
    attn_bwd_q_simt_kernel(const __grid_constant__ SimtArgs<E> a) {
  pdl_enter();
  extern __shared__ __align__(16) float sm[];
  const int dh = a.x.dh, ldh = dh + 4;
  float *Qs = sm, *Gs = Qs + kTile * ldh, *Ks = Gs + kTile * ldh, *Vs = Ks + kTile * ldh,
        *Ss = Vs + kTile * ldh;
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  const TileAt tt = tile_at<true>(a);
  const int h = tt.h, b = tt.b;
  if (tt.rows <= 0) return;
  const long row0 = (long)b * a.x.T;
  const int c0 = h * dh;
  fill(Qs, ldh, a.x.Q + (row0 + tt.t0) * a.x.ld + c0, a.x.ld, tt.rows, dh, a.vec);
  fill(Gs, ldh, a.x.dO + (row0 + tt.t0) * a.x.ld_o + c0, a.x.ld_o, tt.rows, dh, true);
  using C = Cols<C4, CB>;
  float drow[4], lse[4], acc[C::RT][CB][4];
  drow4(a, b, h, tt.t0, tt.rows, drow);
  rows_lse(a, b, h, tt.t0, tt.rows, a.lse, lse);
  if (tx == 0 && a.Drow) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (4 * ty + i < tt.rows)
        a.Drow[((long)b * a.x.H + h) * a.x.T + tt.t0 + 4 * ty + i] = drow[i];
  }
  zero<C::RT, CB>(acc);
  for (int kt = 0; kt <= tt.j; ++kt) {
    const bool diag = kt == tt.j;
    const int k0 = tt.kstart + kt * kTile, nk = diag ? tt.rows : kTile;
    if (kt > 0) __syncthreads();
    fill(Ks, ldh, a.x.K + (row0 + k0) * a.x.ld + c0, a.x.ld, nk, dh, a.vec);
    fill(Vs, ldh, a.x.V + (row0 + k0) * a.x.ld + c0, a.x.ld, nk, dh, a.vec);
    __syncthreads();
    p_ds<CB>(a, Qs, Ks, Gs, Vs, ldh, diag, tt.rows, lse, drow, nullptr, Ss);
    __syncthreads();
    rows_times<C4, CB>(Ss, kPld, Ks, ldh, dh, 0,
                       C::row() >= tt.rows ? 0 : diag ? min(C::row() + C::RT, nk) : kTile, 0, acc);
  }
  const unsigned bad = store_dq<E, C4, CB>(a, tt, b, h, acc);
  if (__syncthreads_or(bad)) redo_dq<E, C4, CB>(a, tt, sm, bad);
}

// Per key tile: dV_j = sum_t P_tj dO_t, dK_j = scale * sum_t P_tj (dO_t . v_j - Drow_t) q_t
// over queries t in [j, blockend(j)), tile by tile.  FUSED (L <= 64, where the
// tile is its own and only query tile): Drow is formed here and dQ joins, one
// pass instead of two.  Without scratch for Drow (the allocation-free backward) each
// query tile's is formed again here, by the same sums.
template <class E, int C4, int CB, bool FUSED>
__global__ void __launch_bounds__(kThreads, CB == 1 ? 2 : 1)
    attn_bwd_kv_simt_kernel(const __grid_constant__ SimtArgs<E> a) {
  pdl_enter();
  extern __shared__ __align__(16) float sm[];
  const int dh = a.x.dh, ldh = dh + 4;
  float *Ks = sm, *Vs = Ks + kTile * ldh, *Qs = Vs + kTile * ldh, *Gs = Qs + kTile * ldh,
        *Ps = Gs + kTile * ldh, *Ss = Ps + kTile * kPld;
  const TileAt tt = tile_at<false>(a);
  const int h = tt.h, b = tt.b;
  if (tt.rows <= 0) return;
  const long row0 = (long)b * a.x.T;
  const int c0 = h * dh;
  fill(Ks, ldh, a.x.K + (row0 + tt.t0) * a.x.ld + c0, a.x.ld, tt.rows, dh, a.vec);
  fill(Vs, ldh, a.x.V + (row0 + tt.t0) * a.x.ld + c0, a.x.ld, tt.rows, dh, a.vec);
  using C = Cols<C4, CB>;
  float dk[C::RT][CB][4], dv[C::RT][CB][4];
  zero<C::RT, CB>(dk);
  zero<C::RT, CB>(dv);
  const int jend = FUSED ? 1 : (min(a.x.L, a.x.T - tt.kstart) + kTile - 1) / kTile;
  for (int i = tt.j; i < jend; ++i) {
    const bool diag = i == tt.j;
    const int t0 = FUSED ? tt.t0 : tt.kstart + i * kTile;
    const int rows = FUSED ? tt.rows : min(min(kTile, a.x.L - i * kTile), a.x.T - t0);
    if (!diag) __syncthreads();
    fill(Qs, ldh, a.x.Q + (row0 + t0) * a.x.ld + c0, a.x.ld, rows, dh, a.vec);
    fill(Gs, ldh, a.x.dO + (row0 + t0) * a.x.ld_o + c0, a.x.ld_o, rows, dh, true);
    float drow[4], lse[4];
    if (FUSED || !a.Drow)
      drow4(a, b, h, t0, rows, drow);
    else
      rows_lse(a, b, h, t0, rows, a.Drow, drow);
    rows_lse(a, b, h, t0, rows, a.lse, lse);
    __syncthreads();
    p_ds<CB>(a, Qs, Ks, Gs, Vs, ldh, diag, rows, lse, drow, Ps, Ss);
    __syncthreads();
    // the queries that see any of the thread's keys
    const int lo = diag ? C::row() : 0;
    const int hi = min(rows, diag ? block_end(C::row() + C::RT - 1, a.x.L) : kTile);
    cols_times<C4, CB>(Ps, Gs, ldh, dh, lo, hi, dv);
    cols_times<C4, CB>(Ss, Qs, ldh, dh, lo, hi, dk);
  }
  const int c = C::col();
  unsigned badk = 0u, badv = 0u;
#pragma unroll
  for (int i = 0; i < C::RT; ++i) {
    const int r = C::row() + i, t = tt.t0 + r;
    if (r >= tt.rows) break;
#pragma unroll
    for (int m = 0; m < CB; ++m)
      if (c + 64 * m < dh) {
        if (!finite4(dk[i][m])) badk |= 1u << (i * CB + m);
        if (!finite4(dv[i][m])) badv |= 1u << (i * CB + m);
        const long o = (row0 + t) * a.ld_d + c0 + c + 64 * m;
        put4(a.dV + o, dv[i][m], a.vec);
        put4(a.dK + o, dk[i][m], a.vec);
      }
  }
  if (FUSED) {
    float dq[C::RT][CB][4];
    zero<C::RT, CB>(dq);
    rows_times<C4, CB>(Ss, kPld, Ks, ldh, dh, block_row(C::row(), a.x.L),
                       C::row() >= tt.rows ? 0 : min(C::row() + C::RT, tt.rows), 0, dq);
    const unsigned badq = store_dq<E, C4, CB>(a, tt, b, h, dq);
    if (__syncthreads_or(badq)) redo_dq<E, C4, CB>(a, tt, sm, badq);
  }
  if (__syncthreads_or(badk | badv)) redo_dkv<E, C4, CB>(a, tt, sm, badk, badv);
}

namespace {
template <class E>
SimtArgs<E> simt_args(const AttnArgs& f, const AttnBwdArgs* ab) {
  SimtArgs<E> a;
  a.x = AttnPtrs<E>{(const E*)f.Q, (const E*)f.K, (const E*)f.V, (const E*)f.O,
                    ab ? (const E*)ab->dO : nullptr, f.ld_qkv, f.ld_o, f.lse,
                    ab && f.L > kTile ? ab->Drow : nullptr, f.T, f.H, f.dh, f.L,
                    1.0f / sqrtf((float)f.dh), f.ld_qkv % 8 == 0};
  a.Out = (E*)f.O;
  a.dQ = ab ? (E*)ab->dQ : nullptr;
  a.dK = ab ? (E*)ab->dK : nullptr;
  a.dV = ab ? (E*)ab->dV : nullptr;
  a.ld_d = ab ? ab->ld_dqkv : 0;
  a.lse = f.lse;
  a.Drow = ab ? ab->Drow : nullptr;
  a.rows = f.L <= kTile ? (kTile / f.L) * f.L : kTile;
  // (a block is no longer than the sequence: no tiles for the rest of it)
  a.tpb = f.L <= kTile ? 1 : (std::min(f.L, f.T) + kTile - 1) / kTile;
  a.nb = f.L <= kTile ? (f.T + a.rows - 1) / a.rows : (f.T + f.L - 1) / f.L;
  a.B = f.B;
  // rows of q, k, v and of the gradients may have any stride; those of O and dO
  // are D elements apart, a multiple of 64
  a.vec = f.ld_qkv % 4 == 0 && a.ld_d % 4 == 0;
  return a;
}

// Bytes of `tiles` tiles of dh + 4 columns and `cols` columns of scores per row.
int simt_smem(int tiles, int cols, int dh) {
  return kTile * (tiles * (dh + 4) + cols) * (int)sizeof(float);
}

constexpr int kHalfSm = 113 * 1024;  // shared memory of each of two CTAs on an SM

template <class K, class E, class... X>
cudaError_t simt_launch(const Launch& lc, K kern, std::atomic<unsigned long long>* opted, int tiles,
                        int cols, int max_cols, const AttnArgs& f, const SimtArgs<E>& a, X... x) {
  // the limit is raised once per kernel and device, to the largest size needed
  if (cudaError_t e = smem_opt_in(kern, simt_smem(std::max(tiles, 3), max_cols, kMaxDh), opted);
      e != cudaSuccess)
    return e;
  const double grid = (double)a.nb * a.tpb * f.H * f.B;
  if (grid > INT_MAX) return cudaErrorInvalidConfiguration;
  cudaError_t e = launch_k(kern, dim3((unsigned)grid), dim3(kThreads),
                           simt_smem(tiles, cols, f.dh), lc.stream, a, x...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// f(C4, CB) for the head width: column groups of four over 16 threads, blocks
// of 64 columns.
template <class F>
cudaError_t with_cols(int dh, F&& f) {
  using std::integral_constant;
  if (dh <= 16) return f(integral_constant<int, 4>(), integral_constant<int, 1>());
  if (dh <= 32) return f(integral_constant<int, 8>(), integral_constant<int, 1>());
  if (dh <= 64) return f(integral_constant<int, 16>(), integral_constant<int, 1>());
  return f(integral_constant<int, 16>(), integral_constant<int, 2>());
}

template <class E>
cudaError_t fwd_typed(const Launch& lc, const AttnArgs& f) {
  const SimtArgs<E> a = simt_args<E>(f, nullptr);
  return with_cols(f.dh, [&](auto c4, auto cb) {
    static std::atomic<unsigned long long> opted{0};
    // the row's scores (four more columns of padding), and one for the sums
    const int ldp = a.tpb <= kKeep ? a.tpb * kTile + 4 : kPld;
    const int share = simt_smem(3, ldp + 1, f.dh) > kHalfSm && simt_smem(2, ldp + 1, f.dh) <= kHalfSm;
    return simt_launch(lc, attn_fwd_simt_kernel<E, decltype(c4)::value, decltype(cb)::value>,
                       &opted, 3 - share, ldp + 1, kKeep * kTile + 5, f, a, ldp, share);
  });
}

template <class E>
cudaError_t bwd_typed(const Launch& lc, const AttnBwdArgs& ab) {
  const SimtArgs<E> a = simt_args<E>(ab.f, &ab);
  return with_cols(ab.f.dh, [&](auto c4, auto cb) {
    constexpr int C4 = decltype(c4)::value, CB = decltype(cb)::value;
    static std::atomic<unsigned long long> o1{0}, o2{0}, o3{0};
    if (ab.f.L <= kTile)
      return simt_launch(lc, attn_bwd_kv_simt_kernel<E, C4, CB, true>, &o1, 4, 2 * kPld, 2 * kPld, ab.f, a);
    cudaError_t e = simt_launch(lc, attn_bwd_q_simt_kernel<E, C4, CB>, &o2, 4, kPld, kPld, ab.f, a);
    if (e != cudaSuccess) return e;
    return simt_launch(lc, attn_bwd_kv_simt_kernel<E, C4, CB, false>, &o3, 4, 2 * kPld, 2 * kPld, ab.f, a);
  });
}
}  // namespace

cudaError_t attn_fwd_simt(const Launch& lc, int dtype, const AttnArgs& a) {
  if (a.dh > kMaxDh || a.L > kMaxL) return cudaErrorInvalidValue;
  return dtype == 0 ? fwd_typed<float>(lc, a) : fwd_typed<bf16>(lc, a);
}

cudaError_t attn_bwd_simt(const Launch& lc, int dtype, const AttnBwdArgs& a) {
  if (a.f.dh > kMaxDh || a.f.L > kMaxL) return cudaErrorInvalidValue;
  return dtype == 0 ? bwd_typed<float>(lc, a) : bwd_typed<bf16>(lc, a);
}

}  // namespace bcmt
