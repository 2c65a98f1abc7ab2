// Backward of the intra-block causal attention on the tcgen05 tensor cores (Sec.
// 3.3) for the bf16 shapes that attn_tc.cu and attn_flash.cu do not take: any
// head width that is a multiple of 8 up to 128, any block size up to 1024.  (Their
// forward is attn_simt.cu's.)
//
// Tiles.  A head's 128-token tile comes in by TMA as NC = ceil(dh / 64) boxes
// of 128 rows x 64 columns (128-byte swizzle).  The tensor maps are 4-D
// (dh, H, T, B), so columns past the head and tokens past the sequence are
// zero-filled (and clipped on the way out) whatever dh is.  For L <= 128 a
// tile starts at a block and holds the 128 / L whole blocks that fit: keys and
// queries are the same tile, the mask is block-diagonal causal.  For L > 128 a
// tile is up to 128 rows of one block and walks the block's other tiles.
// Loads always bring 128 rows; the rows that belong to the next tile are
// masked, and output boxes are as high as the tile has rows of its own.
//
// Precision.  The probabilities P and the score gradients dS are fp32 values; as
// operands of the tensor-core products they enter as the sum of three bf16 numbers,
// which is exact (24 significand bits; below 2^-110 the last part underflows).  The other
// operands are the bf16 tensors themselves.  Exponentials are ex2.approx of an argument
// that is right to 2^-24 of its terms (Exp2; expf took 91 us where this takes 79).  Against
// float64 on the same O, over 82 shapes (heads of 8 to 128, blocks of 16 to 1024), the
// relative error of the bf16 gradients is the CUDA-core kernels' times 1.0000003 on average
// (1.0000056 at most; times 0.9999986 against the gradients of the unrounded O), and 0.22 %
// of the values round to another bf16 number than float64's (0.15 % there; with P and dS
// as two parts each 0.63 %).
//
// Work split: 256 threads; warp w owns TMEM lane quarter w % 4 (thread = one
// query row) and half w / 4 of the 128 key columns (of the dh output columns
// in the epilogues).  What bounds it: the chain load -> S, dP -> P -> dV -> dS
// -> dK, dQ of one CTA, several microseconds, covered by a second CTA per SM
// where shared memory allows (heads up to 64, which then keep two parts in shared
// memory at a time and the third in registers until the first two are multiplied).
// Against the CUDA-core kernels that served these shapes before (one warp per row,
// operands re-read from L2 per row): B4 T2048 D1024 heads of 128 L128 8230 -> 79 us,
// B4 T1000 D768 heads of 96 L48 1161 -> 43 us (73 and 39 with two parts per value).
//
// A masked key's weight is exactly 0, but 0 x inf = NaN in the products: a row
// whose result is not finite is formed again from its visible keys alone
// (attn_slow.cuh).
#include "attn_common.cuh"
#include "attn_slow.cuh"
#include "common.cuh"
#include "internal.h"
#include "tc.cuh"
#include "tmap.h"

namespace bcmt {
using namespace attn;

namespace {
constexpr int kTile = 128;
constexpr int kThreads = 256;
constexpr uint32_t kChunk = 16384;  // one 128-row x 64-column box
constexpr uint32_t kP = 32768;      // one 128 x 128 bf16 operand (a part of P or dS)

// What the kernels need beside their tensor maps.
struct GenArgs {
  AttnPtrs<bf16> x;
  float* Drow;
  int rows;   // L <= 128: rows per tile (whole blocks)
  int tpb;    // L > 128: tiles per block
  unsigned* status;
};

// a, b as bf16 pairs h + m + l, exactly.
__device__ __forceinline__ void split3(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack2(a, b);
  a -= __uint_as_float(h << 16);
  b -= __uint_as_float(h & 0xffff0000u);
  m = pack2(a, b);
  l = pack2(a - __uint_as_float(m << 16), b - __uint_as_float(m & 0xffff0000u));
}
// Eight values' parts, a 16-byte unit each.
__device__ __forceinline__ void split_unit(const float* v, uint4& h, uint4& m, uint4& l) {
  split3(v[0], v[1], h.x, m.x, l.x);
  split3(v[2], v[3], h.y, m.y, l.y);
  split3(v[4], v[5], h.z, m.z, l.z);
  split3(v[6], v[7], h.w, m.w, l.w);
}

// e^(s scale - lse) as a power of two, the argument to 2^-24 of its terms: `c` = scale
// log2 e and `n` = -lse log2 e as sums of two floats.
struct Exp2 {
  float ch, cl, nh, nl;
  __device__ __forceinline__ Exp2(float scale, float lse) {
    constexpr float kl = 1.92596299e-8f;  // log2 e - float(log2 e)
    ch = scale * kLog2e;
    cl = fmaf(scale, kLog2e, -ch) + scale * kl;
    nh = -lse * kLog2e;
    nl = -fmaf(lse, kLog2e, nh) - lse * kl;
  }
  __device__ __forceinline__ float operator()(float s) const {
    return ex2(fmaf(s, ch, nh) + fmaf(s, cl, nl));
  }
};

// One head tile: NC boxes of 64 columns.
template <int NC>
__device__ __forceinline__ void load_tile(uint8_t* dst, const CUtensorMap* m, uint64_t* bar, int h,
                                          int t, int b) {
#pragma unroll
  for (int c = 0; c < NC; ++c) tc::tma_load_4d(dst + c * kChunk, m, bar, 64 * c, h, t, b);
}
template <int NC>
__device__ __forceinline__ void store_tile(const CUtensorMap* m, const uint8_t* src, int h, int t,
                                           int b) {
#pragma unroll
  for (int c = 0; c < NC; ++c) tc::tma_store_4d(m, src + c * kChunk, 64 * c, h, t, b);
}

// Operand descriptors: a head tile K-major (K = columns, step kk of 16) or
// MN-major (N = columns, K = rows, step kk), P / dS K-major (K = keys) or
// MN-major (M = keys, K = queries).  All are 64-column swizzle-128 chunks
// 16 KB apart.
__device__ __forceinline__ uint64_t d_kmaj(const uint8_t* t, int kk) {
  return tc::desc_at(tc::sdesc(tc::smem_u32(t), 16, 1024), (kk >> 2) * kChunk + (kk & 3) * 32);
}
__device__ __forceinline__ uint64_t d_mnmaj(const uint8_t* t, int kk) {
  return tc::desc_at(tc::sdesc(tc::smem_u32(t), kChunk, 1024), kk * 2048);
}

// Columns of the tile the thread's half owns in the epilogues: OC = 32 NC from
// column hf * OC.  Stages OC values of row r as bf16 into a head tile.
template <int NC>
__device__ __forceinline__ void stage_half(uint8_t* tile, int r, int hf, const float* v) {
#pragma unroll
  for (int u = 0; u < 4 * NC; ++u) {
    const int unit = hf * 4 * NC + u;
    *reinterpret_cast<uint4*>(tile + (unit >> 3) * kChunk + tc::sw128_offset(r, unit & 7)) =
        pack8(v + 8 * u);
  }
}
template <int NC>
__device__ __forceinline__ void tmem_half(uint32_t taddr, float* v) {
  uint32_t x[NC][32];
#pragma unroll
  for (int c = 0; c < NC; ++c) tc::tmem_ld32_issue(taddr + 32u * c, x[c]);
  tc::tmem_wait();
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int j = 0; j < 32; ++j) v[32 * c + j] = __uint_as_float(x[c][j]);
}

// Tile x of a sequence: its first token, its rows, the first row of its block
// (L > 128), its index within the block.
struct TileAt {
  int t0, rows, kstart, j;
};
__device__ __forceinline__ TileAt tile_at(const GenArgs& a, int x) {
  TileAt t;
  if (a.x.L <= kTile) {
    t.t0 = t.kstart = x * a.rows;
    t.j = 0;
    t.rows = min(a.rows, a.x.T - t.t0);
  } else {
    const int i = x / a.tpb;
    t.j = x - i * a.tpb;
    t.kstart = i * a.x.L;
    t.t0 = t.kstart + t.j * kTile;
    t.rows = min(min(kTile, a.x.L - t.j * kTile), a.x.T - t.t0);
  }
  return t;
}

// Drow = dO_t . O_t.
__device__ __forceinline__ float drow_of(const GenArgs& a, long row, int h) {
  const bf16* o = a.x.O + row * a.x.ld_o + h * a.x.dh;
  const bf16* g = a.x.dO + row * a.x.ld_o + h * a.x.dh;
  float s = 0.f;
#pragma unroll 4
  for (int c = 0; c < a.x.dh; c += 8) {
    float ov[8], gv[8];
    load8(o + c, ov);
    load8(g + c, gv);
#pragma unroll
    for (int e = 0; e < 8; ++e) s = fmaf(ov[e], gv[e], s);
  }
  return s;
}

// Swizzled tiles need the 1024-byte alignment that the declaration asks for.
__device__ __forceinline__ bool aligned_smem(const uint8_t* smem, unsigned* status) {
  if ((tc::smem_u32(smem) & 1023u) == 0) return true;
  if (threadIdx.x == 0) atomicOr(status, kStatusBadLaunch);
  return false;
}

// The 16-byte units (eight columns) of the thread's half row that are not finite.
template <int OC>
__device__ __forceinline__ unsigned bad_units(const float* v, int c0, int dh) {
  unsigned bad = 0u;
#pragma unroll
  for (int c = 0; c < OC; ++c)
    if (c0 + c < dh && !is_finite(v[c])) bad |= 1u << (c / 8);
  return bad;
}
// Those of the CTA's rows formed again, row by row, in the staging tiles (bad: of row r
// from unit u0 on; sm: free shared memory).
__device__ __forceinline__ void put_units(uint8_t* tile, int r, const SlowRow& row, unsigned units,
                                          int dh) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int c = (threadIdx.x & 31) + 32 * i, u = c / 8;
    if (c < dh && (units >> u & 1u))
      *reinterpret_cast<bf16*>(tile + (u >> 3) * kChunk + tc::sw128_offset(r, u & 7) + 2 * (c & 7)) =
          from_f<bf16>(row.v[i]);
  }
}
__device__ __noinline__ void restage_dq(const GenArgs& a, int b, int h, int t0, uint8_t* tile, int r,
                                        int u0, unsigned bad, uint8_t* sm) {
  slow_rows<kTile>(reinterpret_cast<float*>(sm), [&](auto set) {
    for (int u = 0; u < 8; ++u)
      if (bad >> u & 1u) set(r, u0 + u);
  }, [&](int n, unsigned units, float* w) {
    SlowRow dq;
    slow_dq(a.x, b, h, t0 + n, w, dq);
    put_units(tile, n, dq, units, a.x.dh);
  });
}
__device__ __noinline__ void restage_dkv(const GenArgs& a, int b, int h, int t0, uint8_t* tk,
                                         uint8_t* tv, int r, int u0, unsigned badk, unsigned badv,
                                         uint8_t* sm) {
  slow_rows<2 * kTile>(reinterpret_cast<float*>(sm), [&](auto set) {
    for (int u = 0; u < 8; ++u) {
      if (badk >> u & 1u) set(r, u0 + u);
      if (badv >> u & 1u) set(kTile + r, u0 + u);
    }
  }, [&](int n, unsigned units, float* w) {
    const int row = n & (kTile - 1);
    SlowRow d;
    if (n < kTile)
      slow_dkv<false>(a.x, b, h, t0 + row, w, d);
    else
      slow_dkv<true>(a.x, b, h, t0 + row, w, d);
    put_units(n < kTile ? tk : tv, row, d, units, a.x.dh);
  });
}
}  // namespace

// ============================================================ backward: dQ
// For L > 128: per query tile, Drow, then per key tile S and dP (128 + 128 TMEM
// columns), dS = P (dP - Drow) scale as three parts (the first over the consumed V),
// the product dS K into the S columns, accumulated in registers.  NC = 1: 112 KB, two
// CTAs per SM, the third part through the first's buffer; NC = 2: 192 KB.
template <int NC> constexpr int dq_smem() { return 3 * NC * (int)kChunk + (NC + 1) * (int)kP; }

template <int NC>
__global__ void __launch_bounds__(kThreads, NC == 1 ? 2 : 1)
    attn_bwd_dq_gen_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
                           const __grid_constant__ CUtensorMap mV, const __grid_constant__ CUtensorMap mdO,
                           const __grid_constant__ CUtensorMap mdQ, const __grid_constant__ CUtensorMap mdQt,
                           const __grid_constant__ GenArgs a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr uint32_t kT = NC * kChunk;
  constexpr int OC = 32 * NC;
  uint8_t* sQ = smem;
  uint8_t* sdO = smem + kT;
  uint8_t* sK = smem + 2 * kT;
  uint8_t* sV = smem + 3 * kT;
  uint8_t* sS = sV;  // dS's parts, kP apart, over V (and, NC = 1, the 16 KB after it)
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + dq_smem<NC>());  // loads, S/dP, dQ
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 3);

  const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;
  const bool warp0 = warp == 0;
  const int q = warp & 3, hf = warp >> 2;
  const int h = blockIdx.y, b = blockIdx.z;
  const TileAt tt = tile_at(a, blockIdx.x);
  if (tt.rows <= 0 || !aligned_smem(smem, a.status)) {
    pdl_enter();
    return;
  }
  if (warp0 && tc::elect_one()) {
    for (int i = 0; i < 3; ++i) tc::mbar_init(&bar[i], 1);
    tc::fence_mbar_init();
    tc::prefetch_tmap(&mQ);
    tc::prefetch_tmap(&mK);
    tc::prefetch_tmap(&mV);
    tc::prefetch_tmap(&mdO);
  }
  pdl_enter();
  if (warp0 && tc::elect_one()) {
    tc::mbar_arrive_expect_tx(&bar[0], 4 * kT);
    load_tile<NC>(sQ, &mQ, &bar[0], h, tt.t0, b);
    load_tile<NC>(sK, &mK, &bar[0], h, tt.kstart, b);
    load_tile<NC>(sdO, &mdO, &bar[0], h, tt.t0, b);
    load_tile<NC>(sV, &mV, &bar[0], h, tt.kstart, b);
  }
  __syncwarp();
  if (warp == 0) {
    tc::tmem_alloc(tslot, 256);
    tc::tmem_relinquish();
  }
  const int r = q * 32 + lane;
  const bool row_ok = r < tt.rows;
  const long lrow = ((long)b * a.x.H + h) * a.x.T + tt.t0 + r;
  const float drow = row_ok ? drow_of(a, (long)b * a.x.T + tt.t0 + r, h) : 0.f;
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
  const int nk = (a.x.dh + 15) / 16;
  if (row_ok && hf == 0) a.Drow[lrow] = drow;
  const Exp2 prob(a.x.scale, row_ok ? a.x.lse[lrow] : 0.f);
  float acc[OC];
#pragma unroll
  for (int c = 0; c < OC; ++c) acc[c] = 0.f;
  bool ok = true;

  for (int kt = 0; kt <= tt.j; ++kt) {
    const bool diag = kt == tt.j;
    if (warp0 && tc::elect_one()) {
      const bool okk = tc::mbar_wait(&bar[0], kt & 1, a.status);
      tc::fence_after_sync();
      if (okk) {
        constexpr uint32_t id = tc::idesc_bf16(128, 128, 0, 0);
        for (int kk = 0; kk < nk; ++kk)
          tc::mma_bf16(tmem, d_kmaj(sQ, kk), d_kmaj(sK, kk), id, kk > 0 ? 1u : 0u);
        for (int kk = 0; kk < nk; ++kk)
          tc::mma_bf16(tmem + 128, d_kmaj(sdO, kk), d_kmaj(sV, kk), id, kk > 0 ? 1u : 0u);
      }
      tc::mma_commit(&bar[1]);
    }
    __syncwarp();
    ok = tc::mbar_wait(&bar[1], kt & 1, a.status) && ok;
    tc::fence_after_sync();
    uint4 last[8];  // NC = 1: the third parts
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int k0 = hf * 64 + c * 32;
      const bool use = !diag || k0 <= q * 32 + 31;
      float s[32], dp[32];
      tc::tmem_ld32_issue(trow + (uint32_t)k0, reinterpret_cast<uint32_t*>(s));
      tc::tmem_ld32_issue(trow + 128u + (uint32_t)k0, reinterpret_cast<uint32_t*>(dp));
      tc::tmem_wait();
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const bool vis = use && row_ok && (!diag || k0 + j <= r);
        s[j] = vis ? prob(s[j]) * (dp[j] - drow) * a.x.scale : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        uint4 hm[2];
        split_unit(s + 8 * u, hm[0], hm[1], last[4 * c + u]);
        put_unit(sS, r, hf * 8 + c * 4 + u, hm[0]);
        put_unit(sS + kP, r, hf * 8 + c * 4 + u, hm[1]);
        if (NC == 2) put_unit(sS + 2 * kP, r, hf * 8 + c * 4 + u, last[4 * c + u]);
      }
    }
    tc::fence_proxy_async_smem();
    tc::fence_before_sync();
    __syncthreads();  // dS is in place, S and dP are read
    const uint32_t idQ = tc::idesc_bf16(128, nk * 16, 0, 1);
    const int nkk = diag ? (tt.rows + 15) / 16 : 8;
    if (warp0 && tc::elect_one()) {
      tc::fence_after_sync();
      if (ok)
        for (int part = NC; part >= 0; --part)  // the smallest first
          for (int kk = 0; kk < nkk; ++kk)
            tc::mma_bf16(tmem, p_kmaj(sS + part * kP, 0, kk), d_mnmaj(sK, kk), idQ,
                         part < NC || kk > 0 ? 1u : 0u);
      tc::mma_commit(&bar[2]);
    }
    __syncwarp();
    ok = tc::mbar_wait(&bar[2], NC == 1 ? 0u : (uint32_t)(kt & 1), a.status) && ok;
    tc::fence_after_sync();
    if (NC == 1) {  // the third part, in the first's place
#pragma unroll
      for (int u = 0; u < 8; ++u) put_unit(sS, r, hf * 8 + u, last[u]);
      tc::fence_proxy_async_smem();
      tc::fence_before_sync();
      __syncthreads();
      if (warp0 && tc::elect_one()) {
        tc::fence_after_sync();
        if (ok)
          for (int kk = 0; kk < nkk; ++kk)
            tc::mma_bf16(tmem, p_kmaj(sS, 0, kk), d_mnmaj(sK, kk), idQ, 1u);
        tc::mma_commit(&bar[2]);
      }
      __syncwarp();
      ok = tc::mbar_wait(&bar[2], 1u, a.status) && ok;
      tc::fence_after_sync();
    }
    if (warp0 && tc::elect_one() && kt < tt.j) {  // K, V and dS are consumed: the next key tile
      tc::mbar_arrive_expect_tx(&bar[0], 2 * kT);
      load_tile<NC>(sK, &mK, &bar[0], h, tt.kstart + (kt + 1) * kTile, b);
      load_tile<NC>(sV, &mV, &bar[0], h, tt.kstart + (kt + 1) * kTile, b);
    }
    __syncwarp();
    float o[OC];
    tmem_half<NC>(trow + (uint32_t)(hf * OC), o);
#pragma unroll
    for (int c = 0; c < OC; ++c) acc[c] += o[c];
    tc::fence_before_sync();
    __syncthreads();  // the product is read before the next S overwrites it
    tc::fence_after_sync();
  }

  const unsigned bad = row_ok ? bad_units<OC>(acc, hf * OC, a.x.dh) : 0u;
  stage_half<NC>(sQ, r, hf, acc);
  if (__syncthreads_or(bad)) restage_dq(a, b, h, tt.t0, sQ, r, hf * OC / 8, bad, sS);
  tc::fence_proxy_async_smem();
  __syncthreads();
  if (warp0 && tc::elect_one() && ok) {
    store_tile<NC>(tt.j == a.tpb - 1 ? &mdQt : &mdQ, sQ, h, tt.t0, b);
    tc::tma_store_commit();
    tc::tma_store_wait_read<0>();
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// ====================================================== backward: dK, dV (dQ)
// Per key tile, its query tiles in turn: S = Q K^T and dP = dO V^T, P as three parts
// for dV += P^T dO, dS = P (dP - Drow) scale, which waits in fp32 in dP's TMEM columns
// until the dV product has consumed P, as three parts in P's buffers for dK += dS^T Q.
// FUSED (L <= 128: the key tile is its own and only query tile): Drow is computed
// here and dQ = dS K joins; P's first part covers the consumed V, and the products
// reuse the columns of S and dP.  At NC = 1 that form has two buffers (112 KB and 256
// columns, two CTAs per SM) and three rounds of products: P's first two parts; its
// third and dS's first; dS's others.
template <int NC, bool FUSED> constexpr int dkv_parts() { return FUSED && NC == 1 ? 2 : 3; }
template <int NC, bool FUSED> constexpr int dkv_smem() {
  return (FUSED ? 3 : 4) * NC * (int)kChunk + dkv_parts<NC, FUSED>() * (int)kP;
}
template <int NC, bool FUSED> constexpr int dkv_cols() { return FUSED && NC == 1 ? 256 : 512; }

template <int NC, bool FUSED>
__global__ void __launch_bounds__(kThreads, FUSED && NC == 1 ? 2 : 1)
    attn_bwd_dkv_gen_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
                            const __grid_constant__ CUtensorMap mV, const __grid_constant__ CUtensorMap mdO,
                            const __grid_constant__ CUtensorMap mdQ, const __grid_constant__ CUtensorMap mdK,
                            const __grid_constant__ CUtensorMap mdV, const __grid_constant__ CUtensorMap mdKt,
                            const __grid_constant__ CUtensorMap mdVt, const __grid_constant__ GenArgs a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr uint32_t kT = NC * kChunk;
  constexpr int OC = 32 * NC;
  constexpr int PARTS = dkv_parts<NC, FUSED>();
  constexpr uint32_t kDV = FUSED ? 0 : 256, kDK = kDV + 64 * NC, kDQ = FUSED ? 128 * NC : 0;
  uint8_t* sQ = smem;              // Q; FUSED: then dQ staging
  uint8_t* sdO = smem + kT;        // dO; then dV staging
  uint8_t* sK = smem + 2 * kT;     // K; then dK staging
  uint8_t* sV = smem + 3 * kT;
  uint8_t* sP = FUSED ? sV : smem + 4 * kT;  // the parts of P, then of dS, kP apart
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + dkv_smem<NC, FUSED>());  // loads, S/dP, dV, dK
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 4);

  const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;
  const bool warp0 = warp == 0;
  const int q = warp & 3, hf = warp >> 2;
  const int h = blockIdx.y, b = blockIdx.z;
  const TileAt tt = tile_at(a, blockIdx.x);
  if (tt.rows <= 0 || !aligned_smem(smem, a.status)) {
    pdl_enter();
    return;
  }
  // query tiles tt.j .. jend-1 of the block
  const int jend = FUSED ? 1 : min(a.tpb, (min(a.x.L, a.x.T - tt.kstart) + kTile - 1) / kTile);
  if (warp0 && tc::elect_one()) {
    for (int i = 0; i < 4; ++i) tc::mbar_init(&bar[i], 1);
    tc::fence_mbar_init();
    tc::prefetch_tmap(&mQ);
    tc::prefetch_tmap(&mK);
    tc::prefetch_tmap(&mV);
    tc::prefetch_tmap(&mdO);
  }
  pdl_enter();
  if (warp0 && tc::elect_one()) {
    tc::mbar_arrive_expect_tx(&bar[0], 4 * kT);
    load_tile<NC>(sQ, &mQ, &bar[0], h, tt.t0, b);
    load_tile<NC>(sK, &mK, &bar[0], h, tt.t0, b);
    load_tile<NC>(sdO, &mdO, &bar[0], h, tt.t0, b);
    load_tile<NC>(sV, &mV, &bar[0], h, tt.t0, b);
  }
  __syncwarp();
  if (warp == 0) {
    tc::tmem_alloc(tslot, dkv_cols<NC, FUSED>());
    tc::tmem_relinquish();
  }
  const int r = q * 32 + lane;
  float drow = 0.f;
  if (FUSED && r < tt.rows) drow = drow_of(a, (long)b * a.x.T + tt.t0 + r, h);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
  const int nk = (a.x.dh + 15) / 16;
  const uint32_t idMN = tc::idesc_bf16(128, nk * 16, 1, 1);
  const int rbs = FUSED ? (r / a.x.L) * a.x.L : 0;
  const int wbs = FUSED ? ((q * 32) / a.x.L) * a.x.L : 0;
  bool ok = true;

  // products over the query rows with one part: dst (+)= part^T t, dQ (+)= part K
  // (operand descriptors formed once; a step along one adds its bytes / 16)
  const uint64_t pT = tc::sdesc(tc::smem_u32(sP), kChunk, 1024),
                 pK = tc::sdesc(tc::smem_u32(sP), 16, 1024), bQ = d_mnmaj(sQ, 0),
                 bO = d_mnmaj(sdO, 0), bK = d_mnmaj(sK, 0);
  auto times_t = [&](uint32_t dst, int part, uint64_t t, int nkk, bool first) {
    const uint64_t p = pT + part * (kP / 16);
#pragma unroll 4
    for (int kk = 0; kk < nkk; ++kk)
      tc::mma_bf16(tmem + dst, p + kk * 128, t + kk * 128, idMN, first && kk == 0 ? 0u : 1u);
  };
  auto times_k = [&](int part, int nkk, bool first) {
    const uint32_t idQ = tc::idesc_bf16(128, nk * 16, 0, 1);
    const uint64_t p = pK + part * (kP / 16);
#pragma unroll 4
    for (int kk = 0; kk < nkk; ++kk)
      tc::mma_bf16(tmem + kDQ, p + (kk >> 2) * 1024 + (kk & 3) * 2, bK + kk * 128, idQ,
                   first && kk == 0 ? 0u : 1u);
  };
  for (int i = tt.j, it = 0; i < jend; ++i, ++it) {  // FUSED: j = 0, jend = 1
    const bool diag = it == 0;
    const int t0 = FUSED ? tt.t0 : tt.kstart + i * kTile;
    const int rows = FUSED ? tt.rows : min(min(kTile, a.x.L - i * kTile), a.x.T - t0);
    const bool row_ok = r < rows;
    const long lrow = ((long)b * a.x.H + h) * a.x.T + t0 + r;
    const Exp2 prob(a.x.scale, row_ok ? a.x.lse[lrow] : 0.f);
    if (!FUSED) drow = row_ok ? a.Drow[lrow] : 0.f;
    if (warp0 && tc::elect_one()) {
      const bool okk = tc::mbar_wait(&bar[0], it & 1, a.status);
      tc::fence_after_sync();
      if (okk) {
        constexpr uint32_t id = tc::idesc_bf16(128, 128, 0, 0);
        for (int kk = 0; kk < nk; ++kk)
          tc::mma_bf16(tmem, d_kmaj(sQ, kk), d_kmaj(sK, kk), id, kk > 0 ? 1u : 0u);
        for (int kk = 0; kk < nk; ++kk)
          tc::mma_bf16(tmem + 128, d_kmaj(sdO, kk), d_kmaj(sV, kk), id, kk > 0 ? 1u : 0u);
      }
      tc::mma_commit(&bar[1]);
    }
    __syncwarp();
    ok = tc::mbar_wait(&bar[1], it & 1, a.status) && ok;
    tc::fence_after_sync();
    // P to shared memory, dS (fp32) over dP in TMEM
    uint4 third[8];  // two buffers: P's third parts, then dS's second and third
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int k0 = hf * 64 + c * 32;
      const bool use = !diag || (k0 <= q * 32 + 31 && k0 + 31 >= wbs);
      float s[32], dp[32];
      tc::tmem_ld32_issue(trow + (uint32_t)k0, reinterpret_cast<uint32_t*>(s));
      tc::tmem_ld32_issue(trow + 128u + (uint32_t)k0, reinterpret_cast<uint32_t*>(dp));
      tc::tmem_wait();
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const int kk = k0 + j;
        const bool vis = use && row_ok && (!diag || (kk >= rbs && kk <= r));
        s[j] = vis ? prob(s[j]) : 0.f;
        dp[j] = vis ? s[j] * (dp[j] - drow) * a.x.scale : 0.f;
      }
      tc::tmem_st32(trow + 128u + (uint32_t)k0, dp);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int unit = hf * 8 + c * 4 + u;
        uint4 h, m;
        split_unit(s + 8 * u, h, m, third[4 * c + u]);
        put_unit(sP, r, unit, h);
        put_unit(sP + kP, r, unit, m);
        if (PARTS == 3) put_unit(sP + 2 * kP, r, unit, third[4 * c + u]);
      }
    }
    tc::tmem_st_wait();
    tc::fence_proxy_async_smem();
    tc::fence_before_sync();
    __syncthreads();  // P is in place, S is read
    const int nkk = (rows + 15) / 16;  // queries past the tile's rows have P = dS = 0
    if (warp0 && tc::elect_one()) {
      tc::fence_after_sync();
      if (ok)
        for (int part = PARTS - 1; part >= 0; --part)  // dV += P^T dO, the smallest first
          times_t(kDV, part, bO, nkk, it == 0 && part == PARTS - 1);
      tc::mma_commit(&bar[2]);
    }
    __syncwarp();
    ok = tc::mbar_wait(&bar[2], it & 1, a.status) && ok;
    tc::fence_after_sync();
    uint4 second[8];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float ds[32];
      tc::tmem_ld32(trow + 128u + (uint32_t)(hf * 64 + c * 32), ds);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int unit = hf * 8 + c * 4 + u;
        if (PARTS == 2) put_unit(sP, r, unit, third[4 * c + u]);
        uint4 h;
        split_unit(ds + 8 * u, h, second[4 * c + u], third[4 * c + u]);
        if (PARTS == 2) {
          put_unit(sP + kP, r, unit, h);
        } else {
          put_unit(sP, r, unit, h);
          put_unit(sP + kP, r, unit, second[4 * c + u]);
          put_unit(sP + 2 * kP, r, unit, third[4 * c + u]);
        }
      }
    }
    tc::fence_proxy_async_smem();
    tc::fence_before_sync();
    __syncthreads();  // dS is in place; its TMEM columns are read
    if (warp0 && tc::elect_one()) {
      tc::fence_after_sync();
      if (ok) {
        if (PARTS == 2) {
          times_t(kDV, 0, bO, nkk, false);
          times_t(kDK, 1, bQ, nkk, true);
          times_k(1, nkk, true);
        } else {
          for (int part = 2; part >= 0; --part)  // dK += dS^T Q, dQ = dS K
            times_t(kDK, part, bQ, nkk, it == 0 && part == 2);
          if (FUSED)
            for (int part = 2; part >= 0; --part) times_k(part, nkk, part == 2);
        }
      }
      tc::mma_commit(&bar[3]);
    }
    __syncwarp();
    ok = tc::mbar_wait(&bar[3], it & 1, a.status) && ok;
    tc::fence_after_sync();
    if (PARTS == 2) {  // dS's other parts
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        put_unit(sP, r, hf * 8 + u, second[u]);
        put_unit(sP + kP, r, hf * 8 + u, third[u]);
      }
      tc::fence_proxy_async_smem();
      tc::fence_before_sync();
      __syncthreads();
      if (warp0 && tc::elect_one()) {
        tc::fence_after_sync();
        if (ok)
          for (int part = 0; part < 2; ++part) {
            times_t(kDK, part, bQ, nkk, false);
            times_k(part, nkk, false);
          }
        tc::mma_commit(&bar[3]);
      }
      __syncwarp();
      ok = tc::mbar_wait(&bar[3], 1u, a.status) && ok;
      tc::fence_after_sync();
    }
    if (!FUSED && warp0 && tc::elect_one() && i + 1 < jend) {  // the next query tile
      tc::mbar_arrive_expect_tx(&bar[0], 2 * kT);
      load_tile<NC>(sQ, &mQ, &bar[0], h, t0 + kTile, b);
      load_tile<NC>(sdO, &mdO, &bar[0], h, t0 + kTile, b);
    }
    __syncwarp();
  }

  // ---- rows of dV, dK (key r) and, FUSED, dQ (query r) through staging tiles
  auto staged = [&](uint32_t col, uint8_t* tile) {  // the row's units that are not finite
    float v[OC];
    tmem_half<NC>(trow + col + (uint32_t)(hf * OC), v);
    stage_half<NC>(tile, r, hf, v);
    return r < tt.rows ? bad_units<OC>(v, hf * OC, a.x.dh) : 0u;
  };
  const unsigned badv = staged(kDV, sdO), badk = staged(kDK, sK),
                 badq = FUSED ? staged(kDQ, sQ) : 0u;
  if (__syncthreads_or(badk | badv | badq)) {
    restage_dkv(a, b, h, tt.t0, sK, sdO, r, hf * OC / 8, badk, badv, sP);
    __syncthreads();
    if (FUSED) restage_dq(a, b, h, tt.t0, sQ, r, hf * OC / 8, badq, sP);
  }
  tc::fence_proxy_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  if (warp0 && tc::elect_one() && ok) {
    const bool tail = !FUSED && tt.j == a.tpb - 1;
    if (FUSED) store_tile<NC>(&mdQ, sQ, h, tt.t0, b);
    store_tile<NC>(tail ? &mdKt : &mdK, sK, h, tt.t0, b);
    store_tile<NC>(tail ? &mdVt : &mdV, sdO, h, tt.t0, b);
    tc::tma_store_commit();
    tc::tma_store_wait_read<0>();
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, dkv_cols<NC, FUSED>());
}

// ========================================================================= host
bool attn_gen_supported(int dtype, int dh, int L) {
  return dtype == 1 && dh >= 8 && dh <= 128 && dh % 8 == 0 && L >= 1 && L <= 1024 &&
         tmap_encoder() != nullptr;
}

namespace {
// [B, T] rows of H heads of dh columns, boxes of `rows` tokens x 64 columns
bool gen_map(CUtensorMap* m, const void* base, long ld, const AttnArgs& a, int rows) {
  if (ld % 8 != 0) return false;
  const uint64_t dims[4] = {(uint64_t)a.dh, (uint64_t)a.H, (uint64_t)a.T, (uint64_t)a.B};
  const uint64_t st[3] = {(uint64_t)a.dh * 2, (uint64_t)ld * 2, (uint64_t)ld * 2 * (uint64_t)a.T};
  const uint32_t box[4] = {64, 1, (uint32_t)rows, 1};
  return make_tmap_bf16(m, base, 4, dims, st, box);
}

constexpr int kExtra = 64;  // beside the tiles: barriers and the TMEM slot

GenArgs gen_args(const Launch& lc, const AttnBwdArgs& ab) {
  const AttnArgs& a = ab.f;
  GenArgs g;
  g.x = AttnPtrs<bf16>{(const bf16*)a.Q, (const bf16*)a.K, (const bf16*)a.V, (const bf16*)a.O,
                       (const bf16*)ab.dO, a.ld_qkv, a.ld_o, a.lse,
                       a.L > kTile ? ab.Drow : nullptr, a.T, a.H, a.dh, a.L,
                       1.0f / sqrtf((float)a.dh), 1};
  g.Drow = ab.Drow;
  g.rows = a.L <= kTile ? (kTile / a.L) * a.L : kTile;
  g.tpb = a.L <= kTile ? 1 : (a.L + kTile - 1) / kTile;
  g.status = lc.status;
  return g;
}
dim3 gen_grid(const AttnArgs& a, const GenArgs& g) {
  const int nx = a.L <= kTile ? (a.T + g.rows - 1) / g.rows : (a.T + a.L - 1) / a.L * g.tpb;
  return dim3(nx, a.H, a.B);
}
// rows of the last tile of a block (L > 128)
int tail_rows(const GenArgs& g) { return g.x.L <= kTile ? g.rows : g.x.L - (g.tpb - 1) * kTile; }

template <class K, class... A>
cudaError_t gen_launch(const Launch& lc, K kern, std::atomic<unsigned long long>* opted, int smem,
                       dim3 grid, A&&... args) {
  if (cudaError_t e = smem_opt_in(kern, smem, opted); e != cudaSuccess) return e;
  cudaError_t e = launch_k(kern, grid, dim3(kThreads), smem, lc.stream, args...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int NC>
cudaError_t bwd_nc(const Launch& lc, const AttnBwdArgs& ab) {
  const AttnArgs& a = ab.f;
  const GenArgs g = gen_args(lc, ab);
  const int tr = tail_rows(g);
  CUtensorMap mQ, mK, mV, mdO, dq, dk, dv, dqt, dkt, dvt;
  if (!gen_map(&mQ, a.Q, a.ld_qkv, a, kTile) || !gen_map(&mK, a.K, a.ld_qkv, a, kTile) ||
      !gen_map(&mV, a.V, a.ld_qkv, a, kTile) || !gen_map(&mdO, ab.dO, a.ld_o, a, kTile) ||
      !gen_map(&dq, ab.dQ, ab.ld_dqkv, a, g.rows) || !gen_map(&dk, ab.dK, ab.ld_dqkv, a, g.rows) ||
      !gen_map(&dv, ab.dV, ab.ld_dqkv, a, g.rows) || !gen_map(&dqt, ab.dQ, ab.ld_dqkv, a, tr) ||
      !gen_map(&dkt, ab.dK, ab.ld_dqkv, a, tr) || !gen_map(&dvt, ab.dV, ab.ld_dqkv, a, tr))
    return cudaErrorInvalidValue;
  static std::atomic<unsigned long long> o1{0}, o2{0}, o3{0};
  if (a.L <= kTile)
    return gen_launch(lc, attn_bwd_dkv_gen_kernel<NC, true>, &o1, dkv_smem<NC, true>() + kExtra, gen_grid(a, g), mQ, mK, mV, mdO, dq, dk, dv, dkt, dvt, g);
  cudaError_t e = gen_launch(lc, attn_bwd_dq_gen_kernel<NC>, &o2, dq_smem<NC>() + kExtra, gen_grid(a, g), mQ,
                             mK, mV, mdO, dq, dqt, g);
  if (e != cudaSuccess) return e;
  return gen_launch(lc, attn_bwd_dkv_gen_kernel<NC, false>, &o3, dkv_smem<NC, false>() + kExtra, gen_grid(a, g), mQ, mK, mV, mdO, dq, dk, dv, dkt, dvt, g);
}
}  // namespace

cudaError_t attn_bwd_gen(const Launch& lc, const AttnBwdArgs& a) {
  if (!attn_gen_supported(1, a.f.dh, a.f.L)) return cudaErrorNotSupported;
  return a.f.dh <= 64 ? bwd_nc<1>(lc, a) : bwd_nc<2>(lc, a);
}

}  // namespace bcmt
