// Backward of the intra-block causal attention on the tcgen05 tensor cores (Sec.
// 3.3) for blocks of several 128-token tiles, one pass: head widths DH in {16, 32,
// 64}, L = 128 m with m <= 8, 6, 2 (what TMEM holds).
//
// A CTA takes one (block, head) at a time and walks its pairs (key tile kt, query
// tile qt >= kt), kt outer, forming S = Q K^T and dP = dO V^T of a pair once for
// all three gradients:  dV_kt += P^T dO_qt, dK_kt += dS^T Q_qt, dQ_qt += dS K_kt.
// The block's Q and dO tiles stay in shared memory, K and V are double-buffered;
// TMEM holds S and dP (128 columns each), dK, dV of the current kt and dQ of every
// query tile.  dQ_kt is complete with key tile kt, so each kt ends by storing dQ,
// dK and dV of one tile.  One CTA per SM, persistent, with a warp for each job that
// would otherwise sit in the elementwise warps' way:
//   warps 0-7  a pair's S and dP into registers, P and dS to shared memory; a
//              finished tile's gradients to the buffers that held its operands
//              (warp w: TMEM lane quarter w % 4, half w / 4 of the key columns);
//   warp 8     issues the products: the next pair's S and dP as soon as the columns
//              are free, then the pair's three gradient products;
//   warp 9     stores finished tiles and loads the next block's into their place, so
//              a block's first loads run under the last one's work;
//   warps 10, 11  a tile's row statistics (Drow = dO . O) as soon as its slot is
//              loaded, from the O and dO tiles in shared memory (O through one buffer
//              of its own).  Read from global memory, a row a thread, they took as
//              long as all the rest: B16 T1024 D768 h12 L256 73 us, 65 so.
//
// What bounds it: a pair's 26 or more MMAs and their issue (about 1700 cycles at DH =
// 16) next to the elementwise chain (1400: 64 exponentials a thread, 64 KB of stores),
// the two overlapping but for the first pair of a block; at DH = 64, also the loads.
// Per pair 1.4 us at DH = 16, 3.9 us at DH = 64 (L 256, HBM's share 1.9 us).  The
// two-kernel form (attn_flash.cu, which keeps the shapes that do not fit) forms S and
// dP once for dQ and once more for dK, dV, and is the slower one from the smallest
// grid on: in us, two kernels -> this, for 8 / 152 / 608 (block, head)s:
//   DH 16, L 256     21 -> 13      27 -> 15      62 -> 33
//   DH 16, L 1024    57 -> 56     139 -> 60     441 -> 206
//   DH 32, L 512     38 -> 25      70 -> 27     195 -> 78
//   DH 64, L 256     25 -> 15      36 -> 21     111 -> 50
#include "attn_common.cuh"
#include "common.cuh"
#include "internal.h"
#include "tc.cuh"
#include "tmap.h"

namespace bcmt {
using namespace attn;

namespace {
constexpr int kTile = 128;
constexpr int kWorkers = 256;
constexpr int kMmaWarp = 8, kIoWarp = 9, kStatWarp = 10;
constexpr int kStatThreads = 64;
constexpr int kThreads = 384;
constexpr int kMaxM = 8;

struct BlkArgs {
  const float* lse;
  float* Drow;
  int T, H, L, m;
  int nb, total;  // blocks a sequence, (block, head, batch) items
  float scale;
  unsigned* status;
};

// P and dS (32 KB each), m tiles of Q and of dO, two of K and of V, one of O, the row
// statistics, barriers.
template <int DH> constexpr int blk_smem(int m) {
  return 1024 + 65536 + (2 * m + 5) * (int)Geo<DH>::tile + m * kTile * 8 + 384;
}

// Item it: heads of one block are neighbours (their rows share memory pages).
struct Item {
  int t0, h, b, nq;
  __device__ Item(const BlkArgs& a, int it) {
    const int x = it / a.H;
    h = it - x * a.H;
    b = x / a.nb;
    t0 = (x - b * a.nb) * a.L;
    nq = (min(a.L, a.T - t0) + kTile - 1) / kTile;
  }
};

// The bf16 tile row r as a TMA store takes it.
template <int DH>
__device__ __forceinline__ void blk_stage(uint8_t* tile, int r, const float* v) {
#pragma unroll
  for (int u = 0; u < DH / 8; ++u)
    *reinterpret_cast<uint4*>(tile + Geo<DH>::unit(r, u)) = pack8(v + 8 * u);
}
}  // namespace

template <int DH>
__global__ void __launch_bounds__(kThreads, 1)
    attn_bwd_blk_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
                        const __grid_constant__ CUtensorMap mV, const __grid_constant__ CUtensorMap mdO,
                        const __grid_constant__ CUtensorMap mdQ, const __grid_constant__ CUtensorMap mdK,
                        const __grid_constant__ CUtensorMap mdV, const __grid_constant__ CUtensorMap mO,
                        const __grid_constant__ BlkArgs a) {
  using G = Geo<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* sP = smem;
  uint8_t* sS = smem + 32768;
  uint8_t* sQ = smem + 65536;            // m tiles; a finished dQ tile is staged in its own
  uint8_t* sdO = sQ + a.m * G::tile;     // m tiles; dV likewise
  uint8_t* sK = sdO + a.m * G::tile;     // two; dK likewise
  uint8_t* sV = sK + 2 * G::tile;        // two
  uint8_t* sO = sV + 2 * G::tile;        // one
  float2* stat = reinterpret_cast<float2*>(sO + G::tile);  // [m * 128]: -lse log2 e, -Drow scale
  // Barriers in pairs are used in turn; c counts a CTA's key tiles, p its pairs and o
  // its query tiles, over all items.  Slots and statistics need no "free" barrier of
  // their own: a slot is loaded again, and its rows' statistics formed, only after
  // the gradients of its tile are stored.
  uint64_t* bar_q = reinterpret_cast<uint64_t*>(stat + a.m * kTile);  // [8] Q, dO tile loaded
  uint64_t* bar_k = bar_q + kMaxM;  // [2] K, V of key tile c loaded
  uint64_t* bar_e = bar_k + 2;      // [2] gradients of key tile c staged (8 warps)
  uint64_t* bar_t = bar_e + 2;      // [8] row statistics of a tile written (2 warps)
  uint64_t* bar_o = bar_t + kMaxM;  // O of query tile o loaded
  uint64_t* bar_s = bar_o + 1;      // S, dP of pair p
  uint64_t* bar_g = bar_s + 1;      // gradient products of pair p
  uint64_t* bar_r = bar_g + 1;      // S and dP of pair p in registers (8 warps)
  uint64_t* bar_p = bar_r + 1;      // P and dS of pair p in shared memory (8 warps)
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar_p + 1);
  constexpr uint32_t kDK = 256, kDV = kDK + DH, kDQ = kDV + DH;

  const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;
  const int step = gridDim.x;

  if (warp == 0 && tc::elect_one()) {
    for (int i = 0; i < kMaxM; ++i) {
      tc::mbar_init(&bar_q[i], 1);
      tc::mbar_init(&bar_t[i], kStatThreads / 32);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&bar_k[i], 1);
      tc::mbar_init(&bar_e[i], kWorkers / 32);
    }
    tc::mbar_init(bar_o, 1);
    tc::mbar_init(bar_s, 1);
    tc::mbar_init(bar_g, 1);
    tc::mbar_init(bar_r, kWorkers / 32);
    tc::mbar_init(bar_p, kWorkers / 32);
    tc::fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tc::tmem_alloc(tslot, 512);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  pdl_enter();
  bool ok = true;

  if (warp == kMmaWarp) {
    // ------------------------------------------------------------ products
    constexpr uint32_t idS = tc::idesc_bf16(128, 128, 0, 0), idMN = tc::idesc_bf16(128, DH, 1, 1),
                       idKM = tc::idesc_bf16(128, DH, 0, 1);
    // operand descriptors of the buffers' starts; a step along one adds its bytes / 16
    const uint64_t kq = G::kmaj(sQ, 0, 0), kg = G::kmaj(sdO, 0, 0), kk0 = G::kmaj(sK, 0, 0),
                   kv = G::kmaj(sV, 0, 0), nq0 = G::mnmaj(sQ, 0, 0), ng = G::mnmaj(sdO, 0, 0),
                   nk = G::mnmaj(sK, 0, 0), ap = tc::sdesc(tc::smem_u32(sP), 16384, 1024),
                   as = tc::sdesc(tc::smem_u32(sS), 16384, 1024), ks = p_kmaj(sS, 0, 0);
    constexpr uint32_t kT = G::tile / 16, kN = G::span;  // a tile; 16 rows of one
    uint32_t qph = 0;  // parity of each Q, dO slot's next load
    // S and dP of pair (kt, qt), whose key tile is the CTA's c-th, into columns 0 .. 255
    auto issue_s = [&](int c, int kt, int qt) {
      if (qt == kt) ok = ok && tc::mbar_wait(&bar_k[c & 1], (c >> 1) & 1, a.status);
      if (kt == 0) {
        ok = ok && tc::mbar_wait(&bar_q[qt], (qph >> qt) & 1, a.status);
        qph ^= 1u << qt;
      }
      tc::fence_after_sync();
      if (tc::elect_one()) {
        if (ok) {
          const uint64_t q0 = kq + qt * kT, g0 = kg + qt * kT, k0 = kk0 + (c & 1) * kT,
                         v0 = kv + (c & 1) * kT;
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk)
            tc::mma_bf16(tmem, q0 + kk * 2, k0 + kk * 2, idS, kk > 0 ? 1u : 0u);
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk)
            tc::mma_bf16(tmem + 128, g0 + kk * 2, v0 + kk * 2, idS, kk > 0 ? 1u : 0u);
        }
        tc::mma_commit(bar_s);
      }
      __syncwarp();
    };
    issue_s(0, 0, 0);
    int p = 0, c = 0;
    for (int it = blockIdx.x; it < a.total; it += step) {
      const int nq = Item(a, it).nq;
      for (int kt = 0; kt < nq; ++kt, ++c)
        for (int qt = kt; qt < nq; ++qt, ++p) {
          ok = ok && tc::mbar_wait(bar_r, p & 1, a.status);
          if (qt + 1 < nq)
            issue_s(c, kt, qt + 1);
          else if (kt + 1 < nq)
            issue_s(c + 1, kt + 1, kt + 1);
          ok = ok && tc::mbar_wait(bar_p, p & 1, a.status);
          tc::fence_after_sync();
          if (tc::elect_one()) {
            if (ok) {
              const uint64_t q0 = nq0 + qt * kT, g0 = ng + qt * kT, k0 = nk + (c & 1) * kT;
              const uint32_t dq = tmem + kDQ + (uint32_t)(qt * DH);
              const uint32_t first = qt == kt ? 0u : 1u, firstq = kt == 0 ? 0u : 1u;
#pragma unroll
              for (int kk = 0; kk < kTile / 16; ++kk)  // dV += P^T dO
                tc::mma_bf16(tmem + kDV, ap + kk * 128, g0 + kk * kN, idMN, kk > 0 ? 1u : first);
#pragma unroll
              for (int kk = 0; kk < kTile / 16; ++kk)  // dK += dS^T Q
                tc::mma_bf16(tmem + kDK, as + kk * 128, q0 + kk * kN, idMN, kk > 0 ? 1u : first);
#pragma unroll
              for (int kk = 0; kk < kTile / 16; ++kk)  // dQ += dS K
                tc::mma_bf16(dq, ks + (kk >> 2) * 1024 + (kk & 3) * 2, k0 + kk * kN, idKM,
                             kk > 0 ? 1u : firstq);
            }
            tc::mma_commit(bar_g);
          }
          __syncwarp();
          // the next block's first tiles may come in only after these products
          if (kt + 1 == nq && it + step < a.total) issue_s(c + 1, 0, 0);
        }
    }
  } else if (warp == kIoWarp) {
    // ------------------------------------------------------ loads and stores
    if (tc::elect_one()) {
      auto load_kv = [&](const Item& i, int kt, int c) {
        tc::mbar_arrive_expect_tx(&bar_k[c & 1], 2 * G::tile);
        tc::tma_load_3d(sK + (c & 1) * G::tile, &mK, &bar_k[c & 1], i.h * DH, i.t0 + kt * kTile, i.b);
        tc::tma_load_3d(sV + (c & 1) * G::tile, &mV, &bar_k[c & 1], i.h * DH, i.t0 + kt * kTile, i.b);
      };
      uint32_t qn = 0, qodd = 0;  // slots loaded so far, and those an odd number of times
      auto load_q = [&](const Item& i, int qt) {
        qn |= 1u << qt;
        qodd ^= 1u << qt;
        tc::mbar_arrive_expect_tx(&bar_q[qt], 2 * G::tile);
        tc::tma_load_3d(sQ + qt * G::tile, &mQ, &bar_q[qt], i.h * DH, i.t0 + qt * kTile, i.b);
        tc::tma_load_3d(sdO + qt * G::tile, &mdO, &bar_q[qt], i.h * DH, i.t0 + qt * kTile, i.b);
      };
      int kit = blockIdx.x, kkt = 0, kc = 0;  // the next key tile to load
      auto next_kv = [&]() {
        if (kit >= a.total) return;
        const Item i(a, kit);
        load_kv(i, kkt, kc++);
        if (++kkt == i.nq) kkt = 0, kit += step;
      };
      next_kv();
      {
        const Item i(a, blockIdx.x);
        load_q(i, 0);
        next_kv();
        for (int qt = 1; qt < i.nq; ++qt) load_q(i, qt);
      }
      int c = 0;
      for (int it = blockIdx.x; it < a.total; it += step) {
        const Item i(a, it);
        const bool more = it + step < a.total;
        const Item j(a, more ? it + step : it);
        for (int kt = 0; kt < i.nq; ++kt, ++c) {
          ok = ok && tc::mbar_wait(&bar_e[c & 1], (c >> 1) & 1, a.status);
          if (ok) {
            const int x = i.h * DH, t = i.t0 + kt * kTile;
            tc::tma_store_3d(&mdQ, sQ + kt * G::tile, x, t, i.b);
            tc::tma_store_3d(&mdK, sK + (c & 1) * G::tile, x, t, i.b);
            tc::tma_store_3d(&mdV, sdO + kt * G::tile, x, t, i.b);
            tc::tma_store_commit();
            tc::tma_store_wait_read<0>();  // the staging is read: its buffers are free
            next_kv();
            if (more && kt < j.nq) load_q(j, kt);
            if (more && kt + 1 == i.nq)
              for (int qt = i.nq; qt < j.nq; ++qt) load_q(j, qt);
          }
        }
      }
      if (!ok) {  // a wait has run out: what is on its way has to land before the CTA ends
        for (int qt = 0; qt < kMaxM; ++qt)
          if (qn >> qt & 1u) tc::mbar_wait(&bar_q[qt], (qodd >> qt & 1u) ^ 1u, a.status);
        for (int n = max(kc - 2, 0); n < kc; ++n)
          tc::mbar_wait(&bar_k[n & 1], (n >> 1) & 1, a.status);
      }
    }
    __syncwarp();
  } else if (warp >= kStatWarp) {
    // ------------------------------------- row statistics, from the O and dO tiles
    const float* lse = after_wait(a.lse);
    const int w = tid - kStatWarp * 32;
    struct At {  // a query tile of the CTA's items
      int it, qt;
    };
    auto after = [&](At t) {
      if (++t.qt == Item(a, t.it).nq) t = {t.it + step, 0};
      return t;
    };
    // its O on the way to shared memory and its log-sum-exp into v
    int loads = 0;  // of O, by the lane that issues them
    auto fetch = [&](At t, float* v) {
      if (t.it >= a.total) return;
      const Item j(a, t.it);
      const int r0 = j.t0 + t.qt * kTile;
      if (warp == kStatWarp && tc::elect_one() && ok) {
        ++loads;
        tc::mbar_arrive_expect_tx(bar_o, G::tile);
        tc::tma_load_3d(sO, &mO, bar_o, j.h * DH, r0, j.b);
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = r0 + w + u * kStatThreads;
        v[u] = i < a.T ? lse[((long)j.b * a.H + j.h) * a.T + i] : 0.f;
      }
    };
    uint32_t qph = 0;
    At t{(int)blockIdx.x, 0};
    float ls[2] = {0.f, 0.f};
    fetch(t, ls);
    for (int o = 0; t.it < a.total; ++o) {
      const Item j(a, t.it);
      ok = ok && tc::mbar_wait(bar_o, o & 1, a.status);
      ok = ok && tc::mbar_wait(&bar_q[t.qt], (qph >> t.qt) & 1, a.status);
      qph ^= 1u << t.qt;
      const uint8_t* g = sdO + t.qt * G::tile;
      float d[2] = {0.f, 0.f};
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int k = 0; k < DH / 8; ++k) {
          float ov[8], gv[8];
          load8(reinterpret_cast<const bf16*>(sO + G::unit(w + u * kStatThreads, k)), ov);
          load8(reinterpret_cast<const bf16*>(g + G::unit(w + u * kStatThreads, k)), gv);
#pragma unroll
          for (int e = 0; e < 8; ++e) d[u] = fmaf(ov[e], gv[e], d[u]);
        }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = t.qt * kTile + w + u * kStatThreads;
        float2 st = make_float2(0.f, 0.f);
        if (j.t0 + i < a.T) {
          a.Drow[((long)j.b * a.H + j.h) * a.T + j.t0 + i] = d[u];
          st = make_float2(-ls[u] * kLog2e, -d[u] * a.scale);
        }
        stat[i] = st;
      }
      tc::bar_sync(2, kStatThreads);  // O is read
      if (lane == 0) tc::mbar_arrive(&bar_t[t.qt]);
      t = after(t);
      fetch(t, ls);
    }
    if (!ok && loads > 0) tc::mbar_wait(bar_o, (loads - 1) & 1, a.status);  // as the loads above
    __syncwarp();
  } else {
    // ------------------------------------------------- elementwise, results
    const int q = warp & 3, hf = warp >> 2;
    const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
    const int r = q * 32 + lane;
    const float sl2 = a.scale * kLog2e;
    const float2 sl2x2 = make_float2(sl2, sl2), sc2 = make_float2(a.scale, a.scale);
    uint32_t tph = 0;  // parity of each tile's next statistics
    int p = 0, c = 0;
    for (int it = blockIdx.x; it < a.total; it += step) {
      const int nq = Item(a, it).nq;
      for (int kt = 0; kt < nq; ++kt, ++c) {
        for (int qt = kt; qt < nq; ++qt, ++p) {
          const bool diag = qt == kt;
          if (kt == 0) {
            ok = ok && tc::mbar_wait(&bar_t[qt], (tph >> qt) & 1, a.status);
            tph ^= 1u << qt;
          }
          const float2 st = stat[qt * kTile + r];
          ok = ok && tc::mbar_wait(bar_s, p & 1, a.status);
          tc::fence_after_sync();
          uint32_t s[2][32], dp[2][32];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            tc::tmem_ld32_issue(trow + (uint32_t)(hf * 64 + c * 32), s[c]);
            tc::tmem_ld32_issue(trow + 128u + (uint32_t)(hf * 64 + c * 32), dp[c]);
          }
          tc::tmem_wait();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(bar_r);  // the columns are free
          // P = 2^(s scale log2 e - lse log2 e), dS = P (dP scale - Drow scale): packed
          // bf16 pairs in place of the loaded words; keys past the row are 0 (diagonal)
          const float2 nl2 = make_float2(st.x, st.x), nd2 = make_float2(st.y, st.y);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int ch = 2 * hf + c;  // the warp's rows end in chunk q of the diagonal pair
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              const float2 e = __ffma2_rn(
                  make_float2(__uint_as_float(s[c][j]), __uint_as_float(s[c][j + 1])), sl2x2, nl2);
              const float2 d = __ffma2_rn(
                  make_float2(__uint_as_float(dp[c][j]), __uint_as_float(dp[c][j + 1])), sc2, nd2);
              const float x = ex2(e.x), y = ex2(e.y);
              s[c][j >> 1] = pack2(x, y);
              dp[c][j >> 1] = pack2(x * d.x, y * d.y);
            }
            if (diag && ch >= q) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int k = 32 * ch + 2 * j;
                const uint32_t keep = (k <= r ? 0xffffu : 0u) | (k < r ? 0xffff0000u : 0u);
                s[c][j] &= keep;
                dp[c][j] &= keep;
              }
            }
          }
          // the last pair's products have read P and dS
          if (p > 0) ok = ok && tc::mbar_wait(bar_g, (p - 1) & 1, a.status);
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              put_unit(sP, r, hf * 8 + c * 4 + u,
                       make_uint4(s[c][4 * u], s[c][4 * u + 1], s[c][4 * u + 2], s[c][4 * u + 3]));
              put_unit(sS, r, hf * 8 + c * 4 + u,
                       make_uint4(dp[c][4 * u], dp[c][4 * u + 1], dp[c][4 * u + 2], dp[c][4 * u + 3]));
            }
          tc::fence_proxy_async_smem();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(bar_p);
        }
        // ---- key tile kt is done: its dK and dV, and dQ of query tile kt
        ok = ok && tc::mbar_wait(bar_g, (p - 1) & 1, a.status);
        tc::fence_after_sync();
        {
          float v[DH];
          if (hf == 0) {
            tmem_row<DH>(trow + kDV, v);
            blk_stage<DH>(sdO + kt * G::tile, r, v);
            tmem_row<DH>(trow + kDQ + (uint32_t)(kt * DH), v);
            blk_stage<DH>(sQ + kt * G::tile, r, v);
          } else {
            tmem_row<DH>(trow + kDK, v);
            blk_stage<DH>(sK + (c & 1) * G::tile, r, v);
          }
        }
        tc::fence_proxy_async_smem();
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_e[c & 1]);
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) tc::tmem_dealloc(tmem, 512);
}

// ========================================================================= host
// TMEM: S, dP (256 columns), dK, dV, and dQ of each of the block's tiles.
bool attn_blk_supported(int dh, int L) {
  const int m = L / kTile;
  return L % kTile == 0 && m >= 2 && m <= kMaxM && 256 + (2 + m) * dh <= 512;
}

namespace {
template <int DH>
bool blk_map(CUtensorMap* m, const void* base, long ld, int D, int T, int B) {
  const uint64_t dims[3] = {(uint64_t)D, (uint64_t)T, (uint64_t)B};
  const uint64_t st[2] = {(uint64_t)ld * 2, (uint64_t)ld * 2 * (uint64_t)T};
  const uint32_t box[3] = {DH, kTile, 1};
  const CUtensorMapSwizzle sw = DH == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                                : DH == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                           : CU_TENSOR_MAP_SWIZZLE_32B;
  return make_tmap_bf16(m, base, 3, dims, st, box, sw);
}

template <int DH>
cudaError_t bwd_blk(const Launch& lc, const AttnBwdArgs& ab) {
  const AttnArgs& f = ab.f;
  const int D = f.H * DH;
  CUtensorMap m[8];
  if (!blk_map<DH>(&m[0], f.Q, f.ld_qkv, D, f.T, f.B) ||
      !blk_map<DH>(&m[1], f.K, f.ld_qkv, D, f.T, f.B) ||
      !blk_map<DH>(&m[2], f.V, f.ld_qkv, D, f.T, f.B) ||
      !blk_map<DH>(&m[3], ab.dO, f.ld_o, D, f.T, f.B) ||
      !blk_map<DH>(&m[4], ab.dQ, ab.ld_dqkv, D, f.T, f.B) ||
      !blk_map<DH>(&m[5], ab.dK, ab.ld_dqkv, D, f.T, f.B) ||
      !blk_map<DH>(&m[6], ab.dV, ab.ld_dqkv, D, f.T, f.B) ||
      !blk_map<DH>(&m[7], f.O, f.ld_o, D, f.T, f.B))
    return cudaErrorInvalidValue;
  BlkArgs a;
  a.lse = f.lse;
  a.Drow = ab.Drow;
  a.T = f.T;
  a.H = f.H;
  a.L = f.L;
  a.m = f.L / kTile;
  a.nb = (f.T + f.L - 1) / f.L;
  const long total = (long)a.nb * f.H * f.B;
  if (total > INT_MAX / 2) return cudaErrorNotSupported;
  a.total = (int)total;
  a.scale = 1.0f / sqrtf((float)DH);
  a.status = lc.status;
  auto kern = attn_bwd_blk_kernel<DH>;
  constexpr int most = blk_smem<DH>(DH == 64 ? 2 : DH == 32 ? 6 : kMaxM);
  static std::atomic<unsigned long long> opted{0};
  if (cudaError_t e = smem_opt_in(kern, most, &opted); e != cudaSuccess) return e;
  cudaError_t e = launch_k(kern, dim3(a.total < sm_count() ? a.total : sm_count()), dim3(kThreads),
                           blk_smem<DH>(a.m), lc.stream, m[0], m[1], m[2], m[3], m[4], m[5], m[6],
                           m[7], a);
  return e != cudaSuccess ? e : cudaGetLastError();
}
}  // namespace

cudaError_t attn_bwd_blk(const Launch& lc, const AttnBwdArgs& a) {
  if (!attn_blk_supported(a.f.dh, a.f.L)) return cudaErrorNotSupported;
  switch (a.f.dh) {
    case 16: return bwd_blk<16>(lc, a);
    case 32: return bwd_blk<32>(lc, a);
    case 64: return bwd_blk<64>(lc, a);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace bcmt
