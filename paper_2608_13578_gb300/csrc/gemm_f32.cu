// Dense products of fp32 tensors on the tcgen05 tensor cores, to fp32 accuracy.
//
// Every fp32 operand value is taken as the sum of three bf16 numbers x = h + m + l,
// which is exact (24 significand bits) from |x| = 2^-110 up; below, where l and then m
// fall under bf16's smallest subnormal 2^-133, x is off by up to 2^-134 (14 significant
// bits are left at 1e-36; the CUDA-core kernel keeps 24 down to 2^-126).  Of the nine
// partial products of two values the six of 2^-16 and above are formed, h h, h m, m h,
// m m, h l and l h; each is exact in fp32.  The dropped ones are below 2^-24 of the
// product.
// The tensor core's own accumulation is the weak point (its adds do not round
// to nearest), so no accumulator lives longer than one 64-deep K slice: h h goes
// to one TMEM accumulator and the five small products to a second, and the
// epilogue warps add both to fp32 sums in registers after every slice.  (The small
// products left in their accumulator for eight slices: 8192 x 1536 x 512 84 us instead
// of 88, but a relative error of 13.1e-8 instead of 12.7e-8 at K = 2048.)
// Against float64 (N(0,1) rows x N(0,1/K) weights) the relative 2-norm error is below
// that of the CUDA-core kernel with its chain of K fused multiply-adds: 7.1e-8 and 14.5e-8
// at K = 64, 9.0 and 40.5 at 512, 12.7 and 80.9 at 2048, 21.7 and 162 at 8192, and with rows
// scaled by powers of two the same down to 2^-110 (at 2^-114 56e-8 and 40e-8, at 2^-118
// 880e-8).
//
// One CTA per SM walks 128 x BN output tiles.  Warps 0-7 bring fp32 operands
// from global memory into registers a slice ahead, split them and write the
// three bf16 parts to a two-stage shared ring in the 128-byte-swizzled operand
// layout (K-major or MN-major, whichever way the operand lies in memory); warps
// 8-15 drain the accumulators (two, alternating) and store finished tiles through
// shared memory with TMA; warp 8 also issues the MMAs, one slice ahead of its
// draining (a warp of its own for that would cost every thread a quarter of its
// registers, and a loader that issues them holds up all the splitting).
// 8192 x 1536 x 512 takes 88 us (146 TFLOP/s of fp32 products; 122 us with a loader
// warp issuing the MMAs, 96 with their branch taken by lane number, see elect_one),
// 512 x 1536 x 8192 in 3 splits 73 us (177); the CUDA-core kernel took 497 and 749
// us.  A 64-deep slice of a 128 x 128 tile is 1536 cycles of tensor work and 2300 of
// shared-memory traffic (96 KB of parts written, 192 KB read by the 24 MMAs); it
// takes about 3700, the splitting and the hand-over between the two stages.
//
// A row or column holding an infinity (or a value above bf16's range) makes
// partial products like inf x 0: outputs that come out non-finite are recomputed
// as the CUDA-core kernel computes them, in K order.  A warp finds where its rows
// and columns hold non-finite values in one walk over K each (both of its 32 x 32
// runs: 4 K loads a lane, kScan of them in flight), and an output then takes the terms
// from the first of them to the last, or to the first NaN.  Outputs without any, whose
// products or sums left the range, take a whole chain, up to 64 K terms a lane: the
// only ones that can hold up a CTA for long (50 ns a term), so its waits go on while a
// chain makes progress (wait_beat).  A product with a NaN in every row, with all finite:
// 8192 x 1536 x 512 1.9 ms and 0.09, 512 x 1536 x 8192 0.76 and 0.16.
#include <string.h>

#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"
#include "tmap.h"

namespace bcmt {

namespace {
constexpr int kBM = 128, kBK = 64;
constexpr int kLoadThreads = 256;
constexpr int kThreads = 512;
constexpr int kStages = 2;

template <int BN>
struct Cfg {
  static constexpr int A_PART = kBM * kBK * 2;  // one bf16 part of a slice of A
  static constexpr int B_PART = BN * kBK * 2;
  static constexpr int STAGE = 3 * (A_PART + B_PART);
  static constexpr int OUT_OFF = kStages * STAGE;
  static constexpr int BAR_OFF = OUT_OFF + 8 * 4096;  // 4 KB of staging per epilogue warp
  static constexpr int SMEM = BAR_OFF + 1024 + 256;
  static constexpr int COLS = 4 * BN;  // two accumulators of (h h | rest)
};

struct Operand {
  const float* p;
  long sr, sk;  // element strides of the row (m or n) and of k; one of them is 1
};

// What a finished 32-column run of a row goes through before it is stored.
struct F32Store {
  __device__ __forceinline__ void apply(int, int, float*) const {}
};
struct F32Gate {  // Sec. 3.8
  __device__ __forceinline__ void apply(int, int, float* v) const {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = sigmoidf_(v[j]);
  }
};
struct F32Score {  // Sec. 3.4: the run's share of the pooling score H w_p
  const float* w_p;
  float* spart;
  long n_rows;
  __device__ __forceinline__ void apply(int row, int col, float* v) const {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
      const float4 w = __ldg(reinterpret_cast<const float4*>(w_p + col + j));
      s = fmaf(v[j], w.x, s);
      s = fmaf(v[j + 1], w.y, s);
      s = fmaf(v[j + 2], w.z, s);
      s = fmaf(v[j + 3], w.w, s);
    }
    spart[(long)(col / 32) * n_rows + row] = s;
  }
};

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&t);
}
// Two values' three parts as bf16 pairs.
__device__ __forceinline__ void split3(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack_bf16(a, b);
  a -= __uint_as_float(h << 16);
  b -= __uint_as_float(h & 0xffff0000u);
  m = pack_bf16(a, b);
  l = pack_bf16(a - __uint_as_float(m << 16), b - __uint_as_float(m & 0xffff0000u));
}

// 16 columns of the warp's TMEM lane quarter, without waiting.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// The loader's share of a ROWS x 64 slice of one operand: units of eight
// consecutive elements (along K when K-major, along the rows when MN-major),
// ROWS * 8 units over 256 threads.  Units past the operand's edge are zero.
template <int ROWS, bool MN>
struct Slice {
  static constexpr int U = ROWS * 8 / kLoadThreads;
  float v[U][8];
  __device__ __forceinline__ static void where(int i, int tid, int& r, int& k) {
    const int idx = tid + i * kLoadThreads;
    if (MN) {
      k = idx / (ROWS / 8);
      r = (idx % (ROWS / 8)) * 8;
    } else {
      r = idx / 8;
      k = (idx % 8) * 8;
    }
  }
  __device__ __forceinline__ void load(const Operand& o, int r0, int k0, int nr, int ke, int tid) {
#pragma unroll
    for (int i = 0; i < U; ++i) {
      int r, k;
      where(i, tid, r, k);
      r += r0;
      k += k0;
      if (r < nr && k < ke) {
        const float* p = o.p + (MN ? (long)k * o.sk + r : (long)r * o.sr + k);
        const float4 x = *reinterpret_cast<const float4*>(p);
        const float4 y = *reinterpret_cast<const float4*>(p + 4);
        v[i][0] = x.x; v[i][1] = x.y; v[i][2] = x.z; v[i][3] = x.w;
        v[i][4] = y.x; v[i][5] = y.y; v[i][6] = y.z; v[i][7] = y.w;
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[i][e] = 0.f;
      }
    }
  }
  // splits the units into the three parts at dst, dst + part, dst + 2 part
  __device__ __forceinline__ void store(uint8_t* dst, int part, int tid) const {
#pragma unroll
    for (int i = 0; i < U; ++i) {
      int r, k;
      where(i, tid, r, k);
      // MN-major: 64-row chunks of [64 k][128 B]; K-major: [rows][128 B]
      uint8_t* d = dst + (MN ? (r >> 6) * 8192 + tc::sw128_offset(k, (r & 63) >> 3)
                             : tc::sw128_offset(r, k >> 3));
      uint4 h, m, l;
      split3(v[i][0], v[i][1], h.x, m.x, l.x);
      split3(v[i][2], v[i][3], h.y, m.y, l.y);
      split3(v[i][4], v[i][5], h.z, m.z, l.z);
      split3(v[i][6], v[i][7], h.w, m.w, l.w);
      *reinterpret_cast<uint4*>(d) = h;
      *reinterpret_cast<uint4*>(d + part) = m;
      *reinterpret_cast<uint4*>(d + 2 * part) = l;
    }
  }
};

// ---- outputs that come out non-finite
__device__ __forceinline__ bool finite(float v) { return fabsf(v) <= 3.402823466e38f; }
// A wait for a warp that may be busy with such outputs, which can take longer than a
// wait's bound: it starts over as long as *beat moves.
__device__ __forceinline__ bool wait_beat(uint64_t* bar, uint32_t parity, unsigned* status,
                                          const volatile unsigned* beat) {
  const uint32_t addr = tc::smem_u32(bar);
  if (tc::mbar_try_wait(addr, parity)) return true;
  long long t0 = clock64();
  unsigned seen = *beat;
  while (true) {
    if (tc::mbar_try_wait(addr, parity)) return true;
    if (clock64() - t0 > tc::kWaitCycles) {
      const unsigned now = *beat;
      if (now == seen) {
        atomicOr(status, kStatusTimeout);
        return false;
      }
      seen = now;
      t0 = clock64();
    }
  }
}
constexpr int kScan = 16;      // terms whose loads go out together
constexpr int kBeat = 1 << 14;  // terms between two steps of the beat
// The k ranges [first, last) in steps of kScan outside which row r of the operand is
// finite (first = ke: everywhere).
__device__ __forceinline__ int2 non_finite_range(Operand o, int r, int kb, int ke, unsigned* beat) {
  int2 f = make_int2(ke, kb);
  const float* p = o.p + (long)r * o.sr;
  for (int k = kb; k < ke; k += kScan) {
    float x[kScan];
#pragma unroll
    for (int u = 0; u < kScan; ++u) x[u] = k + u < ke ? p[(long)(k + u) * o.sk] : 0.f;
    bool bad = false;
#pragma unroll
    for (int u = 0; u < kScan; ++u) bad |= !finite(x[u]);
    if (bad) f = make_int2(min(f.x, k), min(k + kScan, ke));
    if ((k & (kBeat - 1)) == 0) atomicAdd(beat, 1u);
  }
  return f;
}
// One output as the CUDA-core kernel forms it, a chain in K order.  `at`: where the
// operands' row and column hold non-finite values.  A term with one makes the sum
// non-finite for good, NaN stays NaN, and finite terms leave an infinity as it is: only
// the terms in that range matter, up to the first NaN; without any, up to overflow.
__device__ __forceinline__ float dot_in_order(Operand a, Operand b, int row, int col, int kb,
                                              int ke, int2 at, unsigned* beat) {
  const bool all = at.x >= ke;
  const int k1 = all ? ke : at.y;
  const float *pa = a.p + (long)row * a.sr, *pb = b.p + (long)col * b.sr;
  float s = 0.f;
  for (int k = all ? kb : at.x; k < k1; k += kScan) {
    float x[kScan], y[kScan];
#pragma unroll
    for (int u = 0; u < kScan; ++u) {
      x[u] = k + u < k1 ? pa[(long)(k + u) * a.sk] : 0.f;
      y[u] = k + u < k1 ? pb[(long)(k + u) * b.sk] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kScan; ++u) s = fmaf(x[u], y[u], s);
    if (s != s || (all && !finite(s))) break;
    if ((k & (kBeat - 1)) == 0) atomicAdd(beat, 1u);
  }
  return s;
}
// The non-finite outputs of a warp's 32 x 32 run from column col, the lane's row of it
// in v (a function of its own, values in shared memory: inlined it took the kernel's
// registers).
__device__ __noinline__ void redo_run(Operand a, Operand b, int row, int M, int col, int kb, int ke,
                                      float* v, unsigned* beat) {
  const int2 fr = non_finite_range(a, min(row, M - 1), kb, ke, beat),
             fc = non_finite_range(b, col + (threadIdx.x & 31), kb, ke, beat);
  for (int j = 0; j < 32; ++j) {
    const int2 at = make_int2(min(fr.x, __shfl_sync(0xffffffffu, fc.x, j)),
                              max(fr.y, __shfl_sync(0xffffffffu, fc.y, j)));
    if (row < M && !finite(v[j])) v[j] = dot_in_order(a, b, row, col + j, kb, ke, at, beat);
  }
}
}  // namespace

template <int BN, bool A_MN, bool B_MN, class Epi>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_f32_kernel(const Operand A, const Operand B, const __grid_constant__ CUtensorMap mC, int M,
                    int N, int K, int kps, int tiles_m, int tiles_n, int n_tiles, const Epi epi,
                    unsigned* status) {
  using C = Cfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF);
  uint64_t* empty = full + kStages;
  uint64_t* tfull = empty + kStages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tempty + 2);
  unsigned* beat = reinterpret_cast<unsigned*>(tslot + 1);
  const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&full[s], kLoadThreads / 32);
      tc::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(&tfull[a], 1);
      tc::mbar_init(&tempty[a], 8);
    }
    *beat = 0u;
    tc::fence_mbar_init();
    tc::prefetch_tmap(&mC);
  }
  if (warp == 8) {
    tc::tmem_alloc(tslot, C::COLS);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  pdl_enter();

  // a tile's origin and K range
  auto tile_at = [&](int tile, int& m0, int& n0, int& z, int& kb, int& ke) {
    const int per_z = tiles_m * tiles_n;
    z = tile / per_z;
    const int t = tile - z * per_z;
    n0 = (t / tiles_m) * BN;
    m0 = (t % tiles_m) * kBM;
    kb = z * kps * kBK;
    ke = min(K, kb + kps * kBK);
  };

  // slice `it`'s MMAs, into accumulator pair it & 1 (one thread)
  constexpr uint32_t idesc = tc::idesc_bf16(kBM, BN, A_MN ? 1 : 0, B_MN ? 1 : 0);
  auto issue = [&](int it) {
    const int s = it % kStages, acc = it & 1, use = it >> 1;
    if ((use > 0 && !wait_beat(&tempty[acc], (use - 1) & 1, status, beat)) ||
        !wait_beat(&full[s], (it / kStages) & 1, status, beat))
      return false;
    tc::fence_after_sync();
    const uint32_t sa = tc::smem_u32(smem + s * C::STAGE);
    const uint64_t ad = tc::sdesc(sa, A_MN ? 8192 : 16, 1024),
                   bd = tc::sdesc(sa + 3 * C::A_PART, B_MN ? 8192 : 16, 1024);
    const uint32_t d = tmem + (uint32_t)(acc * 2 * BN);
    auto product = [&](int pa, int pb, uint32_t dst, bool first) {
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk) {
        tc::mma_bf16(dst, tc::desc_at(ad, pa * C::A_PART + kk * (A_MN ? 2048 : 32)),
                     tc::desc_at(bd, pb * C::B_PART + kk * (B_MN ? 2048 : 32)), idesc,
                     first && kk == 0 ? 0u : 1u);
      }
    };
    product(0, 0, d, true);       // h h
    product(0, 2, d + BN, true);  // the small products, smallest first
    product(2, 0, d + BN, false);
    product(1, 1, d + BN, false);
    product(0, 1, d + BN, false);
    product(1, 0, d + BN, false);
    tc::mma_commit(&empty[s]);
    tc::mma_commit(&tfull[acc]);
    return true;
  };

  if (warp < 8) {
    // ---- loaders: a slice's registers are refilled right after they are split
    Slice<kBM, A_MN> a;
    Slice<BN, B_MN> b;
    int m0, n0, z, kb, ke, it = 0;
    int tile = blockIdx.x;
    if (tile < n_tiles) {
      tile_at(tile, m0, n0, z, kb, ke);
      a.load(A, m0, kb, M, ke, tid);
      b.load(B, n0, kb, N, ke, tid);
    }
    bool ok = true;
    while (tile < n_tiles && ok) {
      for (int k = kb; k < ke && ok; k += kBK, ++it) {
        // the slice after this one: in this tile or the CTA's next
        int nm = m0, nn = n0, nk = k + kBK, nke = ke;
        if (nk >= ke) {
          const int nt = tile + gridDim.x;
          int nz;
          if (nt < n_tiles)
            tile_at(nt, nm, nn, nz, nk, nke);
          else
            nke = nk;  // none: the loads below fetch nothing
        }
        const int s = it % kStages;
        if (it >= kStages && !wait_beat(&empty[s], ((it / kStages) - 1) & 1, status, beat)) {
          ok = false;
          break;
        }
        uint8_t* sa = smem + s * C::STAGE;
        a.store(sa, C::A_PART, tid);
        a.load(A, nm, nk, M, nke, tid);
        b.store(sa + 3 * C::A_PART, C::B_PART, tid);
        b.load(B, nn, nk, N, nke, tid);
        tc::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&full[s]);
      }
      tile += gridDim.x;
      if (tile < n_tiles) tile_at(tile, m0, n0, z, kb, ke);
    }
  } else {
    // ---- epilogue: warps 8-15, TMEM lane quarter warp % 4, half of the columns
    constexpr int NC = BN / 2;  // columns per warp
    const int q = warp & 3, c_beg = ((warp - 8) >> 2) * NC;
    uint8_t* sbuf = smem + C::OUT_OFF + (warp - 8) * 4096;
    const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c_beg;
    int it = 0, slices = 0;  // warp 8 also issues the MMAs, a slice ahead of its draining
    if (warp == 8)
      for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        int m0, n0, z, kb, ke;
        tile_at(tile, m0, n0, z, kb, ke);
        slices += (ke - kb + kBK - 1) / kBK;
      }
    if (slices > 0 && tc::elect_one()) issue(0);
    __syncwarp();
    bool ok = true;
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      int m0, n0, z, kb, ke;
      tile_at(tile, m0, n0, z, kb, ke);
      float acc[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = 0.f;
      for (int k = kb; k < ke; k += kBK, ++it) {
        const int ab = it & 1, use = it >> 1;
        if (it + 1 < slices && tc::elect_one()) issue(it + 1);
        __syncwarp();
        ok = wait_beat(&tfull[ab], use & 1, status, beat) && ok;
        tc::fence_after_sync();
#pragma unroll
        for (int c = 0; c < NC; c += 16) {
          uint32_t x[16], y[16];
          tmem_ld16_issue(trow + (uint32_t)(ab * 2 * BN + c), x);
          tmem_ld16_issue(trow + (uint32_t)(ab * 2 * BN + BN + c), y);
          tc::tmem_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j)
            acc[c + j] += __uint_as_float(x[j]) + __uint_as_float(y[j]);
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&tempty[ab]);
        if (!ok) break;
      }
      const int row0 = m0 + q * 32, row = row0 + lane;
#pragma unroll
      for (int c = 0; c < NC; c += 32) {
        const int col = n0 + c_beg + c;
        if (col < N) {  // N is a multiple of 32: runs are whole
          float v[32];
          bool fin = true;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            v[j] = acc[c + j];
            fin = fin && finite(v[j]);
          }
          if (__any_sync(0xffffffffu, row < M && !fin)) {
            if (lane == 0) tc::tma_store_wait_read<0>();
            __syncwarp();
            float* mine = reinterpret_cast<float*>(sbuf) + 32 * lane;
#pragma unroll
            for (int j = 0; j < 32; ++j) mine[j] = v[j];
            redo_run(A, B, row, M, col, kb, ke, mine, beat);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = mine[j];
          }
          if (row < M) {
            epi.apply(row, col, v);
          }
          if (lane == 0) tc::tma_store_wait_read<0>();
          __syncwarp();
#pragma unroll
          for (int u = 0; u < 8; ++u)
            *reinterpret_cast<float4*>(sbuf + lane * 128 + ((u ^ (lane & 7)) << 4)) =
                make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
          tc::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0 && ok) {
            tc::tma_store_3d(&mC, sbuf, col, row0, z);
            tc::tma_store_commit();
          }
        }
      }
    }
    if (lane == 0) tc::tma_store_wait_read<0>();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 8) tc::tmem_dealloc(tmem, C::COLS);
}

// ========================================================================= host
namespace {
template <int BN, bool A_MN, bool B_MN, class Epi>
cudaError_t launch(const Launch& lc, int M, int N, int K, const Operand& A, const Operand& B,
                   const Epi& epi, const EpiArgs& ea, int splits) {
  using C = Cfg<BN>;
  auto kern = gemm_f32_kernel<BN, A_MN, B_MN, Epi>;
  static std::atomic<unsigned long long> opted{0};
  if (cudaError_t e = smem_opt_in(kern, C::SMEM, &opted); e != cudaSuccess) return e;
  CUtensorMap mC;
  const long ss = ea.split_stride > 0 ? ea.split_stride : (long)M * ea.ldo;
  const uint64_t d[3] = {(uint64_t)N, (uint64_t)M, (uint64_t)splits};
  const uint64_t st[2] = {(uint64_t)ea.ldo * 4, (uint64_t)ss * 4};
  const uint32_t box[3] = {32, 32, 1};
  if (!make_tmap(&mC, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ea.out, 3, d, st, box,
                 CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  const int nkb = (K + kBK - 1) / kBK, kps = (nkb + splits - 1) / splits;
  const int tm = (M + kBM - 1) / kBM, tn = (N + BN - 1) / BN, tiles = tm * tn * splits;
  cudaError_t e = launch_k(kern, dim3(tiles < sm_count() ? tiles : sm_count()), dim3(kThreads), C::SMEM,
                           lc.stream, A, B, mC, M, N, K, kps, tm, tn, tiles, epi, lc.status);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int BN, bool A_MN, bool B_MN>
cudaError_t pick_epi(const Launch& lc, int M, int N, int K, const Operand& A, const Operand& B,
                     EpiKind epi, const EpiArgs& ea, int splits) {
  if (epi == EPI_STORE || epi == EPI_PARTIAL)
    return launch<BN, A_MN, B_MN>(lc, M, N, K, A, B, F32Store{}, ea, splits);
  // the fused epilogues, in the layout the layer uses them in
  if constexpr (!A_MN && B_MN) {
    if (epi == EPI_GATE) return launch<BN, A_MN, B_MN>(lc, M, N, K, A, B, F32Gate{}, ea, 1);
    if (epi == EPI_STORE_SCORE)
      return launch<BN, A_MN, B_MN>(lc, M, N, K, A, B,
                                    F32Score{(const float*)ea.w_p, ea.spart, M}, ea, 1);
  }
  return cudaErrorNotSupported;
}

template <int BN>
cudaError_t pick_layout(const Launch& lc, int M, int N, int K, const Operand& A, const Operand& B,
                        EpiKind epi, const EpiArgs& ea, int splits) {
  const bool am = A.sk != 1, bm = B.sk != 1;
  if (!am && bm) return pick_epi<BN, false, true>(lc, M, N, K, A, B, epi, ea, splits);
  if (!am && !bm) return pick_epi<BN, false, false>(lc, M, N, K, A, B, epi, ea, splits);
  if (am && bm) return pick_epi<BN, true, true>(lc, M, N, K, A, B, epi, ea, splits);
  return pick_epi<BN, true, false>(lc, M, N, K, A, B, epi, ea, splits);
}

// An operand the loaders can read in 16-byte pieces of eight elements.
bool loadable(const Operand& o, int rows, int K) {
  if (reinterpret_cast<uintptr_t>(o.p) % 16 != 0) return false;
  if (o.sk == 1) return o.sr % 4 == 0 && K % 8 == 0;
  return o.sr == 1 && o.sk % 4 == 0 && rows % 8 == 0;
}
}  // namespace

cudaError_t gemm_f32(const Launch& lc, int M, int N, int K, const void* A, long sam, long sak,
                     const void* B, long sbk, long sbn, EpiKind epi, const EpiArgs& ea,
                     int splits) {
  if (M < 1 || K < 1 || N % 64 != 0) return cudaErrorInvalidValue;
  const Operand a{(const float*)A, sam, sak}, b{(const float*)B, sbn, sbk};
  if (!tmap_encoder() || !loadable(a, M, K) || !loadable(b, N, K) || ea.ldo % 4 != 0 ||
      ea.split_stride % 4 != 0 || reinterpret_cast<uintptr_t>(ea.out) % 16 != 0)
    return cudaErrorNotSupported;
  splits = (epi == EPI_PARTIAL) ? effective_splits(K, splits) : 1;
  // 64-wide tiles spread a product that would leave half of the SMs idle
  const long tiles = (long)((M + kBM - 1) / kBM) * ((N + 127) / 128) * splits;
  if (tiles * 2 <= sm_count()) return pick_layout<64>(lc, M, N, K, a, b, epi, ea, splits);
  return pick_layout<128>(lc, M, N, K, a, b, epi, ea, splits);
}

}  // namespace bcmt
