// FP8 grouped expert GEMM on CTA pairs: e4m3 operands with fp32 block scales
// (tcgen05 cta_group::2 kind::f8f6f4, TMA, TMEM).
//
// The FP8 configuration of the MoE layer stores expert weights as e4m3 with
// one fp32 scale per 128 x 128 block and quantises activations per token per
// 128 channels.  The scales are arbitrary fp32 values, so they cannot ride in
// the tensor core's power-of-two block-scale path; instead every 128-wide K
// block is multiplied into one of kSlots TMEM partials and the epilogue warps
// add it, times (token scale x block scale), into fp32 register accumulators
// while the tensor core works on the next blocks.
//
// A tile is the 256 weight rows of an n-tile (M, 128 per CTA) and up to
// kMaxN token rows of one expert (N, half per CTA's shared memory), so a
// partial is N columns of each CTA's TMEM and four of them fit: the hand-back
// of a partial (commit, TMEM loads, arrival at the issuer) hides behind three
// K blocks, and its cost follows the rows of the tile.
//
// Roles of a CTA (384 threads):
//   warp 0 : weight producer; warp 10: token producer (one stage holds both)
//   warp 1 : TMEM; MMA issuer in CTA 0, tile scheduler in CTA 1
//   warps 2-9: epilogue; warp w owns TMEM lanes 32 (w % 4) .. and half of the
//            tile's tokens
//   warp 11: scales; the products (token scale x block scale) of each K block
//            go through a ring in shared memory
// Bounded waits as in the bf16 kernel.
#include "common.cuh"
#include "gemm_config.h"
#include "gemm_sched.cuh"
#include "internal.h"
#include "pair.cuh"

#include <cuda_fp8.h>

#include <mutex>

namespace asap {

namespace {

constexpr int kMaxN = kFp8PairRows;          // tokens of a tile
constexpr int kSlots = 4;                    // TMEM partials
constexpr int kSlotCols = 128;
constexpr int kStages = ASAP_RING_CTA2_F8;
constexpr int kWBytes = 128 * kFp8BK;        // 128 weight rows
constexpr int kXBytes = kMaxN / 2 * kFp8BK;  // up to kMaxN / 2 token rows
constexpr int kStageStride = kWBytes + kXBytes;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (4 + kEpiWarps);
constexpr int kXProdWarp = 2 + kEpiWarps;
constexpr int kScaleWarp = 3 + kEpiWarps;
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxU = kMaxN / 32;            // 16-token units per epilogue warp
static_assert(kMaxU == kFp8Boxes, "token boxes");
constexpr int kScaleSlots = 8;
constexpr int kScaleSlotBytes = kMaxN * 8;   // two products per token
constexpr int kBoxBytes = 16 * 128;          // [16 tokens, 64 bf16] store box
constexpr int kHalfStage = kMaxU * 2 * kBoxBytes;  // a half's tokens x 128 bf16 channels
constexpr int kStageBytes = 2 * kHalfStage;
constexpr int kAmaxBytes = 2 * 8 * kMaxN * 4;  // [tile parity][CTA, lane quarter][token]
constexpr int kNumBars = 2 * kStages + 2 * kSlots + 2 * kScaleSlots + 2 + 1;
constexpr int kQOff = (8 * kNumBars + 15) / 16 * 16;
constexpr int kBarBytes = kQOff + kPairQBytes + 16;
constexpr size_t kSmem = kStages * kStageStride + kStageBytes + kBarBytes + kScaleSlots * kScaleSlotBytes + kAmaxBytes +
                         sizeof(Sched);
static_assert(kSmem <= 227 * 1024, "shared memory budget");
static_assert(kSlots * kSlotCols <= 512 && kMaxN <= kSlotCols, "TMEM partials");
// consumers of a tile: both CTAs' producers, scale and epilogue warps, the MMA issuer
constexpr int kQueueConsumers = 2 * (3 + kEpiWarps) + 1;

struct PairMapsF8 {
  CUtensorMap x[2][kMaxU];  // problem; boxes of 16, 32, ... token rows
  CUtensorMap o[2];         // problem; [16 rows, 64 columns] boxes of the bf16 output
};

// kind::f8f6f4: fp32 accumulator (bits 4-5 = 1), A and B e4m3 (format 0), both
// K-major, N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__device__ __forceinline__ uint32_t idesc_f8(int n) {
  return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(256 >> 4) << 24);
}
__device__ __forceinline__ void tc_mma_f8_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// 16 lanes x 16 U columns in fragments (see tmem_ld_frag64).
template <int U>
__device__ __forceinline__ void tmem_ld_units(uint32_t taddr, uint32_t (&r)[8 * kMaxU]) {
  if constexpr (U == 4) {
    uint32_t(&a)[32] = *reinterpret_cast<uint32_t(*)[32]>(&r[0]);
    tmem_ld_frag64(taddr, a);
  } else {
    if constexpr (U >= 2) {
      uint32_t(&a)[16] = *reinterpret_cast<uint32_t(*)[16]>(&r[0]);
      tmem_ld_frag32(taddr, a);
    }
    if constexpr (U & 1) {
      uint32_t(&a)[8] = *reinterpret_cast<uint32_t(*)[8]>(&r[8 * (U - 1)]);
      tmem_ld_frag16(taddr + 16 * (U - 1), a);
    }
  }
}

struct Acc {
  // [lane half][8-token group][lane t/4 at 2 tokens, lane t/4 + 8 at 2 tokens]
  float v[2][2 * kMaxU][4];
};

// acc += scale x partial for the warp's 32 lanes and 16 U tokens; the slot is
// handed back (arrive) as soon as the partial is in registers.
template <int EPI, int U>
__device__ __forceinline__ void promote(Acc& acc, uint32_t taddr, uint32_t sc, int lane, uint32_t empty_bar,
                                        bool lead) {
  uint32_t p[2][8 * kMaxU];
  tmem_ld_units<U>(taddr, p[0]);
  tmem_ld_units<U>(taddr + (16u << 16), p[1]);
  tmem_ld_wait();
  tc_fence_before();
  __syncwarp();
  if (lane == 0) {
    if (lead) mbar_arrive(empty_bar);
    else mbar_arrive_pair(empty_bar);
  }
#pragma unroll
  for (int n = 0; n < 2 * U; ++n) {
    float s[4];  // lane t/4: tokens 0, 1; lane t/4 + 8: tokens 0, 1
    if constexpr (EPI == EPI_SWIGLU) {
      const uint32_t a = sc + (8 * n + 2 * (lane & 3)) * 8;
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(s[0]), "=f"(s[2]), "=f"(s[1]), "=f"(s[3])
                   : "r"(a)
                   : "memory");
    } else {
      const uint32_t a = sc + (8 * n + 2 * (lane & 3)) * 4;
      asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(s[0]), "=f"(s[1]) : "r"(a) : "memory");
      s[2] = s[0];
      s[3] = s[1];
    }
#pragma unroll
    for (int hl = 0; hl < 2; ++hl)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc.v[hl][n][i] = fmaf(s[i], __uint_as_float(p[hl][4 * n + i]), acc.v[hl][n][i]);
  }
}

// The 128 threads of one token half.
__device__ __forceinline__ void half_barrier(int half) {
  __syncwarp();
  asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
}
// Whether ok holds in every thread of the epilogue warps.
__device__ __forceinline__ bool epi_all(bool ok) {
  uint32_t r;
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 3, 256, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi) {
  return __nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
}

// Down GEMM: bf16 rows of the half's tokens [t0, t0 + 16 units), 128 channels
// of the CTA from column col0.
__device__ __forceinline__ void store_bf16(const Acc& acc, const PairTile& T, const GemmArgs& a, int units, int t0,
                                           int q, int lane, int half, int col0, uint32_t stage,
                                           const CUtensorMap* tm) {
  const int mx = lane >> 3, mi = lane & 7;
  const int tid = q * 32 + lane;
  // the previous tile's stores have read this half's staging boxes
  if (tid == 0) bulk_wait_group_read0();
  half_barrier(half);
  // box (unit u, 64-channel block b) at (2 u + b) kBoxBytes, 128-byte swizzle
#pragma unroll
  for (int n = 0; n < 2 * kMaxU; ++n) {
    if (n < 2 * units) {
      uint32_t pk[4];  // matrices (lane half, row half): channels 32 q + 8 mx ..
#pragma unroll
      for (int hl = 0; hl < 2; ++hl)
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) pk[2 * hl + rh] = pack_bf16x2(acc.v[hl][n][2 * rh], acc.v[hl][n][2 * rh + 1]);
      const int c = 4 * q + mx;
      const int r = 8 * (n & 1) + mi;
      stmatrix_x4_trans(stage + (n - (n & 1) + (c >> 3)) * kBoxBytes + r * 128 + (((c & 7) ^ mi) << 4), pk[0], pk[1],
                        pk[2], pk[3]);
    }
  }
  fence_proxy_async_smem();
  half_barrier(half);
  uint16_t* out = static_cast<uint16_t*>(T.p1 ? a.out1 : a.out0);
  const long long ldo = T.p1 ? a.ldo1 : a.ldo0;
  for (int u = 0; u < units; ++u) {
    const int left = T.rows - t0 - 16 * u;
    if (left >= 16) {
      if (tid == 0) {
        tma_store_2d(tm, stage + 2 * u * kBoxBytes, col0, T.row + t0 + 16 * u);
        tma_store_2d(tm, stage + (2 * u + 1) * kBoxBytes, col0 + 64, T.row + t0 + 16 * u);
      }
    } else if (left > 0) {
      // 16 threads per row
      for (int r = tid >> 4; r < left; r += 8) {
        const int j = tid & 7, b = (tid >> 3) & 1;
        uint4 v;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "r"(stage + (2 * u + b) * kBoxBytes + r * 128 + ((j ^ (r & 7)) << 4))
                     : "memory");
        *reinterpret_cast<uint4*>(out + (static_cast<long long>(T.row) + t0 + 16 * u + r) * ldo + col0 + 64 * b +
                                  8 * j) = v;
      }
    }
  }
  if (tid == 0) bulk_commit_group();
  __syncwarp();
}

// Gate/up GEMM: h = silu(gate) up of the half's tokens, e4m3 with one scale per
// token over the tile's 128 channels.  A channel block spans both CTAs (64
// channels each) and the four lane quarters: every warp reduces its 16 channels
// with shuffles and writes the partial maxima into both CTAs' tables.
// form_h leaves h in the accumulators and returns whether the maxima of both
// CTAs have arrived (false: the wait ran out); store_h quantises and stores.
__device__ __forceinline__ bool form_h(Acc& acc, const PairTile& T, int units, int t0, int q, int lane, int half,
                                       uint32_t rank, uint32_t amax, uint32_t peer_amax, uint32_t xbar,
                                       uint32_t peer_xbar, uint32_t xphase, volatile int* abort_flag) {
#pragma unroll
  for (int n = 0; n < 2 * kMaxU; ++n) {
    if (n < 2 * units) {
      float m0 = 0.f, m1 = 0.f;
#pragma unroll
      for (int hl = 0; hl < 2; ++hl) {
        float* v = acc.v[hl][n];
        // the first two entries become h of the two tokens
        v[0] = __fdividef(v[0], 1.0f + __expf(-v[0])) * v[2];
        v[1] = __fdividef(v[1], 1.0f + __expf(-v[1])) * v[3];
        m0 = fmaxf(m0, fabsf(v[0]));
        m1 = fmaxf(m1, fabsf(v[1]));
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o));
        m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
      }
      if (lane < 4) {
        const uint32_t o = ((rank * 4 + q) * kMaxN + t0 + 8 * n + 2 * lane) * 4;
        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(amax + o), "f"(m0), "f"(m1) : "memory");
        st_async_v2(peer_amax + o, peer_xbar, __float_as_uint(m0), __float_as_uint(m1));
      }
    }
  }
  __syncwarp();
  // every warp of this CTA arrives; the other CTA's four quarters of all T.n
  // tokens count as bytes
  if (lane == 0) {
    if (q == 0 && half == 0) mbar_arrive_expect_tx(xbar, 4 * 4 * T.n);
    else mbar_arrive(xbar);
  }
  return mbar_wait(xbar, xphase, abort_flag);
}

__device__ __forceinline__ void store_h(const Acc& acc, const PairTile& T, const Fp8Args& fa, int units, int t0, int q,
                                        int lane, int half, uint32_t rank, uint32_t stage, uint32_t amax) {
  const GemmArgs& a = fa.g;
  const int mx = lane >> 3, mi = lane & 7;
  const int tid = q * 32 + lane;
  uint32_t pk[2 * kMaxU];
#pragma unroll
  for (int n = 0; n < 2 * kMaxU; ++n) {
    pk[n] = 0;
    if (n < 2 * units) {
      const int tk = t0 + 8 * n + 2 * (lane & 3);
      float m0 = 0.f, m1 = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        float x, y;
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];"
                     : "=f"(x), "=f"(y)
                     : "r"(amax + (c * kMaxN + tk) * 4)
                     : "memory");
        m0 = fmaxf(m0, x);
        m1 = fmaxf(m1, y);
      }
      const float s0 = m0 > 0.f ? m0 / 448.0f : 1.0f, s1 = m1 > 0.f ? m1 / 448.0f : 1.0f;
      const float i0 = 1.0f / s0, i1 = 1.0f / s1;  // one division; the quotients are products
      // channels 2 j (lane half 0) and 2 j + 1 (lane half 1) of a token in one 16-bit element
      pk[n] = e4m3x2(acc.v[0][n][0] * i0, acc.v[1][n][0] * i0) | (e4m3x2(acc.v[0][n][1] * i1, acc.v[1][n][1] * i1) << 16);
      if (rank == 0 && q == 0 && lane < 4) {
        float* os = T.p1 ? fa.out_scale1 : fa.out_scale0;
        const int osld = T.p1 ? fa.o_sld1 : fa.o_sld0;
        const long long row = static_cast<long long>(T.row) + tk;
        if (tk < T.rows) os[row * osld + T.n_tile] = s0;
        if (tk + 1 < T.rows) os[(row + 1) * osld + T.n_tile] = s1;
      }
    }
  }
  half_barrier(half);  // the previous tile's rows have left this half's staging
  // token rows of 64 bytes, 16-byte chunk q at q ^ ((row / 2) % 4)
#pragma unroll
  for (int n = 0; n < 2 * kMaxU; n += 4) {
    if (n < 2 * units) {  // (groups past the tile's tokens are written, not stored)
      const int r = 8 * (n + mx) + mi;
      stmatrix_x4_trans(stage + r * 64 + ((q ^ ((r >> 1) & 3)) << 4), pk[n], pk[n + 1], pk[n + 2], pk[n + 3]);
    }
  }
  half_barrier(half);
  uint8_t* out = static_cast<uint8_t*>(T.p1 ? a.out1 : a.out0);
  const long long ldo = T.p1 ? a.ldo1 : a.ldo0;
  const int rows = min(16 * units, T.rows - t0);
  // 4 threads per row
  for (int r = tid >> 2; r < rows; r += 32) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(stage + r * 64 + (((tid & 3) ^ ((r >> 1) & 3)) << 4))
                 : "memory");
    *reinterpret_cast<uint4*>(out + (static_cast<long long>(T.row) + t0 + r) * ldo + T.n_tile * 128 +
                              static_cast<int>(rank) * 64 + (tid & 3) * 16) = v;
  }
  __syncwarp();
}

// Producer warp of the weights (W) or the tokens; both fill parts of the same
// stage, whose full barrier in CTA 0 expects the bytes of all four loads.
template <bool W>
__device__ __forceinline__ bool produce(const GemmArgs& args, const PairMapsF8& maps, const CUtensorMap* const* tmW,
                                        PairQueue& tq, uint32_t full, uint32_t empty, uint32_t ring_base,
                                        uint32_t rank, volatile int* abort_flag) {
  const bool issuer = elect_one();
  const uint64_t pol = l2_policy(W ? args.hint_b : args.hint_a);
  const uint32_t lead_full = pair_map(full, 0);
  Ring<kStages> r;
  bool ready = true;  // slot r.s has been seen to be free
  PairTile T;
  while (true) {
    if (!__all_sync(0xffffffffu, tq.pop(T, abort_flag))) return false;
    if (issuer) tq.release();
    ++tq.n;
    if (T.k_iters == 0) break;
    // weights: box (w_tile, kb) is rows (w_tile k_iters + kb) 256 of 128
    // bytes, this CTA loads its half of it; tokens: the CTA's half of the rows
    const int half = T.n / 2;
    const CUtensorMap* m = W ? tmW[T.p1] : &maps.x[T.p1][half / 16 - 1];
    const int y0 = W ? static_cast<int>(static_cast<long long>(T.w_tile) * T.k_iters * 256 + rank * 128)
                     : T.row + static_cast<int>(rank) * half;
    const uint32_t tx = 2 * (kWBytes + half * kFp8BK);
    for (int kb = 0; kb < T.k_iters; ++kb) {
      if (!__all_sync(0xffffffffu, ready) &&
          !__all_sync(0xffffffffu, mbar_wait(empty + 8u * r.s, r.phase ^ 1u, abort_flag)))
        return false;
      const int s = r.s;
      r.advance();
      ready = mbar_test_wait(empty + 8u * r.s, r.phase ^ 1u);
      if (issuer) {
        if (W && rank == 0) mbar_arrive_expect_tx(full + 8u * s, tx);
        tma_load_2d_pair(ring_base + s * kStageStride, m, lead_full + 8u * s, W ? 0 : kb * kFp8BK,
                         W ? y0 + kb * 256 : y0, pol);
      }
    }
  }
  // every commit on the ring's barriers has arrived before the CTA may leave
  for (int i = 0; i < kStages; ++i) {
    if (!__all_sync(0xffffffffu, mbar_wait(empty + 8u * r.s, r.phase ^ 1u, abort_flag))) return false;
    r.advance();
  }
  return true;
}

// Scale warp: the products of four K blocks at a time are formed from scales
// loaded one batch ahead and written into the ring, two per token for gate/up
// tiles (gate block, up block), one for down tiles (the CTA's block).
template <int EPI>
__device__ __forceinline__ bool produce_scales(const Fp8Args& fa, PairQueue& tq, uint32_t full, uint32_t empty,
                                               uint32_t ring_base, uint32_t rank, int lane, int layer,
                                               volatile int* abort_flag) {
  const GemmArgs& args = fa.g;
  constexpr int KB = 4, NT = kMaxN / 32;
  Ring<kScaleSlots> r;
  PairTile T;
  while (true) {
    if (!__all_sync(0xffffffffu, tq.pop(T, abort_flag))) return false;
    if (lane == 0) tq.release();
    ++tq.n;
    if (T.k_iters == 0) return true;
    const int sld = T.p1 ? fa.a_sld1 : fa.a_sld0;
    const float* as = T.p1 ? fa.a_scale1 : fa.a_scale0;
    const float* rows[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i)  // rows past the tile repeat its last one
      rows[i] = as + (static_cast<long long>(T.row) + min(32 * i + lane, T.rows - 1)) * sld;
    const float* bs = args.lref.table[layer].scale[T.p1 ? args.bmap1 - MAP_PAIR : args.bmap0 - MAP_PAIR] +
                      static_cast<long long>(T.group) * (T.p1 ? fa.b_nblk1 : fa.b_nblk0) * sld;
    const float* b0 = bs + static_cast<long long>(2 * T.n_tile + (EPI == EPI_SWIGLU ? 0 : rank)) * sld;
    const float* b1 = b0 + sld;  // the up block
    float ta[NT][KB], tg[KB], tu[KB];
    auto load = [&](int kb) {
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int k = min(kb + u, T.k_iters - 1);
        tg[u] = __ldg(b0 + k);
        tu[u] = EPI == EPI_SWIGLU ? __ldg(b1 + k) : 0.f;
#pragma unroll
        for (int i = 0; i < NT; ++i) ta[i][u] = 32 * i < T.n ? __ldg(rows[i] + k) : 0.f;
      }
    };
    load(0);
    for (int kb = 0; kb < T.k_iters; kb += KB) {
      float pg[NT][KB], pu[NT][KB];
#pragma unroll
      for (int u = 0; u < KB; ++u)
#pragma unroll
        for (int i = 0; i < NT; ++i) {
          pg[i][u] = ta[i][u] * tg[u];
          pu[i][u] = ta[i][u] * tu[u];
        }
      if (kb + KB < T.k_iters) load(kb + KB);
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        if (kb + u < T.k_iters) {
          if (!__all_sync(0xffffffffu, mbar_wait(empty + 8u * r.s, r.phase ^ 1u, abort_flag))) return false;
          const uint32_t d = ring_base + r.s * kScaleSlotBytes;
#pragma unroll
          for (int i = 0; i < NT; ++i) {
            if constexpr (EPI == EPI_SWIGLU)
              asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(d + (32 * i + lane) * 8), "f"(pg[i][u]),
                           "f"(pu[i][u])
                           : "memory");
            else
              asm volatile("st.shared.f32 [%0], %1;" ::"r"(d + (32 * i + lane) * 4), "f"(pg[i][u]) : "memory");
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(full + 8u * r.s);
          r.advance();
        }
      }
    }
  }
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    pair_gemm_fp8_kernel(const __grid_constant__ PairMapsF8 maps, const Fp8Args fa) {
  const GemmArgs& args = fa.g;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  if (base & 1023u) {  // the same in both CTAs: nothing is initialised yet
    if (threadIdx.x == 0) record_status(args.status, ST_SMEM_ALIGN);
    return;
  }
  const uint32_t stage = base + kStages * kStageStride;
  uint8_t* bar_area = smem_raw + kStages * kStageStride + kStageBytes;
  const uint32_t bar0 = smem_u32(bar_area);
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto pfull = [&](int s) { return bar0 + 8u * (2 * kStages + s); };
  auto pempty = [&](int s) { return bar0 + 8u * (2 * kStages + kSlots + s); };
  auto sfull = [&](int s) { return bar0 + 8u * (2 * kStages + 2 * kSlots + s); };
  auto sempty = [&](int s) { return bar0 + 8u * (2 * kStages + 2 * kSlots + kScaleSlots + s); };
  auto xchg = [&](int b) { return bar0 + 8u * (2 * kStages + 2 * kSlots + 2 * kScaleSlots + b); };
  const uint32_t drain = xchg(2);
  const uint32_t tq0 = bar0 + kQOff;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_area + kQOff + kPairQBytes);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* layer_slot = reinterpret_cast<int*>(tmem_slot + 2);
  const uint32_t scales = bar0 + kBarBytes;
  const uint32_t amax = scales + kScaleSlots * kScaleSlotBytes;
  Sched* sch = reinterpret_cast<Sched*>(bar_area + kBarBytes + kScaleSlots * kScaleSlotBytes + kAmaxBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = pair_rank();
  const bool leader = rank == 0;
  const int G = args.groups;
  const CUtensorMap* tmW[2] = {nullptr, nullptr};

  if (warp == 0) {
    const int l = load_layer(args.lref.layer, args.lref.n_layers, args.status, blockIdx.x == 0 && lane == 0);
    tmW[0] = &args.lref.table[l].map[args.bmap0];
    tmW[1] = &args.lref.table[l].map[args.bmap1];
    tensormap_acquire(tmW[0]);
    if (args.m1 > 0) tensormap_acquire(tmW[1]);
    if (lane == 0) {
      *layer_slot = l;
      for (int s = 0; s < kStages; ++s) {
        mbar_init(full(s), 1);
        mbar_init(empty(s), 1);
      }
      for (int s = 0; s < kSlots; ++s) {
        mbar_init(pfull(s), 1);
        mbar_init(pempty(s), 2 * kEpiWarps);
      }
      for (int s = 0; s < kScaleSlots; ++s) {
        mbar_init(sfull(s), 1);
        mbar_init(sempty(s), kEpiWarps);
      }
      mbar_init(xchg(0), kEpiWarps);
      mbar_init(xchg(1), kEpiWarps);
      mbar_init(drain, 1);
      for (int s = 0; s < kPairQ; ++s) {
        mbar_init(PairQueue::full(tq0, s), 1);
        mbar_init(PairQueue::empty(tq0, s), kQueueConsumers);
      }
      *abort_flag = 0;
      fence_barrier_init();
      tma_prefetch_desc(tmW[0]);
      if (args.m1 > 0) tma_prefetch_desc(tmW[1]);
    }
  } else if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
  } else if (warp == kScaleWarp && !leader) {
    build_schedule<kMaxN>(args, sch, G, lane);
  }
  tc_fence_before();
  __syncthreads();
  pair_sync();  // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the queue's home is CTA 1, whose warp 1 schedules
  PairQueue tq{tq0, pair_map(tq0, 1), !leader};
  // a role that gives up also ends the other CTA's waits
  auto give_up = [&]() {
    *abort_flag = 1;
    st_pair_u32(pair_map(smem_u32(const_cast<int*>(abort_flag)), rank ^ 1u), 1u);
    record_status(args.status, ST_WAIT_TIMEOUT);
  };

  if (warp == 0 || warp == kXProdWarp) {
    bool ok;
    if (warp == 0)
      ok = produce<true>(args, maps, tmW, tq, full(0), empty(0), base, rank, abort_flag);
    else
      ok = produce<false>(args, maps, tmW, tq, full(0), empty(0), base + kWBytes, rank, abort_flag);
    if (!ok) {
      if (lane == 0) give_up();
      drain_delay();
    }
  } else if (warp == kScaleWarp) {
    if (!produce_scales<EPI>(fa, tq, sfull(0), sempty(0), scales, rank, lane, *layer_slot, abort_flag) && lane == 0)
      give_up();
  } else if (warp == 1 && !leader) {
    // ------------------------------------------------------------ scheduler
    if (lane == 0 && !pair_schedule<kMaxN>(args, sch, G, tq, pair_map(tq0, 0), abort_flag)) give_up();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const bool issuer = elect_one();
    Ring<kStages> r;
    Ring<kSlots> p;
    bool ok = true, issued = false;
    bool ready = false;  // stage r.s has been seen to be loaded and slot p.s to be free
    const uint64_t wdesc = smem_desc_sw128(base), xdesc = smem_desc_sw128(base + kWBytes);
    PairTile T;
    while (ok) {
      ok = __all_sync(0xffffffffu, tq.pop(T, abort_flag));
      if (!ok) break;
      if (issuer) tq.release();
      ++tq.n;
      if (T.k_iters == 0) break;
      const uint32_t id = idesc_f8(T.n);
      for (int kb = 0; kb < T.k_iters; ++kb) {
        if (!__all_sync(0xffffffffu, ready)) {
          ok = mbar_wait(pempty(p.s), p.phase ^ 1u, abort_flag) && mbar_wait(full(r.s), r.phase, abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
        }
        tc_fence_after();
        const int cs = r.s, cp = p.s;
        r.advance();
        p.advance();
        ready = mbar_test_wait(pempty(p.s), p.phase ^ 1u) & mbar_test_wait(full(r.s), r.phase);
        if (issuer) {
          const uint64_t wd = wdesc + static_cast<uint32_t>(cs * (kStageStride >> 4));
          const uint64_t xd = xdesc + static_cast<uint32_t>(cs * (kStageStride >> 4));
          const uint32_t d = tmem_base + cp * kSlotCols;
#pragma unroll
          for (int kk = 0; kk < kFp8BK / 32; ++kk) tc_mma_f8_pair(d, wd + 2 * kk, xd + 2 * kk, id, kk > 0 ? 1u : 0u);
          tc_commit_pair(pfull(cp));
          tc_commit_pair(empty(cs));
        }
        issued = true;
      }
    }
    if (!ok) {
      if (lane == 0) give_up();
      if (issued) {
        int dummy = 0;
        if (elect_one()) tc_commit_pair(drain);
        __syncwarp();
        mbar_wait(drain, 0, &dummy);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;
    const int half = (warp - 2) >> 2;
    const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    const uint32_t pe = leader ? pempty(0) : pair_map(pempty(0), 0);
    const uint32_t my_stage = stage + half * kHalfStage;
    const uint32_t peer_amax = pair_map(amax, rank ^ 1u), peer_xchg = pair_map(xchg(0), rank ^ 1u);
    Ring<kSlots> p;
    Ring<kScaleSlots> sr;
    bool ok = true, ready = false;
    PairTile T;
    for (int it = 0;; ++it) {
      ok = __all_sync(0xffffffffu, tq.pop(T, abort_flag));
      if (ok) {
        if (lane == 0) tq.release();
        ++tq.n;
      }
      Acc acc;
      const int units = T.n / 32;
      const int t0 = half * (T.n / 2);
      if (ok && T.k_iters > 0) {
#pragma unroll
        for (int hl = 0; hl < 2; ++hl)
#pragma unroll
          for (int n = 0; n < 2 * kMaxU; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc.v[hl][n][i] = 0.f;
        for (int kb = 0; kb < T.k_iters; ++kb) {
          if (!__all_sync(0xffffffffu, ready)) {
            ok = mbar_wait(sfull(sr.s), sr.phase, abort_flag) && mbar_wait(pfull(p.s), p.phase, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
          }
          tc_fence_after();
          const uint32_t ta = lane_addr + p.s * kSlotCols + t0;
          const uint32_t sc = scales + sr.s * kScaleSlotBytes + t0 * (EPI == EPI_SWIGLU ? 8 : 4);
          const uint32_t eb = pe + 8u * p.s;
          const uint32_t sb = sempty(sr.s);
          p.advance();
          sr.advance();
          switch (units) {
            case 1: promote<EPI, 1>(acc, ta, sc, lane, eb, leader); break;
            case 2: promote<EPI, 2>(acc, ta, sc, lane, eb, leader); break;
            case 3: promote<EPI, 3>(acc, ta, sc, lane, eb, leader); break;
            default: promote<EPI, 4>(acc, ta, sc, lane, eb, leader); break;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(sb);
          ready = mbar_test_wait(sfull(sr.s), sr.phase) & mbar_test_wait(pfull(p.s), p.phase);
        }
      }
      // the eight warps share barriers below: all go on or none does
      if (!epi_all(ok)) {
        if (lane == 0) give_up();
        break;
      }
      if (T.k_iters == 0) break;
      if constexpr (EPI == EPI_SWIGLU) {
        const int b = it & 1;
        const uint32_t ao = static_cast<uint32_t>(b) * (kAmaxBytes / 2);
        ok = form_h(acc, T, units, t0, q, lane, half, rank, amax + ao, peer_amax + ao, xchg(b), peer_xchg + 8u * b,
                    (it >> 1) & 1, abort_flag);
        if (!epi_all(ok)) {
          if (lane == 0) give_up();
          break;
        }
        store_h(acc, T, fa, units, t0, q, lane, half, rank, my_stage, amax + ao);
      } else {
        store_bf16(acc, T, args, units, t0, q, lane, half, T.n_tile * 256 + static_cast<int>(rank) * 128, my_stage,
                   &maps.o[T.p1]);
      }
    }
    // the TMA stores are complete before the staging buffers go away
    if (q == 0 && lane == 0) bulk_wait_group0();
  }

  __syncwarp();
  tc_fence_before();
  pair_sync();  // neither CTA leaves while the other may still reach its shared memory or TMEM
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  });
  return fn;
}

}  // namespace

cudaError_t pair_gemm_fp8_set_attributes() {
  cudaError_t e = cudaFuncSetAttribute(pair_gemm_fp8_kernel<EPI_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(kSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pair_gemm_fp8_kernel<EPI_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kSmem));
  return e;
}

cudaError_t pair_gemm_fp8_launch(int epi, const CUtensorMap* maps, const Fp8Args& args, int pairs,
                                 cudaStream_t stream) {
  if (pairs <= 0) return cudaSuccess;
  PairMapsF8 pm;
  for (int p = 0; p < 2; ++p) {
    for (int i = 0; i < kMaxU; ++i) pm.x[p][i] = maps[kMaxU * p + i];
    pm.o[p] = maps[2 * kMaxU + p];
  }
  if (epi == EPI_SWIGLU)
    pair_gemm_fp8_kernel<EPI_SWIGLU><<<2 * pairs, kThreads, kSmem, stream>>>(pm, args);
  else
    pair_gemm_fp8_kernel<EPI_BF16><<<2 * pairs, kThreads, kSmem, stream>>>(pm, args);
  return cudaGetLastError();
}

bool encode_tmap_u8(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows,
                    std::string* err) {
  EncodeFn fn = encode_fn();
  if (!fn) {
    if (err) *err = "cuTensorMapEncodeTiled is not available from the driver";
    return false;
  }
  if ((reinterpret_cast<uintptr_t>(ptr) & 15u) != 0 || cols % 16 != 0 || rows == 0) {
    if (err) *err = "tensor for TMA must be 16-byte aligned with 16-byte row stride and >= 1 row";
    return false;
  }
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(kFp8BK), box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (err) *err = "cuTensorMapEncodeTiled failed with CUresult " + std::to_string(static_cast<int>(r));
    return false;
  }
  return true;
}

}  // namespace asap
