// Grouped GEMM with e4m3 operands and fp32 block scales on the sm_103a tensor
// core (tcgen05.mma kind::f8f6f4), fed by TMA.
//
// The FP8 configuration of the MoE layer stores expert weights as e4m3 with
// one fp32 scale per 128 x 128 block and quantises activations per token per
// 128 channels.  The scales are arbitrary fp32 values, so they cannot ride in
// the tensor core's power-of-two block-scale path; instead every 128-wide K
// block is multiplied into TMEM partials and the epilogue warps add them, times
// (token scale x block scale), into fp32 register accumulators while the tensor
// core works on the next block.
//
// A tile is up to 128 token rows of one expert (M) and the 256 weight rows of
// an n-tile (N), on one SM: handing a partial between the SMs of a CTA pair
// costs more than the operand reads that a pair saves (with 32-column
// chunks, the layer of 4096 tokens: tokens on M over a pair 3100 instead of
// 2615 us; weights on M, with the token scales through shared memory, 4005).  Every 128-wide K block has one of
// two 256-column partials.
//
// Roles (one CTA per SM, persistent, 384 threads):
//   warp 0 : weight producer, boxes [256 rows, 128 B]
//   warp 1 : TMEM; MMA issuer: per K block 4 x tcgen05.mma.cta_group::1
//            .kind::f8f6f4 M=128 N=256 K=32
//   warp 2 : token producer, boxes of 32 .. 128 rows
//   warp 3 : tile scheduler, one decoded tile ahead
//   warps 4-11: epilogue; warp w owns TMEM lanes 32 (w % 4) .. (tokens) and one
//            half of the columns; its warpgroups take registers from the first
//            (56 + 2 x 224 a thread): 128 accumulators, two 16-column chunks
// Tile schedule, masking and bounded waits as in the bf16 kernels.
//
// What bounds it (DeepSeek-V3 shape, Zipf routing, gate/up | down us of one
// call; before: roles issuing from lanes that had left their warps, every role
// decoding its tiles, 16 columns per TMEM wait): 128 tokens 576 | 292 (684 |
// 348), the weight stream; 4096 tokens 1435 | 786 (1778 | 1024) and 16384
// tokens 3650 | 2170 (4730 | 2796): the operands (48 KB per K block through L2
// and shared memory; with every second box left out 4096 tokens take 1231 |
// 687 and 16384 3267 | 1934) and the promotion (with a quarter of it 1412 | 747
// and 3279 | 1844).  In the promotion a 16-column chunk is on its way from TMEM
// while the one before it is added: 4096 tokens took 1469 | 821 with chunks of
// 32 and two on their way or none, which spill in either order (in the order
// used here 2224 | 1148); the row scales as 16-byte loads of four K blocks
// (moves and a branch per K block) 1560 | 851; looking at the next partial's
// barrier ahead 1437 | 788.  Weights prefetched into L2 4, 8 or 16 K blocks
// ahead: 1519, 1532 and 1553 for gate/up.
#include "common.cuh"
#include "gemm_config.h"
#include "gemm_sched.cuh"
#include "internal.h"
#include "pair.cuh"

#include <cuda_fp8.h>

#include <mutex>

namespace asap {

namespace {

constexpr int kSlots = 2;                    // TMEM partials of 256 columns
constexpr int kRows = 128;                   // token rows of a tile (M of the MMA)
constexpr int SW = ASAP_RING_F8_W, SX = ASAP_RING_F8_X;
constexpr int kWBytes = 256 * kFp8BK;
constexpr int kXBytes = kRows * kFp8BK;
constexpr int kCtrlWarps = 4;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (kCtrlWarps + kEpiWarps);
constexpr int kCtrlRegs = 56, kEpiRegs = 224;
static_assert(kCtrlRegs + 2 * kEpiRegs <= 3 * 168, "the register split stays within the launch's registers");
constexpr uint32_t kTmemCols = 512;
constexpr int kCols = 128;                   // accumulator columns per thread
constexpr int kStageWarpBytes = 32 * 4 * 16;  // output staging of an epilogue warp
constexpr int kAmaxBytes = 2 * 2 * kRows * 4;  // [tile parity][column half][row]
constexpr int kNumBars = 2 * SW + 2 * SX + 2 * kSlots + 2 + 1;
constexpr int kQOff = (8 * kNumBars + 15) / 16 * 16;
constexpr int kBarBytes = kQOff + kPairQBytes + 16;
constexpr size_t kSmem =
    SW * kWBytes + SX * kXBytes + kEpiWarps * kStageWarpBytes + kBarBytes + kAmaxBytes + sizeof(MixSched);
static_assert(kSmem <= 227 * 1024, "shared memory budget");
// consumers of a tile: the producers, the epilogue warps and the MMA issuer
constexpr int kQueueConsumers = 2 + kEpiWarps + 1;

struct MapsF8 {
  CUtensorMap x[2][kFp8Boxes];  // problem; boxes of 32, 64, 96 and 128 token rows
};

// kind::f8f6f4: fp32 accumulator (bits 4-5 = 1), A and B e4m3 (format 0), both
// K-major, N >> 3 in bits 17-22, M >> 4 in bits 24-28.
constexpr uint32_t kIdescF8 =
    (1u << 4) | (static_cast<uint32_t>(256 >> 3) << 17) | (static_cast<uint32_t>(kRows >> 4) << 24);
__device__ __forceinline__ void tc_mma_f8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(kIdescF8), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void add16(float* acc, const uint32_t (&v)[16], float s) {
#pragma unroll
  for (int j = 0; j < 16; ++j) acc[j] = fmaf(s, __uint_as_float(v[j]), acc[j]);
}

// One round of a warp's coalesced stores: lane l holds 4 chunks of 16 bytes
// (w, 16 words) of its row l.  Every lane writes them to the warp's 2 KB
// staging buffer (chunk j of row r at slot j ^ ((r / 2) % 4), so neither side
// of the exchange has bank conflicts), then lanes 4u .. 4u+3 store the 4
// chunks of rows u, u + 8, ...: each store instruction writes eight rows x 64
// contiguous bytes instead of 32 rows x 16 bytes.  Rows from ``valid_rows`` on
// are not stored.  out: the warp's first row at the round's first byte.
__device__ __forceinline__ void store_round4(const uint32_t* w, uint4* stage, int lane, uint8_t* out,
                                             long long ldo_bytes, int valid_rows) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    stage[lane * 4 + (j ^ ((lane >> 1) & 3))] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
  __syncwarp();
  const int ru = lane >> 2, cu = lane & 3;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = ru + 8 * k;
    const uint4 v = stage[r * 4 + (cu ^ ((r >> 1) & 3))];
    if (r < valid_rows) *reinterpret_cast<uint4*>(out + r * ldo_bytes + cu * 16) = v;
  }
  __syncwarp();
}

// Producer warp of the weights (W) or the tokens.  The whole warp runs the
// loop, one lane issues, and the next slot is looked at before this slot's
// load is issued.
template <bool W>
__device__ __forceinline__ bool produce(const GemmArgs& args, const MapsF8& maps, const CUtensorMap* const* tmW,
                                        PairQueue& tq, uint32_t full, uint32_t empty, uint32_t ring_base,
                                        volatile int* abort_flag) {
  constexpr int NS = W ? SW : SX;
  constexpr int stride = W ? kWBytes : kXBytes;
  const bool issuer = elect_one();
  const uint64_t pol = l2_policy(W ? args.hint_b : args.hint_a);
  Ring<NS> r;
  bool ready = true;  // slot r.s has been seen to be free
  uint32_t issued = 0;
  PairTile T;
  bool ok = true;
  while (ok) {
    ok = __all_sync(0xffffffffu, tq.pop(T, abort_flag));
    if (!ok) break;
    tq.release(issuer);
    if (T.k_iters == 0) return true;
    // weights: box (w_tile, kb) is rows (w_tile k_iters + kb) 256 of 128
    // bytes; tokens: a box of the next multiple of 32 rows
    const int box = (T.rows + 31) / 32;
    const CUtensorMap* m = W ? tmW[T.p1] : &maps.x[T.p1][box - 1];
    const int y0 = W ? T.w_tile * T.k_iters * 256 : T.row;
    const uint32_t tx = W ? kWBytes : box * 32 * kFp8BK;
    for (int kb = 0; kb < T.k_iters; ++kb) {
      if (!__all_sync(0xffffffffu, ready)) {
        ok = __all_sync(0xffffffffu, mbar_wait(empty + 8u * r.s, r.phase ^ 1u, abort_flag));
        if (!ok) break;
      }
      const int s = r.s;
      r.advance();
      ready = mbar_test_wait(empty + 8u * r.s, r.phase ^ 1u);
      if (issuer) {
        mbar_arrive_expect_tx(full + 8u * s, tx);
        tma_load_2d(ring_base + s * stride, m, full + 8u * s, W ? 0 : kb * kFp8BK, W ? y0 + kb * 256 : y0, pol);
      }
      issued = min(issued + 1, static_cast<uint32_t>(NS));
    }
  }
  // the copies in flight land before the CTA's memory goes away: the last
  // ``issued`` slots, oldest first
  int dummy = 0;
  for (uint32_t i = issued; i > 0; --i) {
    const int back = r.s - static_cast<int>(i);
    mbar_wait(full + 8u * (back < 0 ? back + NS : back), back < 0 ? r.phase ^ 1u : r.phase, &dummy);
  }
  return false;
}

template <int EPI>
__global__ void __launch_bounds__(kThreads, 1)
    grouped_gemm_fp8_kernel(const __grid_constant__ MapsF8 maps, const Fp8Args fa) {
  const GemmArgs& args = fa.g;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  if (base & 1023u) {  // uniform for the CTA: nothing is initialised yet
    pdl_wait();
    if (threadIdx.x == 0) record_status(args.status, ST_SMEM_ALIGN);
    return;
  }
  const uint32_t sW = base, sX = base + SW * kWBytes;
  uint4* stage_all = reinterpret_cast<uint4*>(smem_raw + SW * kWBytes + SX * kXBytes);
  uint8_t* bar_area = smem_raw + SW * kWBytes + SX * kXBytes + kEpiWarps * kStageWarpBytes;
  const uint32_t bar0 = smem_u32(bar_area);
  auto bar = [&](int first, int s) { return bar0 + 8u * (first + s); };
  // full and empty of the weight and token rings, full and empty of the
  // partials, amax exchange (per tile parity), drain
  constexpr int B_FW = 0, B_EW = SW, B_FX = 2 * SW, B_EX = 2 * SW + SX, B_PF = 2 * SW + 2 * SX, B_PE = B_PF + kSlots,
                B_XC = B_PE + kSlots, B_DR = B_XC + 2;
  const uint32_t tq0 = bar0 + kQOff;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_area + kQOff + kPairQBytes);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* layer_slot = reinterpret_cast<int*>(tmem_slot + 2);
  float* amax_x = reinterpret_cast<float*>(bar_area + kBarBytes);  // [2][2][kRows]
  MixSched* sch = reinterpret_cast<MixSched*>(bar_area + kBarBytes + kAmaxBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = args.groups;
  const CUtensorMap* tmW[2] = {nullptr, nullptr};

  if (warp == 0) {
    if (lane == 0) {
      // one arrival (or commit) each, but for the epilogue's: its warps per
      // partial, its threads per exchange
      for (int i = 0; i < kNumBars; ++i)
        mbar_init(bar(0, i), i >= B_PE && i < B_XC ? kEpiWarps : i >= B_XC && i < B_DR ? 32 * kEpiWarps : 1);
      for (int s = 0; s < kPairQ; ++s) {
        mbar_init(PairQueue::full(tq0, s), 1);
        mbar_init(PairQueue::empty(tq0, s), kQueueConsumers);
      }
      *abort_flag = 0;
      fence_barrier_init();
    }
    pdl_wait();
    const int l = load_layer(args.lref.layer, args.lref.n_layers, args.status, blockIdx.x == 0 && lane == 0);
    tmW[0] = &args.lref.table[l].map[args.bmap0];
    tmW[1] = &args.lref.table[l].map[args.bmap1];
    tensormap_acquire(tmW[0]);
    if (args.m1 > 0) tensormap_acquire(tmW[1]);
    if (lane == 0) {
      *layer_slot = l;
      tma_prefetch_desc(tmW[0]);
      if (args.m1 > 0) tma_prefetch_desc(tmW[1]);
    }
  } else if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  } else if (warp == 3) {
    pdl_wait();
    build_mix_schedule<kRows>(args, sch, G, lane);
  }
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  PairQueue tq{tq0, tq0, true};
  auto give_up = [&]() {
    *abort_flag = 1;
    record_status(args.status, ST_WAIT_TIMEOUT);
  };

  if (warp < kCtrlWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kCtrlRegs));
    if (warp == 0 || warp == 2) {
      const bool ok = warp == 0 ? produce<true>(args, maps, tmW, tq, bar(B_FW, 0), bar(B_EW, 0), sW, abort_flag)
                                : produce<false>(args, maps, tmW, tq, bar(B_FX, 0), bar(B_EX, 0), sX, abort_flag);
      if (!ok && lane == 0) give_up();
    } else if (warp == 3) {
      // ------------------------------------------------------------ scheduler
      if (lane == 0) {
        if (!tile_schedule<kRows>(args, sch, G, tq, abort_flag)) give_up();
        pdl_launch();  // no tiles left for this CTA
      }
    } else {
      // ------------------------------------------------------------ MMA issuer
      const bool issuer = elect_one();
      Ring<SW> rw;
      Ring<SX> rx;
      Ring<kSlots> p;
      bool ok = true, issued = false;
      const uint64_t wdesc = smem_desc_sw128(sW), xdesc = smem_desc_sw128(sX);
      PairTile T;
      while (ok) {
        ok = __all_sync(0xffffffffu, tq.pop(T, abort_flag));
        if (!ok) break;
        tq.release(issuer);
        if (T.k_iters == 0) break;
        for (int kb = 0; kb < T.k_iters; ++kb) {
          // the stages' operands and the partial, a third of the lanes each
          ok = mbar_wait_all(lane < 10 ? bar(B_FX, rx.s) : lane < 20 ? bar(B_FW, rw.s) : bar(B_PE, p.s),
                             lane < 10 ? rx.phase : lane < 20 ? rw.phase : p.phase ^ 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
          if (issuer) {
            const uint64_t wd = wdesc + static_cast<uint32_t>(rw.s * (kWBytes >> 4));
            const uint64_t xd = xdesc + static_cast<uint32_t>(rx.s * (kXBytes >> 4));
            const uint32_t d = tmem_base + p.s * 256;
#pragma unroll
            for (int kk = 0; kk < kFp8BK / 32; ++kk) tc_mma_f8(d, xd + 2 * kk, wd + 2 * kk, kk > 0 ? 1u : 0u);
            tc_commit(bar(B_PF, p.s));
            tc_commit(bar(B_EW, rw.s));
            tc_commit(bar(B_EX, rx.s));
          }
          __syncwarp();
          issued = true;
          rw.advance();
          rx.advance();
          p.advance();
        }
      }
      if (!ok) {
        if (lane == 0) give_up();
        if (issued) {
          int dummy = 0;
          if (elect_one()) tc_commit(bar(B_DR, 0));
          __syncwarp();
          mbar_wait(bar(B_DR, 0), 0, &dummy);
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // warp w reads TMEM lanes 32 q .. (rows) and one half of the columns:
    // SwiGLU tiles: gate columns [64 cq, +64) and the matching up columns
    // 128 + [64 cq, +64), i.e. h channels [64 cq, +64) of the tile; plain
    // tiles: columns [128 cq, +128)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
    const int q = warp & 3;
    const int cq = (warp - kCtrlWarps) >> 2;
    const int r = q * 32 + lane;
    const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    uint4* stage = stage_all + (warp - kCtrlWarps) * (kStageWarpBytes / 16);
    constexpr int kHi = EPI == EPI_SWIGLU ? 128 : 64;  // column offset of the thread's second half
    const uint32_t col = lane_addr + cq * (EPI == EPI_SWIGLU ? 64 : 128);
    const int layer = *layer_slot;
    Ring<kSlots> p;
    bool ok = true;
    PairTile T, next;
    // the scales of a tile's first two K blocks are loaded (L2 latency) before
    // the tile in front of it is written, the others two K blocks ahead
    float a0 = 0.f, l0 = 0.f, h0 = 0.f, a1 = 0.f, l1 = 0.f, h1 = 0.f;
    const float *arow = nullptr, *bs_lo = nullptr, *bs_hi = nullptr;
    auto ld_scales = [&](int kb, int k_iters, float& a, float& bl, float& bh) {
      if (kb < k_iters) {
        a = ld_dep(arow + kb);
        bl = __ldg(bs_lo + kb);
        bh = EPI == EPI_SWIGLU ? __ldg(bs_hi + kb) : 0.f;
      }
    };
    auto pop_next = [&]() -> bool {
      const bool got = __all_sync(0xffffffffu, tq.pop(next, abort_flag));
      if (!got) return false;
      tq.release(lane == 0);
      const int valid = next.rows - q * 32;
      if (next.k_iters == 0 || valid <= 0) return true;
      const int sld = next.p1 ? fa.a_sld1 : fa.a_sld0;
      arow = (next.p1 ? fa.a_scale1 : fa.a_scale0) +
             (static_cast<long long>(next.row) + q * 32 + min(lane, valid - 1)) * sld;  // masked rows: the last valid one
      // scale rows of this warp's columns: SwiGLU tiles hold gate block nt
      // (scale row 2 nt) and up block nt (2 nt + 1); plain tiles blocks 2 nt, 2 nt + 1
      bs_lo = args.lref.table[layer].scale[next.p1 ? args.bmap1 : args.bmap0] +
              (static_cast<long long>(next.group) * (next.p1 ? fa.b_nblk1 : fa.b_nblk0) + 2 * next.n_tile +
               (EPI == EPI_SWIGLU ? 0 : cq)) *
                  sld;
      bs_hi = bs_lo + sld;
      ld_scales(0, next.k_iters, a0, l0, h0);
      ld_scales(1, next.k_iters, a1, l1, h1);
      return true;
    };
    ok = pop_next();
    for (int it = 0; ok; ++it) {
      T = next;
      if (T.k_iters == 0) break;
      const int valid_rows = T.rows - q * 32;  // rows of this warp
      const long long row = static_cast<long long>(T.row) + r;
      // a warp without rows only hands the partials back
      if (valid_rows <= 0) {
        for (int kb = 0; kb < T.k_iters && ok; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(bar(B_PF, p.s), p.phase, abort_flag));
          if (ok && lane == 0) mbar_arrive(bar(B_PE, p.s));
          p.advance();
        }
        if (EPI == EPI_SWIGLU && ok) mbar_arrive(bar(B_XC, it & 1));
        ok = ok && pop_next();
        continue;
      }
      float acc[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) acc[j] = 0.f;
      uint32_t c0[16], c1[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) c1[j] = 0u;
      float s_prev = 0.f;
      for (int kb = 0; kb < T.k_iters; ++kb) {
        const float s_lo = a0 * l0;
        const float s_hi = EPI == EPI_SWIGLU ? a0 * h0 : s_lo;
        a0 = a1;
        l0 = l1;
        h0 = h1;
        ld_scales(kb + 2, T.k_iters, a1, l1, h1);
        if (!__all_sync(0xffffffffu, mbar_wait(bar(B_PF, p.s), p.phase, abort_flag))) {
          ok = false;
          break;
        }
        tc_fence_after();
        // eight chunks of 16 columns: one is on its way from TMEM while the
        // one before it is added, across K blocks too; the partial is handed
        // back when its last chunk is in registers
        const uint32_t ta = col + p.s * 256;
        tmem_ld16(ta, c0);
        add16(acc + 112, c1, s_prev);
        tmem_ld_wait();
        tmem_ld16(ta + 16, c1);
        add16(acc + 0, c0, s_lo);
        tmem_ld_wait();
        tmem_ld16(ta + 32, c0);
        add16(acc + 16, c1, s_lo);
        tmem_ld_wait();
        tmem_ld16(ta + 48, c1);
        add16(acc + 32, c0, s_lo);
        tmem_ld_wait();
        tmem_ld16(ta + kHi, c0);
        add16(acc + 48, c1, s_lo);
        tmem_ld_wait();
        tmem_ld16(ta + kHi + 16, c1);
        add16(acc + 64, c0, s_hi);
        tmem_ld_wait();
        tmem_ld16(ta + kHi + 32, c0);
        add16(acc + 80, c1, s_hi);
        tmem_ld_wait();
        tmem_ld16(ta + kHi + 48, c1);
        add16(acc + 96, c0, s_hi);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_PE, p.s));
        s_prev = s_hi;
        p.advance();
      }
      add16(acc + 112, c1, s_prev);
      ok = ok && pop_next();
      if (!ok) break;
      const long long wrow0 = row - lane;
      if constexpr (EPI == EPI_SWIGLU) {
        // h = silu(gate) * up for 64 channels, then e4m3 with one scale per
        // row per 128 channels (this tile's 128 h columns): the two column
        // halves of a row exchange their partial amax through shared memory
        float amax = 0.f;
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          const float gv = acc[j];
          const float hv = __fdividef(gv, 1.0f + __expf(-gv)) * acc[64 + j];
          acc[j] = hv;
          amax = fmaxf(amax, fabsf(hv));
        }
        float* xs = amax_x + (it & 1) * 256;
        xs[cq * 128 + r] = amax;
        mbar_arrive(bar(B_XC, it & 1));
        if (!__all_sync(0xffffffffu, mbar_wait(bar(B_XC, it & 1), (it >> 1) & 1, abort_flag))) {
          ok = false;
          break;
        }
        amax = fmaxf(amax, xs[(cq ^ 1) * 128 + r]);
        const float scale = amax > 0.f ? amax / 448.0f : 1.0f;
        const float inv = 1.0f / scale;  // one division; the quotients below are products
        // 64 e4m3 values: 4 chunks of 16 bytes, one staged round
        uint32_t w[16];
#pragma unroll
        for (int j = 0; j < 64; j += 4) {
          const __nv_fp8x2_storage_t lo = __nv_cvt_float2_to_fp8x2(make_float2(acc[j] * inv, acc[j + 1] * inv),
                                                                    __NV_SATFINITE, __NV_E4M3);
          const __nv_fp8x2_storage_t hi = __nv_cvt_float2_to_fp8x2(make_float2(acc[j + 2] * inv, acc[j + 3] * inv),
                                                                    __NV_SATFINITE, __NV_E4M3);
          w[j / 4] = static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
        }
        uint8_t* out = static_cast<uint8_t*>(T.p1 ? args.out1 : args.out0);
        const long long ldo = T.p1 ? args.ldo1 : args.ldo0;
        store_round4(w, stage, lane, out + wrow0 * ldo + static_cast<long long>(T.n_tile) * 128 + cq * 64, ldo,
                     valid_rows);
        if (lane < valid_rows && cq == 0) {
          float* os = T.p1 ? fa.out_scale1 : fa.out_scale0;
          const int osld = T.p1 ? fa.o_sld1 : fa.o_sld0;
          os[row * osld + T.n_tile] = scale;
        }
      } else {
        // 128 bf16 values: 16 chunks, four staged rounds of 64 bytes
        uint8_t* out = static_cast<uint8_t*>(T.p1 ? args.out1 : args.out0);
        const long long ldo_b = 2 * (T.p1 ? args.ldo1 : args.ldo0);
        uint8_t* out_w = out + wrow0 * ldo_b + 2 * (static_cast<long long>(T.n_tile) * 256 + cq * 128);
#pragma unroll
        for (int rd = 0; rd < 4; ++rd) {
          uint32_t w[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) w[i] = pack_bf16x2(acc[32 * rd + 2 * i], acc[32 * rd + 2 * i + 1]);
          store_round4(w, stage, lane, out_w + 64 * rd, ldo_b, valid_rows);
        }
      }
    }
    if (!ok && lane == 0) give_up();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
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

cudaError_t fp8_gemm_set_attributes() {
  cudaError_t e = cudaFuncSetAttribute(grouped_gemm_fp8_kernel<EPI_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(kSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(grouped_gemm_fp8_kernel<EPI_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kSmem));
  return e;
}

cudaError_t fp8_gemm_launch(int epi, const CUtensorMap* maps, const Fp8Args& args, int grid, cudaStream_t stream) {
  if (grid <= 0) return cudaSuccess;
  MapsF8 m;
  for (int p = 0; p < 2; ++p)
    for (int i = 0; i < kFp8Boxes; ++i) m.x[p][i] = maps[kFp8Boxes * p + i];
  return epi == EPI_SWIGLU
             ? launch_pdl(grouped_gemm_fp8_kernel<EPI_SWIGLU>, dim3(grid), dim3(kThreads), kSmem, stream, 1, m, args)
             : launch_pdl(grouped_gemm_fp8_kernel<EPI_BF16>, dim3(grid), dim3(kThreads), kSmem, stream, 1, m, args);
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
