// BF16 grouped expert GEMM on CTA pairs (tcgen05 cta_group::2, TMA, TMEM).
//
// The expert computation of the MoE layer (ASAP Section 3.4.2), as
// grouped_gemm_kernel computes it, on two SMs per tile: the 256 weight rows of
// an n-tile are the M operand (128 rows per CTA) and up to 256 token rows of
// one expert the N operand (half per CTA).  Against one CTA per tile:
//  - every weight and token box is read from shared memory by one SM only, and
//    a stage is 16 + 16 KB, so the rings hold more k-steps;
//  - N follows the rows in steps of 32, so a segment's padding is at most 31
//    rows (63 or 127 with tokens on the M side);
//  - the 256-column accumulators are double-buffered in TMEM at the full tile
//    size, so the epilogue runs beside the next tile's main loop.
//
// Roles of a CTA (256 threads):
//   warp 0: weight producer (its 128 rows of each 256-row box, 16 KB)
//   warp 1: TMEM; in the leader the MMA issuer of the pair
//   warps 2-5: epilogue, one TMEM lane quarter each
//   warp 6: token producer (its half of the tile's rows)
//   warp 7: in the leader the tile scheduler of the pair, in the other CTA the
//           thread that passes tile releases on to it
// The next kernel on the stream starts when this one has ended (no pdl_launch):
// with the call in both CTAs, where their tiles end, the next kernel's CTAs took
// issue slots and bandwidth from the last tiles (layer, us, with | without: Mixtral
// 4096 tokens 1777 | 1668, 1536 726 | 730, DeepSeek-V3 4096 tokens 3580 | 3568, 1
// token 164.2 | 163.0).
// All loads complete on the leader's full barriers; the leader's commits
// arrive on both CTAs' empty and accumulator barriers.
//
// Epilogue: TMEM lanes are output channels and columns are tokens, so the
// accumulator is read as 8 x 8 fragments and stored transposed (stmatrix) into
// a token-major staging box.  Gate and up rows are interleaved in eights, so a
// thread holds a channel's gate and up values of the same tokens.
#include "common.cuh"
#include "gemm_config.h"
#include "gemm_sched.cuh"
#include "internal.h"
#include "pair.cuh"

namespace asap {

namespace {

constexpr int SW = ASAP_RING_CTA2_W, SX = ASAP_RING_CTA2_X;
constexpr int kWBytes = 128 * kGemmBK * 2;  // 128 weight rows
constexpr int kXBytes = 128 * kGemmBK * 2;  // up to 128 token rows
constexpr int kEpiWarps = 4;
constexpr int kThreads = 32 * (4 + kEpiWarps);
constexpr int kXProdWarp = 2 + kEpiWarps;
constexpr int kSchedWarp = 3 + kEpiWarps;
constexpr uint32_t kTmemCols = 512;
// store staging: two buffers of two [32 tokens, 64 channels] boxes
constexpr int kBoxBytes = 32 * 128;
constexpr int kStageBuf = 2 * kBoxBytes;
constexpr int kStageBytes = 2 * kStageBuf;
constexpr int kNumBars = 2 * SW + 2 * SX + 5;
constexpr int kBarBytes = (8 * kNumBars + 15) / 16 * 16 + kPairQBytes + 16;
constexpr size_t kSmem = SW * kWBytes + SX * kXBytes + kStageBytes + kBarBytes + sizeof(MixSched);
static_assert(kSmem <= 227 * 1024, "shared memory budget");
// consumers of a tile: in each CTA the producers and the epilogue warps, in the
// leader also the MMA issuer and the other CTA's forwarding thread
constexpr int kQueueReaders = 2 + kEpiWarps;
constexpr int kQueueConsumers = kQueueReaders + 2;

struct PairMaps {
  CUtensorMap x[2][4];  // problem; boxes of 32, 64, 96 and 128 token rows
  CUtensorMap o[2];     // problem; [32 rows, 64 columns] boxes of the output
};

__device__ __forceinline__ void epi_barrier() {
  __syncwarp();
  asm volatile("bar.sync 1, 128;" ::: "memory");
}
// Whether ok holds in every thread of the epilogue warps.
__device__ __forceinline__ bool epi_all(bool ok) {
  uint32_t r;
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 2, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ float silu_mul(uint32_t g, uint32_t u) {
  const float gf = __uint_as_float(g);
  // the single-CTA kernel's expression: the same bits
  return __fdividef(gf, 1.0f + __expf(-gf)) * __uint_as_float(u);
}
__device__ __forceinline__ uint32_t pack_acc(uint32_t a, uint32_t b) {
  return pack_bf16x2(__uint_as_float(a), __uint_as_float(b));
}

// One tile's epilogue for a warp: the accumulator at taddr (the warp's lane
// quarter q), in rounds of 64 (SwiGLU) or 32 tokens.  A round fills one
// staging buffer (SwiGLU: two boxes of 32 tokens x the CTA's 64 channels;
// plain: 32 tokens x 2 boxes of 64 channels).  Full boxes leave by TMA, a
// box with rows past the tile by plain 16-byte stores.
template <int EPI>
__device__ __forceinline__ void pair_epilogue(const PairTile& T, const GemmArgs& a, uint32_t taddr, int q, int lane,
                                              uint32_t rank, uint32_t stage, uint32_t& buf, const CUtensorMap* tm,
                                              uint32_t tempty) {
  constexpr bool SG = EPI == EPI_SWIGLU;
  constexpr int RT = SG ? 64 : 32;  // tokens per round
  const int tid = q * 32 + lane;    // 0 .. 127 in the epilogue warps
  uint16_t* out = static_cast<uint16_t*>(T.p1 ? a.out1 : a.out0);
  const long long ldo = T.p1 ? a.ldo1 : a.ldo0;
  const int col0 = SG ? T.n_tile * 128 + static_cast<int>(rank) * 64 : T.n_tile * 256 + static_cast<int>(rank) * 128;
  // stmatrix: this thread's row (token i of matrix mx) in the staging boxes
  const int mx = lane >> 3, mi = lane & 7;
  for (int c0 = 0; c0 < T.rows; c0 += RT) {
    uint32_t pk[16];
    __syncwarp();
    if constexpr (SG) {
      // pk[2n + hl]: 8-token group n, lane half hl
      uint32_t v[2][32];
      tmem_ld_frag64(taddr + c0, v[0]);
      tmem_ld_frag64(taddr + (16u << 16) + c0, v[1]);
      tmem_ld_wait();
#pragma unroll
      for (int n = 0; n < 8; ++n)
#pragma unroll
        for (int hl = 0; hl < 2; ++hl)
          pk[2 * n + hl] = pack_bf16x2(silu_mul(v[hl][4 * n], v[hl][4 * n + 2]),
                                       silu_mul(v[hl][4 * n + 1], v[hl][4 * n + 3]));
    } else {
      // pk[4n + 2 hl + rh]: row half rh (lanes + 8 rh)
      uint32_t v[2][16];
      tmem_ld_frag32(taddr + c0, v[0]);
      tmem_ld_frag32(taddr + (16u << 16) + c0, v[1]);
      tmem_ld_wait();
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int hl = 0; hl < 2; ++hl)
#pragma unroll
          for (int rh = 0; rh < 2; ++rh)
            pk[4 * n + 2 * hl + rh] = pack_acc(v[hl][4 * n + 2 * rh], v[hl][4 * n + 2 * rh + 1]);
    }
    if (c0 + RT >= T.rows) {  // the accumulator has been read
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_pair(tempty);
    }
    // the store that last used this buffer has read it
    if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
    epi_barrier();
    const uint32_t sb = stage + (buf & 1u) * kStageBuf;
    if constexpr (SG) {
#pragma unroll
      for (int n = 0; n < 8; n += 2) {
        // matrices (n, hl 0), (n, hl 1), (n + 1, hl 0), (n + 1, hl 1)
        const int r = 8 * (n + (mx >> 1)) + mi;
        const int j = 2 * q + (mx & 1);
        stmatrix_x4_trans(sb + r * 128 + ((j ^ mi) << 4), pk[2 * n], pk[2 * n + 1], pk[2 * n + 2], pk[2 * n + 3]);
      }
    } else {
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        // matrices (hl, rh): channels 32 q + 8 mx ..
        const int r = 8 * n + mi;
        const int c = 4 * q + mx;
        stmatrix_x4_trans(sb + (c >> 3) * kBoxBytes + r * 128 + (((c & 7) ^ mi) << 4), pk[4 * n], pk[4 * n + 1],
                          pk[4 * n + 2], pk[4 * n + 3]);
      }
    }
    fence_proxy_async_smem();
    epi_barrier();
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int br = SG ? c0 + 32 * b : c0;  // the box's first row in the tile
      const int bc = SG ? 0 : 64 * b;        // its first column in the CTA's columns
      const int left = T.rows - br;
      if (left >= 32) {
        if (tid == 0) tma_store_2d(tm, sb + b * kBoxBytes, col0 + bc, T.row + br);
      } else if (left > 0) {
        // 8 threads per row
        for (int r = tid >> 3; r < left; r += 16) {
          uint4 v;
          const uint32_t ad = sb + b * kBoxBytes + r * 128 + (((tid & 7) ^ (r & 7)) << 4);
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                       : "r"(ad)
                       : "memory");
          *reinterpret_cast<uint4*>(out + (static_cast<long long>(T.row) + br + r) * ldo + col0 + bc + (tid & 7) * 8) =
              v;
        }
      }
    }
    if (tid == 0) bulk_commit_group();
    ++buf;
  }
}

// Producer warp of the weights (W) or the tokens.  The whole warp runs the
// loop, one lane issues, and the next slot is looked at before this slot's
// load is issued (with a lane that left its warp, a wait and up to four boxes
// of 16 or 64 token rows per k-step, a k-step took 560 to 700 cycles to issue,
// more than its MMAs: 6.1 ms instead of 5.3 ms for the gate/up GEMM of 16384
// DeepSeek-V3 tokens).
template <bool W>
__device__ __forceinline__ bool produce(const GemmArgs& args, const PairMaps& maps, const CUtensorMap* const* tmW,
                                        PairQueue& tq, uint32_t full, uint32_t empty, uint32_t ring_base,
                                        uint32_t rank, int lane, volatile int* abort_flag) {
  constexpr int NS = W ? SW : SX;
  constexpr int stride = W ? kWBytes : kXBytes;
  const bool issuer = elect_one();
  const uint64_t pol = l2_policy(W ? args.hint_b : args.hint_a);
  const uint32_t lead_full = pair_map(full, 0);
  Ring<NS> r;
  bool ready = true;  // slot r.s has been seen to be free
  PairTile T;
  while (true) {
    if (!__all_sync(0xffffffffu, tq.pop(T, abort_flag))) return false;
    tq.release(issuer);
    if (T.k_iters == 0) break;
    // weights: box (w_tile, kb) is rows (w_tile k_iters + kb) 256 of 64
    // columns, this CTA loads its half of it; tokens: the CTA's half of the
    // tile's rows, in a box of the next multiple of 32 rows
    const int half = T.n / 2;
    const int box = (half + 31) / 32;
    const CUtensorMap* m = W ? tmW[T.p1] : &maps.x[T.p1][box - 1];
    const int y0 = W ? static_cast<int>(static_cast<long long>(T.w_tile) * T.k_iters * 256 + rank * 128)
                     : T.row + static_cast<int>(rank) * half;
    const uint32_t tx = W ? 2 * kWBytes : 2 * box * 32 * 128;
    for (int kb = 0; kb < T.k_iters; ++kb) {
      if (!__all_sync(0xffffffffu, ready) &&
          !__all_sync(0xffffffffu, mbar_wait(empty + 8u * r.s, r.phase ^ 1u, abort_flag)))
        return false;
      const int s = r.s;
      r.advance();
      ready = mbar_test_wait(empty + 8u * r.s, r.phase ^ 1u);
      if (issuer) {
        if (rank == 0) mbar_arrive_expect_tx(full + 8u * s, tx);
        tma_load_2d_pair(ring_base + s * stride, m, lead_full + 8u * s, W ? 0 : kb * kGemmBK, W ? y0 + kb * 256 : y0,
                         pol);
      }
    }
  }
  // every commit on this ring's barriers has arrived before the CTA may leave
  for (int i = 0; i < NS; ++i) {
    if (!__all_sync(0xffffffffu, mbar_wait(empty + 8u * r.s, r.phase ^ 1u, abort_flag))) return false;
    r.advance();
  }
  return true;
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    pair_gemm_kernel(const __grid_constant__ PairMaps maps, const GemmArgs args) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  if (base & 1023u) {  // the same in both CTAs: nothing is initialised yet
    pdl_wait();
    if (threadIdx.x == 0) record_status(args.status, ST_SMEM_ALIGN);
    return;
  }
  const uint32_t sW = base, sX = base + SW * kWBytes, stage = sX + SX * kXBytes;
  uint8_t* bar_area = smem_raw + SW * kWBytes + SX * kXBytes + kStageBytes;
  const uint32_t bar0 = smem_u32(bar_area);
  auto fullW = [&](int s) { return bar0 + 8u * s; };
  auto emptyW = [&](int s) { return bar0 + 8u * (SW + s); };
  auto fullX = [&](int s) { return bar0 + 8u * (2 * SW + s); };
  auto emptyX = [&](int s) { return bar0 + 8u * (2 * SW + SX + s); };
  auto tfull = [&](int b) { return bar0 + 8u * (2 * SW + 2 * SX + b); };
  auto tempty = [&](int b) { return bar0 + 8u * (2 * SW + 2 * SX + 2 + b); };
  const uint32_t drain = bar0 + 8u * (2 * SW + 2 * SX + 4);
  constexpr int kQOff = (8 * kNumBars + 15) / 16 * 16;
  const uint32_t tq0 = bar0 + kQOff;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_area + kQOff + kPairQBytes);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  MixSched* sch = reinterpret_cast<MixSched*>(bar_area + kBarBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = pair_rank();
  const bool leader = rank == 0;
  const int G = args.groups;
  const CUtensorMap* tmW[2] = {nullptr, nullptr};

  if (warp == 0) {
    if (lane == 0) {
      for (int s = 0; s < SW; ++s) {
        mbar_init(fullW(s), 1);
        mbar_init(emptyW(s), 1);
      }
      for (int s = 0; s < SX; ++s) {
        mbar_init(fullX(s), 1);
        mbar_init(emptyX(s), 1);
      }
      for (int b = 0; b < 2; ++b) {
        mbar_init(tfull(b), 1);
        mbar_init(tempty(b), 2 * kEpiWarps);
      }
      mbar_init(drain, 1);
      for (int s = 0; s < kPairQ; ++s) {
        mbar_init(PairQueue::full(tq0, s), 1);
        mbar_init(PairQueue::empty(tq0, s), kQueueConsumers);
        mbar_init(PairQueue::read(tq0, s), kQueueReaders);
      }
      *abort_flag = 0;
      fence_barrier_init();
    }
    pdl_wait();
    const LayerEntry& le =
        args.lref.table[load_layer(args.lref.layer, args.lref.n_layers, args.status, blockIdx.x == 0 && lane == 0)];
    tmW[0] = &le.map[args.bmap0];
    tmW[1] = &le.map[args.bmap1];
    tensormap_acquire(tmW[0]);
    if (args.m1 > 0) tensormap_acquire(tmW[1]);
    if (lane == 0) {
      tma_prefetch_desc(tmW[0]);
      if (args.m1 > 0) tma_prefetch_desc(tmW[1]);
    }
  } else if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
  } else if (warp == kSchedWarp && leader) {
    pdl_wait();
    build_mix_schedule<kPairRows>(args, sch, G, lane);
  }
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  pair_sync();  // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  PairQueue tq{tq0, pair_map(tq0, 0), leader};
  // a role that gives up also ends the other CTA's waits
  auto give_up = [&]() {
    *abort_flag = 1;
    st_pair_u32(pair_map(smem_u32(const_cast<int*>(abort_flag)), rank ^ 1u), 1u);
    record_status(args.status, ST_WAIT_TIMEOUT);
  };

  if (warp == 0 || warp == kXProdWarp) {
    bool ok_role;
    if (warp == 0)
      ok_role = produce<true>(args, maps, tmW, tq, fullW(0), emptyW(0), sW, rank, lane, abort_flag);
    else
      ok_role = produce<false>(args, maps, tmW, tq, fullX(0), emptyX(0), sX, rank, lane, abort_flag);
    if (!ok_role) {
      if (lane == 0) give_up();
      drain_delay();
    }
  } else if (warp == kSchedWarp && lane == 0 && leader) {
    // ------------------------------------------------------------ scheduler
    if (!pair_schedule<kPairRows>(args, sch, G, tq, pair_map(tq0, 1), abort_flag)) give_up();
  } else if (warp == kSchedWarp && lane == 0) {
    if (!pair_forward(tq, abort_flag)) give_up();
  } else if (warp == 1 && leader) {
    // ------------------------------------------------------------ MMA issuer
    // the whole warp runs the loop, one lane issues
    const bool issuer = elect_one();
    Ring<SW> rw;
    Ring<SX> rx;
    bool ok = true, issued = false;
    bool ready = false;  // the stages rw.s, rx.s have been seen to be loaded
    const uint64_t wdesc = smem_desc_sw128(sW), xdesc = smem_desc_sw128(sX);
    PairTile T;
    for (int it = 0; ok; ++it) {
      ok = __all_sync(0xffffffffu, tq.pop(T, abort_flag));
      if (!ok) break;
      tq.release(issuer);
      if (T.k_iters == 0) break;
      const int acc = it & 1;
      ok = __all_sync(0xffffffffu, mbar_wait(tempty(acc), ((it >> 1) & 1) ^ 1u, abort_flag));
      if (!ok) break;
      tc_fence_after();
      const uint32_t d = tmem_base + acc * 256;
      const uint32_t id = idesc_bf16_f32(256, T.n);
      for (int kb = 0; kb < T.k_iters; ++kb) {
        if (!__all_sync(0xffffffffu, ready)) {
          ok = mbar_wait(fullX(rx.s), rx.phase, abort_flag) && mbar_wait(fullW(rw.s), rw.phase, abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
        }
        tc_fence_after();
        const int cw = rw.s, cx = rx.s;
        rw.advance();
        rx.advance();
        ready = mbar_test_wait(fullX(rx.s), rx.phase) & mbar_test_wait(fullW(rw.s), rw.phase);
        if (issuer) {
          const uint64_t wd = wdesc + static_cast<uint32_t>(cw * (kWBytes >> 4));
          const uint64_t xd = xdesc + static_cast<uint32_t>(cx * (kXBytes >> 4));
#pragma unroll
          for (int kk = 0; kk < kGemmBK / 16; ++kk)
            tc_mma_bf16_pair(d, wd + 2 * kk, xd + 2 * kk, id, (kb > 0 || kk > 0) ? 1u : 0u);
          tc_commit_pair(emptyW(cw));
          tc_commit_pair(emptyX(cx));
          if (kb == T.k_iters - 1) tc_commit_pair(tfull(acc));
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
  } else if (warp >= 2 && warp < 2 + kEpiWarps) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;
    const uint32_t tempty_lead[2] = {pair_map(tempty(0), 0), pair_map(tempty(1), 0)};
    uint32_t buf = 0;
    PairTile T;
    for (int it = 0;; ++it) {
      const int acc = it & 1;
      bool ok = __all_sync(0xffffffffu, tq.pop(T, abort_flag));
      if (ok) {
        tq.release(lane == 0);
        if (T.k_iters > 0) ok = mbar_wait(tfull(acc), (it >> 1) & 1, abort_flag);
      }
      // the four warps share barriers below: all go on or none does
      if (!epi_all(ok)) {
        if (lane == 0) give_up();
        break;
      }
      if (T.k_iters == 0) break;
      tc_fence_after();
      pair_epilogue<EPI>(T, args, tmem_base + (static_cast<uint32_t>(q * 32) << 16) + acc * 256, q, lane, rank, stage,
                         buf, &maps.o[T.p1 ? 1 : 0], tempty_lead[acc]);
    }
    // the TMA stores are complete before the staging buffers go away
    if (q == 0 && lane == 0) bulk_wait_group0();
    __syncwarp();
  }

  __syncwarp();
  tc_fence_before();
  pair_sync();  // neither CTA leaves while the other may still reach its shared memory or TMEM
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

template <int EPI>
cudaError_t launch(const PairMaps& maps, const GemmArgs& args, int grid, cudaStream_t stream) {
  return launch_pdl(pair_gemm_kernel<EPI>, dim3(grid), dim3(kThreads), kSmem, stream, 1, maps, args);
}

}  // namespace

cudaError_t pair_gemm_set_attributes() {
  cudaError_t e = cudaFuncSetAttribute(pair_gemm_kernel<EPI_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(kSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pair_gemm_kernel<EPI_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kSmem));
  return e;
}

cudaError_t pair_gemm_launch(int epi, const CUtensorMap* maps, const GemmArgs& args, int pairs, cudaStream_t stream) {
  if (pairs <= 0) return cudaSuccess;
  PairMaps pm;
  for (int p = 0; p < 2; ++p) {
    for (int i = 0; i < 4; ++i) pm.x[p][i] = maps[4 * p + i];
    pm.o[p] = maps[8 + p];
  }
  return epi == EPI_SWIGLU ? launch<EPI_SWIGLU>(pm, args, 2 * pairs, stream)
                           : launch<EPI_BF16>(pm, args, 2 * pairs, stream);
}

}  // namespace asap
