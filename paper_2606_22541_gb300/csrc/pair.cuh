// Device helpers of the CTA-pair grouped GEMMs: thread-block cluster
// addressing, cluster-scope mbarriers, the two-SM forms of TMA and tcgen05,
// fragment-shaped TMEM loads, transposing shared-memory stores, the tile
// queue shared by the two CTAs and the token-tile schedule.
//
// A pair is a cluster of two CTAs on the two SMs of one TPC.  Its tensor cores
// work on one tile together (tcgen05 cta_group::2): weights are the M operand
// (256 rows, 128 in each CTA's shared memory and TMEM lanes), tokens the N
// operand (N rows, N / 2 in each CTA's shared memory), so both operands of an
// MMA are read from shared memory once per SM instead of the N operand twice.
#pragma once

#include "common.cuh"
#include "gemm_config.h"
#include "gemm_sched.cuh"
#include "internal.h"

namespace asap {

constexpr int kPairRows = 256;     // token rows of a tile at most (N of the MMA)
constexpr int kPairRowUnit = 32;   // tile heights are multiples of this (N % 32 == 0)
constexpr uint16_t kPairMask = 3;  // both CTAs of the cluster

// ---------------------------------------------------------------- cluster
__device__ __forceinline__ uint32_t pair_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address, in the cluster's shared window, of this CTA's offset ``addr`` in CTA ``rank``.
__device__ __forceinline__ uint32_t pair_map(uint32_t addr, uint32_t rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}
__device__ __forceinline__ void pair_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void st_pair_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Arrive on a barrier of either CTA (addr from pair_map).  Without .cluster
// scope: what it orders is TMEM (fenced by tcgen05); a cluster-scope release or
// acquire stalled its thread for 2000 to 4000 cycles behind the loads in flight
// (tile changes took 300 cycles without it; gate/up GEMM of 8192 DeepSeek-V3
// tokens 3059 -> 2917 us).
__device__ __forceinline__ void mbar_arrive_pair(uint32_t addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// The same with cluster scope, and the wait for it: this CTA's reads of its
// shared memory, its own and those it has waited for, come before what the
// waiting thread of the other CTA does next.
__device__ __forceinline__ void mbar_arrive_release_pair(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool mbar_wait_acquire_pair(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return bounded_wait(
      [&]() {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        return ok != 0;
      },
      abort_flag);
}
// Arrive on the other CTA's barrier and expect ``bytes`` of st.async on it.
__device__ __forceinline__ void mbar_arrive_expect_tx_pair(uint32_t addr, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(addr), "r"(bytes) : "memory");
}
// 16 bytes into the other CTA's shared memory; its barrier counts them when
// they are visible there.
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t bar, int a, int b, int c, int d) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2, %3, %4, %5}, [%1];" ::"r"(addr),
               "r"(bar), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
// After a failed wait: copies this thread issued complete on a barrier of the
// other CTA, which it cannot wait on, so it lets 2 ms pass (a TMA load takes
// microseconds) before the CTA may wind down.
__device__ __forceinline__ void drain_delay() {
  const uint64_t t0 = globaltimer_ns();
  while (globaltimer_ns() - t0 < 2000000ull) {
  }
}

// ---------------------------------------------------------------- two-SM TMA / tcgen05
// tma_load_2d into this CTA's shared memory, completing on a barrier of either
// CTA of the pair (bar from pair_map).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* m, uint32_t bar, int x, int y,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// Arrive once on the barrier at this offset in both CTAs when every tcgen05 op
// this thread issued so far is done.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(kPairMask)
      : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                 uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// ---------------------------------------------------------------- fragments
// 16 TMEM lanes x 64 (32) columns.  Thread t receives, for each group n of 8
// columns, lane t / 4 at columns 8n + 2 (t % 4), + 1 in r[4n], r[4n + 1] and
// lane t / 4 + 8 at the same columns in r[4n + 2], r[4n + 3].
__device__ __forceinline__ void tmem_ld_frag64(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_frag32(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// Four 8 x 8 matrices of 16-bit values held like the fragments above (thread
// t: row t / 4, columns 2 (t % 4), + 1), each stored transposed: column i of
// matrix m becomes 16 contiguous bytes at the address thread 8m + i passes.
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b),
               "r"(c), "r"(d)
               : "memory");
}

// ---------------------------------------------------------------- token tiles
// The rows of a segment are cut into the fewest tiles of at most MAXR rows, of
// equal height up to kPairRowUnit: a tile's MMA time is proportional to its
// height, and equal tiles keep the weight bytes per MMA cycle (each tile
// streams the same weight boxes, from L2 after the first) at their lowest.
template <int MAXR>
__device__ __forceinline__ int pair_mtiles(int rows) {
  return (rows + MAXR - 1) / MAXR;
}
__device__ __forceinline__ int pair_height(int rows, int mt) {
  const int h = (rows + mt - 1) / mt;
  return (h + kPairRowUnit - 1) / kPairRowUnit * kPairRowUnit;
}

struct alignas(16) PairTile {
  int row, rows;  // first token row, valid rows
  int n;          // N of the MMAs: rows rounded up to kPairRowUnit
  int w_tile;     // 256-row weight tile index in the tensor
  int n_tile;
  int k_iters;    // 0: no more tiles
  int group;
  int p1;
};

// Position, in the order cold groups, hot groups, problem 1, of the t-th tile
// handed out: the tiles from ``cold`` on come in bursts spread evenly over the
// launch (burst k from tile ceil(k Q total / hot) on).
__device__ __forceinline__ int mix_position(int t, int cold, int total) {
  const int hot = total - cold;
  if (hot == 0) return t;
  constexpr int Q = ASAP_MIX_BURST;
  const int k = static_cast<int>(static_cast<long long>(t) * hot / (static_cast<long long>(Q) * total));
  const int tk = static_cast<int>((static_cast<long long>(k) * Q * total + hot - 1) / hot);
  // (t >= tk: k is the last burst that starts at or before t)
  if (t - tk < Q && k * Q + t - tk < hot) return cold + k * Q + t - tk;
  return t - min((k + 1) * Q, hot);
}

// The t-th tile of the launch.  Inside a group: block of m_block token tiles,
// n-tile, then token tile innermost, so the workers that run at the same time
// share a weight tile through L2 and a block's rows stay in L2 over its n-tiles.
template <int MAXR>
__device__ __forceinline__ void pair_decode(int t, const MixSched* s, int G, int total0, int total, const GemmArgs& a,
                                            PairTile& T) {
  int r0, m, local, wt0;
  const int u = mix_position(t, s->cold, total);
  if (u < total0) {
    int lo = 0, hi = G;  // largest g with tile_start[g] <= u
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (s->tile_start[mid] <= u) lo = mid; else hi = mid;
    }
    local = u - s->tile_start[lo];
    T.group = s->group[lo];
    r0 = s->row_base[T.group];
    m = s->row_base[T.group + 1] - r0;
    wt0 = T.group * (a.b_stride0 / kGemmBN);
    T.k_iters = a.k_iters0;
    T.p1 = 0;
  } else {
    local = u - total0;
    r0 = 0;
    m = s->m1;
    wt0 = 0;
    T.group = 0;
    T.k_iters = a.k_iters1;
    T.p1 = 1;
  }
  const int mt = pair_mtiles<MAXR>(m), h = pair_height(m, mt);
  const int mb = T.p1 ? a.m_block1 : a.m_block0;  // token tiles per block
  const int per = mb * (T.p1 ? a.n_tiles1 : a.n_tiles0);
  const int b = local / per;
  local -= b * per;
  const int sz = min(mb, mt - b * mb);
  const int nt = local / sz, mi = b * mb + local - nt * sz;
  T.row = r0 + mi * h;
  T.rows = max(0, min(h, m - mi * h));
  T.n = max(kPairRowUnit, (T.rows + kPairRowUnit - 1) / kPairRowUnit * kPairRowUnit);
  T.n_tile = nt;
  T.w_tile = wt0 + nt;
}

// ---------------------------------------------------------------- tile queue
// One CTA of the pair is the queue's home: its scheduler thread claims tiles,
// decodes them and writes the descriptions into both CTAs' queues, one tile
// ahead of the loads.  The consumers release a slot on a barrier of their own
// CTA: the home's on the empty barrier, the other CTA's on its read barrier,
// whose completions a thread without loads of its own (pair_forward) passes on
// to the home with cluster scope, so that the other CTA's reads of a slot come
// before the home's next store into it and no role pays for the scope.  (With
// every role popping an id and decoding it itself, the id claimed when the loads
// reached it, a tile change cost the MMA issuer about 3200 cycles.)
constexpr int kPairQ = 2;
constexpr int kPairQBytes = kPairQ * (static_cast<int>(sizeof(PairTile)) + 24);

struct PairQueue {
  uint32_t q0;    // this CTA's queue: descriptions, full, empty and read barriers
  uint32_t home;  // the home's, in the cluster window
  bool at_home;   // this CTA is the home
  uint32_t n = 0;

  __device__ __forceinline__ uint32_t slot() const { return n % kPairQ; }
  __device__ __forceinline__ uint32_t phase() const { return (n / kPairQ) & 1u; }
  __device__ __forceinline__ static uint32_t desc(uint32_t b, uint32_t s) { return b + 32u * s; }
  __device__ __forceinline__ static uint32_t full(uint32_t b, uint32_t s) { return b + 32u * kPairQ + 8u * s; }
  __device__ __forceinline__ static uint32_t empty(uint32_t b, uint32_t s) { return b + 40u * kPairQ + 8u * s; }
  __device__ __forceinline__ static uint32_t read(uint32_t b, uint32_t s) { return b + 48u * kPairQ + 8u * s; }

  __device__ __forceinline__ static void store_local(uint32_t addr, const PairTile& T) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(T.row), "r"(T.rows), "r"(T.n),
                 "r"(T.w_tile)
                 : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr + 16), "r"(T.n_tile), "r"(T.k_iters),
                 "r"(T.group), "r"(T.p1)
                 : "memory");
  }
  // scheduler thread; peer: the other CTA's queue in the cluster window
  __device__ __forceinline__ bool push(const PairTile& T, uint32_t peer, volatile int* abort_flag) {
    const uint32_t s = slot();
    if (!mbar_wait_acquire_pair(empty(q0, s), phase() ^ 1u, abort_flag)) return false;
    const uint32_t pd = desc(peer, s), pb = full(peer, s), ld = desc(q0, s);
    mbar_arrive_expect_tx_pair(pb, 32);
    st_async_v4(pd, pb, T.row, T.rows, T.n, T.w_tile);
    st_async_v4(pd + 16, pb, T.n_tile, T.k_iters, T.group, T.p1);
    store_local(ld, T);
    mbar_arrive(full(q0, s));
    ++n;
    return true;
  }
  // whole warps; a role's warp releases the slot once
  __device__ __forceinline__ bool pop(PairTile& T, volatile int* abort_flag) const {
    const uint32_t s = slot();
    if (!mbar_wait(full(q0, s), phase(), abort_flag)) return false;
    const uint32_t a = desc(q0, s);
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(T.row), "=r"(T.rows), "=r"(T.n), "=r"(T.w_tile)
                 : "r"(a)
                 : "memory");
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(T.n_tile), "=r"(T.k_iters), "=r"(T.group), "=r"(T.p1)
                 : "r"(a + 16)
                 : "memory");
    return true;
  }
  // the whole warp calls this once every lane has popped; one lane arrives and
  // the warp goes on to the next slot
  __device__ __forceinline__ void release(bool one) {
    __syncwarp();  // the other lanes' reads come before the arrival
    if (one) mbar_arrive(at_home ? empty(q0, slot()) : read(q0, slot()));
    ++n;
  }
};

// One thread of the CTA that is not the home: passes the releases of its CTA's
// roles on to the home, until the end of the tiles.
__device__ __forceinline__ bool pair_forward(PairQueue& tq, volatile int* abort_flag) {
  PairTile T;
  while (true) {
    if (!tq.pop(T, abort_flag)) return false;
    if (T.k_iters == 0) return true;
    const uint32_t s = tq.slot();
    if (!mbar_wait(PairQueue::read(tq.q0, s), tq.phase(), abort_flag)) return false;
    mbar_arrive_release_pair(PairQueue::empty(tq.home, s));
    ++tq.n;
  }
}

// The same queue within one CTA (home and only consumer).
__device__ __forceinline__ bool local_push(PairQueue& tq, const PairTile& T, volatile int* abort_flag) {
  const uint32_t s = tq.slot();
  if (!mbar_wait(PairQueue::empty(tq.q0, s), tq.phase() ^ 1u, abort_flag)) return false;
  PairQueue::store_local(PairQueue::desc(tq.q0, s), T);
  mbar_arrive(PairQueue::full(tq.q0, s));
  ++tq.n;
  return true;
}

// The scheduler thread: claims and decodes this worker's tiles (worker: a CTA or
// a pair; the first tile is its index, the next ones come from the launch's
// counter) and pushes them.  Returns false when a wait ran out.
template <int MAXR, typename Push>
__device__ __forceinline__ bool feed_tiles(const GemmArgs& args, const MixSched* sch, int G, int worker, int workers,
                                           Push push) {
  const int total0 = sch->tile_start[G];
  const int total = total0 + pair_mtiles<MAXR>(sch->m1) * args.n_tiles1;
  int t = worker;
  PairTile T{};
  do {
    const bool more = t < total;
    if (more) pair_decode<MAXR>(t, sch, G, total0, total, args, T);
    else T.k_iters = 0;
    if (!push(T)) return false;
    if (more) t = workers + (args.tile_counter ? atomicAdd(args.tile_counter, 1) : t);
  } while (T.k_iters != 0);
  return true;
}
template <int MAXR>
__device__ __forceinline__ bool pair_schedule(const GemmArgs& args, const MixSched* sch, int G, PairQueue& tq,
                                              uint32_t peer, volatile int* abort_flag) {
  return feed_tiles<MAXR>(args, sch, G, static_cast<int>(blockIdx.x >> 1), static_cast<int>(gridDim.x >> 1),
                          [&](const PairTile& T) { return tq.push(T, peer, abort_flag); });
}
template <int MAXR>
__device__ __forceinline__ bool tile_schedule(const GemmArgs& args, const MixSched* sch, int G, PairQueue& tq,
                                              volatile int* abort_flag) {
  return feed_tiles<MAXR>(args, sch, G, static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x),
                          [&](const PairTile& T) { return local_push(tq, T, abort_flag); });
}

}  // namespace asap
