// Shared device helpers of libasap_moe: status word bits, bf16 packing and
// thin inline-PTX wrappers for mbarrier, TMA (cp.async.bulk.tensor) and the
// fifth-generation tensor core (tcgen05 + TMEM) of sm_103a.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace asap {

// ---------------------------------------------------------------- status word
// Kernels never trap: they OR one of these bits into the handle's status word
// and skip the offending access.
enum : uint32_t {
  ST_BAD_EXPERT_INDEX = 1u << 0,  // idx outside [0, E)
  ST_BAD_POSITION = 1u << 1,      // permutation position outside [0, n*k)
  ST_WAIT_TIMEOUT = 1u << 2,      // an mbarrier wait passed its time limit
  ST_BAD_OFFSETS = 1u << 3,       // offsets not monotone or past the rows
  ST_BAD_LAYER = 1u << 4,         // layer id outside [0, n_layers); layer 0 was used
  ST_SMEM_ALIGN = 1u << 5,        // dynamic shared memory not 1024-byte aligned; the GEMM did nothing
  ST_MBOX_OVERRUN = 1u << 6,      // a mailbox slot was posted again before its previous post was served
  ST_MBOX_WAIT = 1u << 7,         // a mailbox round's wait for the post it serves ran out
};

__device__ __forceinline__ void record_status(uint32_t* st, uint32_t bits) {
  if (st) atomicOr(st, bits);
}

constexpr int kChunkTokens = 32;  // tokens per routing / dispatch chunk (one warp each)
constexpr int kMaxRouterSplits = 4;  // K slices of the tensor-core router GEMM (1, 2 or 4)
constexpr int kMaxExperts = 256;
constexpr int kMaxTopK = 8;

// ---------------------------------------------------------------- bf16 helpers
__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);  // lo -> low half
  return *reinterpret_cast<uint32_t*>(&p);
}

// ---------------------------------------------------------------- gating
// Sigmoid score of a router logit (grouped gating): 1 / (1 + e^-l) with the
// fast exponential and reciprocal.  __expf(x) is within 2 + 1.16|x| ulp
// (CUDA's documented bound) and __fdividef(1, y) within 2 ulp for y in
// [1, 2^126]; the sigmoid's slope sigma (1 - sigma) is at most 1/4 and falls
// like e^-|l|, so the score is within 5 * 2^-24 of the sigmoid of the float32
// logit.  Every gate kernel uses this one expression, so all routing paths
// give the same bits.  (No slow-path branch, unlike the IEEE division: the
// compiler can overlap the scores of one thread.)
__device__ __forceinline__ float gate_sigmoid(float l) { return __fdividef(1.0f, 1.0f + __expf(-l)); }

// ---------------------------------------------------------------- dependent launches
// Kernels are launched with programmatic stream serialisation (launch_pdl): a
// kernel may start while the one before it on the stream still runs.  Every
// thread calls pdl_wait before it touches global memory; it returns once the
// kernel before has completed with its writes visible (and, as every kernel
// waits so, all kernels before that one).  pdl_launch allows the next kernel to
// start once every CTA has called it or left.  The small kernels call it when
// their own wait is over, the single-CTA GEMMs when a CTA has no tiles left; the
// CTA pairs (gemm_pair.cu) and the CUDA-core router (route.cu) do not.
//
// Such a kernel is resident while the data it will read is still being written,
// so nothing an earlier kernel or the caller writes is read-only for its
// lifetime: it is read with ld_dep or a plain load, never with __ldg or through
// a const __restrict__ pointer (the non-coherent path, whose loads may also be
// moved above pdl_wait).  __ldg is for the weights, their scales and the
// router's bias.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Coherent load that stays behind pdl_wait (volatile) but may pass this
// kernel's own plain stores (no memory clobber): of data this kernel does not
// write.
__device__ __forceinline__ int ld_dep(const int* p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_dep(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_dep(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ld_dep(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// ---------------------------------------------------------------- smem / timers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// The same without suspending the thread.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Every wait in these kernels is bounded: after kWaitLimitNs, or as soon as
// another role of the CTA has given up (abort flag), it returns false and the
// caller records ST_WAIT_TIMEOUT and winds down.  A normal wait lasts
// microseconds.
constexpr uint64_t kWaitLimitNs = 2000000000ull;  // 2 s

template <typename Try>
__device__ __forceinline__ bool bounded_wait(Try done, volatile int* abort_flag) {
  if (done()) return true;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t i = 1;; ++i) {
    if (done()) return true;
    if ((i & 63u) == 0) {
      if (*abort_flag) return false;
      if (globaltimer_ns() - t0 > kWaitLimitNs) return false;
    }
  }
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return bounded_wait([&]() { return mbar_try_wait(bar, parity); }, abort_flag);
}

// ---------------------------------------------------------------- rings
// Position in a ring of N barriers (8 bytes apart from ``bar``): stage s of
// lap parity ``phase``.
template <int N>
struct Ring {
  int s = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void advance() {
    if (++s == N) {
      s = 0;
      phase ^= 1u;
    }
  }
};

// The whole warp waits until every lane's barrier (the lanes may look at
// different ones) has completed its phase.  Bounded like mbar_wait.
__device__ __forceinline__ bool mbar_wait_all(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
    if ((i & 255u) == 0) {
      const uint64_t now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      if (__any_sync(0xffffffffu, *abort_flag != 0 || now - t0 > kWaitLimitNs)) return false;
    }
  }
}

// ---------------------------------------------------------------- TMA
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}

// A descriptor that sits in global memory (the layer table, written before the
// launch) is read by the tensor-map proxy: the issuing thread acquires it once.
__device__ __forceinline__ void tensormap_acquire(const CUtensorMap* m) {
  asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(m))
               : "memory");
}

// Layer id of a layer-oblivious launch (Section 3.4.2), loaded when the kernel
// runs.  Ids outside [0, n_layers) become 0 and are recorded when ``report``.
__device__ __forceinline__ int load_layer(const int32_t* layer, int n_layers, uint32_t* status, bool report) {
  int l = *reinterpret_cast<const volatile int32_t*>(layer);
  if (l < 0 || l >= n_layers) {
    if (report) record_status(status, ST_BAD_LAYER);
    l = 0;
  }
  return l;
}

// 2-D tiled load of one box into shared memory; completes on ``bar`` with the
// box's byte count.  x is the inner (contiguous) coordinate in elements.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int x, int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}

// 2-D tiled store of one box from shared memory (the box's layout in shared
// memory is the tensor map's swizzle); joins the issuing thread's bulk async
// group.  x (inner coordinate) x element size must be a multiple of 16 bytes
// and neither coordinate may be negative.  The writes to the box by other
// threads must be ordered before it with fence_proxy_async_smem() and a
// barrier.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* m, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(m)),
               "r"(src), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until the thread's committed bulk stores have read their shared memory.
__device__ __forceinline__ void bulk_wait_group_read0() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// Waits until the thread's committed bulk stores are complete.
__device__ __forceinline__ void bulk_wait_group0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Orders this thread's generic-proxy shared-memory writes before later
// async-proxy (TMA) accesses.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// L2 eviction priority of TMA loads: 0 normal, 1 evict-first (streamed
// once), 2 evict-last (re-read by other CTAs).
__device__ __forceinline__ uint64_t l2_policy(int hint) {
  uint64_t p;
  if (hint == 1)
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  else if (hint == 2)
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  else
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// ---------------------------------------------------------------- tcgen05 / TMEM
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Arrive once on ``bar`` when every tcgen05 op this thread issued so far is done.
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulator.
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns: thread i of the warp receives
// TMEM lane (lane field of taddr) + i, columns [col, col + 16).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// One lane of a converged warp (the same each time).  Issuing tcgen05
// instructions from ``if (elect_one())`` in a warp that runs its loop converged
// costs far fewer issue cycles than from a lane that left its warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p)::"memory");
  return p != 0;
}

// Shared-memory matrix descriptor of a K-major operand tile written by TMA
// with 128-byte swizzle: rows of 128 bytes (64 bf16), 8-row atoms of 1024
// bytes stacked along M/N (stride byte offset 1024).  The leading byte offset
// is unused for this layout.  Bits 46-48 hold the fixed value 0b001; bits
// 61-63 select the 128-byte swizzle (2).
// Same for 64-byte rows (32 bf16) written with 64-byte swizzle: 8-row atoms
// of 512 bytes; bits 61-63 select the 64-byte swizzle (4).
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(512 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(4) << 61;
  return d;
}

__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// Instruction descriptor of kind::f16: fp32 accumulator (bits 4-5 = 1), bf16
// A and B (bits 7-9 = 1, 10-12 = 1), both K-major (bits 15, 16 = 0),
// N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}

}  // namespace asap
