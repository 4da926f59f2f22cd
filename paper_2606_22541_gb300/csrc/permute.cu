// Data movement of the MoE layer: dispatch (token rows into per-expert
// segments), combine (weighted gather-reduce back to tokens) and the one-off
// gate/up weight packing done at handle creation.
//
// Dispatch is the single-GPU form of the token payload the MoE side receives
// grouped for its experts (ASAP Section 3.2.1); combine returns each expert's
// result to its token through the expert IDs (Section 3.2.2).  Both run one to
// eight tokens per CTA and move rows as 16-byte vectors with every lane of a warp
// on consecutive vectors of the same row, so each warp-wide access is 512
// contiguous bytes.
#include "common.cuh"
#include "internal.h"

#include <cuda_fp8.h>

#include <type_traits>

namespace asap {

namespace {

constexpr unsigned kFull = 0xffffffffu;
// Quantise 8 consecutive values of a 128-channel block held by 16 lanes
// (lanes 0-15 one block, 16-31 the next): scale = amax / 448 over the block,
// q = e4m3(v / scale) with round-to-nearest-even and saturation; the
// quotient is taken as v * (1 / scale) in fp32, which can differ from the
// exact quotient by an ulp before the e4m3 rounding.
__device__ __forceinline__ uint2 quantize8(uint4 v, float& scale) {
  float f[8] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y),
                bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w)};
  float am = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) am = fmaxf(am, fabsf(f[i]));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
  scale = am > 0.f ? am / 448.0f : 1.0f;
  const float inv = 1.0f / scale;  // one division; the quotients below are products
  uint32_t w[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const __nv_fp8x2_storage_t lo =
        __nv_cvt_float2_to_fp8x2(make_float2(f[4 * u] * inv, f[4 * u + 1] * inv), __NV_SATFINITE, __NV_E4M3);
    const __nv_fp8x2_storage_t hi =
        __nv_cvt_float2_to_fp8x2(make_float2(f[4 * u + 2] * inv, f[4 * u + 3] * inv), __NV_SATFINITE, __NV_E4M3);
    w[u] = static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
  }
  return make_uint2(w[0], w[1]);
}

// Token, of the TOK of a 256-thread CTA, that this thread's warp works on.  (From
// a shuffle, so that the compiler knows it to be the same in the whole warp and
// keeps positions and addresses in uniform registers: 40 instead of 64 to 88
// registers in dispatch_kernel.)
template <int TOK>
__device__ __forceinline__ int warp_token() {
  return TOK == 1 ? 0 : __shfl_sync(kFull, static_cast<int>(threadIdx.x), 0) / (256 / TOK);
}

// Dispatch: a CTA of 256 threads takes TOK consecutive tokens of a chunk, 256 /
// TOK threads each.  It finds the tokens' positions and writes their rows to
// them; every thread has its vectors of a row in flight before it looks at the
// routing, so the chain from idx to a position (expert, chunk base, rank) hides
// behind the row's load.  Bound by HBM writes (k per row read).
constexpr int kDispatchThreads = 256;
constexpr int kDispatchAhead = 4;  // vectors of the row per thread in flight
static_assert(kDispatchThreads == kChunkTokens * kMaxTopK, "one thread per entry of a chunk");

// Where the rows of a CTA's tokens go: their chunk's entries (idx, t_local * k +
// j) and bases, the first token's number t_local in the chunk, how many there
// are, and the destinations of the first.
struct DispatchTok {
  const uint4* x;             // the tokens' rows
  const int32_t* idx;         // the chunk's entries
  int tl;                     // first token of the chunk
  int nt;                     // tokens
  const int32_t* base;        // chunk bases of the chunk, per expert
  const int32_t* offsets;     // first position per expert
  int32_t* perm_dst;          // the tokens' k positions each
  int src;                    // perm_src value of the first token
  uint4* x_sh;                // bf16: copy of the rows for the shared expert (nullable)
  uint2* xq_sh;               // FP8: quantised rows and scales for the shared expert (nullable)
  float* xs_sh;
};

// Position of entry (t, j): offsets[e] + (entries of e in earlier chunks) +
// (entries of e before it in this chunk), e its expert; positions increase with
// (t, j) inside every segment.  An expert outside [0, E) is recorded and has none.
template <bool FP8, int TOK>
__device__ __forceinline__ void dispatch_tokens(const DispatchTok& d, int V, int k, int E, long long nk,
                                                void* __restrict__ x_perm_v, float* __restrict__ xs,
                                                int32_t* __restrict__ perm_src, uint32_t* status) {
  constexpr int kPer = kDispatchThreads / TOK;       // threads per token
  constexpr int kRank = kPer / kMaxTopK;             // threads that rank an entry
  static_assert(kPer % 32 == 0 && kChunkTokens % TOK == 0, "whole warps per token, tokens of one chunk");
  __shared__ __align__(16) int s_e[kDispatchThreads];  // the chunk's entries up to this CTA's last
  __shared__ int s_pos[TOK * kMaxTopK];
  const int tid = threadIdx.x, lane = tid & 31;
  const int tk = warp_token<TOK>(), vt = tid % kPer;  // this thread's token and first vector
  const bool live = tk < d.nt;
  const uint4* row = d.x + static_cast<long long>(tk) * V;
  uint4 a[kDispatchAhead];
#pragma unroll
  for (int i = 0; i < kDispatchAhead; ++i)
    if (live && vt + i * kPer < V) a[i] = ld_dep(row + vt + i * kPer);
  const int first = d.tl * k;
  s_e[tid] = tid < first + d.nt * k ? ld_dep(d.idx + tid) : -1;
  __syncthreads();
  {
    // entry (qt, j) by kRank consecutive threads
    const int q = tid / kRank, part = tid % kRank, qt = q / kMaxTopK, j = q % kMaxTopK;
    const bool entry = j < k && qt < d.nt;
    const int i = first + qt * k + j;
    int e = entry ? s_e[i] : -1, at = 0;
    if (e < 0 || e >= E) {
      if (entry && part == 0) record_status(status, ST_BAD_EXPERT_INDEX);
      e = -1;
    }
    if (e >= 0 && part == 0) at = ld_dep(d.offsets + e) + ld_dep(d.base + e);
    int before = 0;
    if (e >= 0) {
#pragma unroll 1
      for (int c = part; 4 * c < i; c += kRank) {
        const int4 o = reinterpret_cast<const int4*>(s_e)[c];
        before += (o.x == e) + (o.y == e && 4 * c + 1 < i) + (o.z == e && 4 * c + 2 < i) + (o.w == e && 4 * c + 3 < i);
      }
    }
#pragma unroll
    for (int o = kRank / 2; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
    if (part == 0) {
      int pos = -1;
      if (e >= 0) {
        pos = at + before;
        if (pos < 0 || pos >= nk) {
          record_status(status, ST_BAD_POSITION);
          pos = -1;
        }
      }
      s_pos[q] = pos;
      if (entry) d.perm_dst[qt * k + j] = pos;
      if (pos >= 0) perm_src[pos] = d.src + qt;
    }
  }
  __syncthreads();
  if (!live) return;
  int p[kMaxTopK];
#pragma unroll
  for (int j = 0; j < kMaxTopK; ++j) p[j] = s_pos[tk * kMaxTopK + j];
  for (int v0 = vt; v0 < V; v0 += kDispatchAhead * kPer) {
    if (v0 != vt) {
#pragma unroll
      for (int i = 0; i < kDispatchAhead; ++i)
        if (v0 + i * kPer < V) a[i] = ld_dep(row + v0 + i * kPer);
    }
#pragma unroll
    for (int i = 0; i < kDispatchAhead; ++i) {
      const int v = v0 + i * kPer;
      if (v < V) {  // (V is a multiple of 32: whole warps)
        if constexpr (!FP8) {
          uint4* x_perm = static_cast<uint4*>(x_perm_v);
#pragma unroll
          for (int j = 0; j < kMaxTopK; ++j)
            if (p[j] >= 0) x_perm[static_cast<long long>(p[j]) * V + v] = a[i];
          if (d.x_sh) d.x_sh[static_cast<long long>(tk) * V + v] = a[i];
        } else {
          // 8 values -> 8 bytes; one scale per 16 vectors (128 channels)
          uint2* xq = static_cast<uint2*>(x_perm_v);
          float scale;
          const uint2 q = quantize8(a[i], scale);
          const int nb = V / 16, blk = v >> 4;
          const bool head = (lane & 15) == 0;
#pragma unroll
          for (int j = 0; j < kMaxTopK; ++j)
            if (p[j] >= 0) {
              xq[static_cast<long long>(p[j]) * V + v] = q;
              if (head) xs[static_cast<long long>(p[j]) * nb + blk] = scale;
            }
          if (d.xq_sh) {
            d.xq_sh[static_cast<long long>(tk) * V + v] = q;
            if (head) d.xs_sh[tk * nb + blk] = scale;
          }
        }
      }
    }
  }
}

template <bool FP8, int TOK>
__global__ void __launch_bounds__(kDispatchThreads)
    dispatch_kernel(const uint4* x, int n, int V, int k, int E, const int32_t* idx, const int32_t* chunk_base,
                    void* __restrict__ x_perm_v, float* __restrict__ xs, uint2* __restrict__ xq_sh,
                    float* __restrict__ xs_sh, int32_t* __restrict__ perm_src, int32_t* __restrict__ perm_dst,
                    uint32_t* status, const DispatchSeg seg) {
  pdl_wait();
  pdl_launch();
  const int t = blockIdx.x * TOK, c = t / kChunkTokens;
  DispatchTok d;
  d.x = x + static_cast<long long>(t) * V;
  d.idx = idx + static_cast<long long>(c) * kChunkTokens * k;
  d.tl = t % kChunkTokens;
  d.nt = min(TOK, n - t);
  d.base = chunk_base + static_cast<long long>(seg.chunk0 + c) * E;
  d.offsets = seg.expert_offsets;
  d.perm_dst = perm_dst + static_cast<long long>(t) * k;
  d.src = seg.tok0 + t;
  d.x_sh = seg.x_sh ? static_cast<uint4*>(seg.x_sh) + static_cast<long long>(t) * V : nullptr;
  d.xq_sh = xq_sh ? xq_sh + static_cast<long long>(t) * V : nullptr;
  d.xs_sh = xq_sh ? xs_sh + static_cast<long long>(t) * (V / 16) : nullptr;
  dispatch_tokens<FP8, TOK>(d, V, k, E, seg.rows_total, x_perm_v, xs, perm_src, status);
}

// Dispatch of a mailbox round: item q is the q % (32 / TOK)-th group of TOK tokens
// of the round's chunk q / (32 / TOK) in the scan's order (the row map lists the
// claimed posts' histogram rows, post after post); CTA b takes the items b, b +
// gridDim.x, ...  A post's tokens come at r->tok0[i] in the combined order; its
// histogram rows and chunk bases are its slot's, its idx / perm_dst entries its
// slot's region.
template <bool FP8, int TOK>
__global__ void __launch_bounds__(kDispatchThreads, 5)
    dispatch_mbox_kernel(const MboxRound* r, const MboxGeom g, const int32_t* rowmap, const int32_t* idx,
                         const int32_t* chunk_base, const int32_t* offsets, void* __restrict__ x_perm_v,
                         float* __restrict__ xs, void* __restrict__ x_sh, float* __restrict__ xs_sh,
                         int32_t* __restrict__ perm_src, int32_t* __restrict__ perm_dst, uint32_t* status) {
  pdl_wait();
  pdl_launch();
  constexpr int kGroups = kChunkTokens / TOK;
  const int V = g.H / 8, items = r->chunks_total * kGroups;
  const long long nk = static_cast<long long>(r->n_total) * g.k;
  for (int q = blockIdx.x; q < items; q += gridDim.x) {
    const int hrow = ld_dep(rowmap + q / kGroups);
    const int slot = hrow / g.slot_chunks, c = hrow % g.slot_chunks;
    const int i = r->index_of[slot], tl = q % kGroups * TOK, t = c * kChunkTokens + tl;
    const int nt = min(TOK, r->n[i] - t);
    if (nt <= 0) continue;
    const int tg = r->tok0[i] + t;
    const int32_t* sidx = idx + static_cast<long long>(slot) * g.slot_tokens * g.k;
    DispatchTok d;
    d.x = static_cast<const uint4*>(r->x[i]) + static_cast<long long>(t) * V;
    d.idx = sidx + static_cast<long long>(c) * kChunkTokens * g.k;
    d.tl = tl;
    d.nt = nt;
    d.base = chunk_base + static_cast<long long>(hrow) * g.E;
    d.offsets = offsets;
    d.perm_dst = perm_dst + (static_cast<long long>(slot) * g.slot_tokens + t) * g.k;
    d.src = tg;
    d.x_sh = !FP8 && x_sh ? static_cast<uint4*>(x_sh) + static_cast<long long>(tg) * V : nullptr;
    d.xq_sh = FP8 && x_sh ? static_cast<uint2*>(x_sh) + static_cast<long long>(tg) * V : nullptr;
    d.xs_sh = FP8 && x_sh ? xs_sh + static_cast<long long>(tg) * (V / 16) : nullptr;
    dispatch_tokens<FP8, TOK>(d, V, g.k, g.E, nk, x_perm_v, xs, perm_src, status);
    __syncthreads();  // the shared tables are rewritten by the next item
  }
}

// Rows of bf16 to e4m3 with a scale per 128 channels; one warp per row.
__global__ void __launch_bounds__(256) quantize_rows_kernel(const uint4* x, int rows, int V,
                                                            uint2* __restrict__ q, float* __restrict__ s) {
  pdl_wait();
  pdl_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long r = static_cast<long long>(blockIdx.x) * 8 + warp;
  if (r >= rows) return;
  const int nb = V / 16;
  constexpr int kAhead = 4;  // vectors of the row per lane in flight
  for (int v0 = lane; v0 < V; v0 += 32 * kAhead) {
    uint4 a[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
      if (v0 + 32 * i < V) a[i] = ld_dep(x + r * V + v0 + 32 * i);
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int v = v0 + 32 * i;
      if (v >= V) break;
      float scale;
      q[r * V + v] = quantize8(a[i], scale);
      if ((lane & 15) == 0) s[r * nb + (v >> 4)] = scale;
    }
  }
}

// acc += w y for a vector of eight bf16; the shared expert's row is added plainly.
__device__ __forceinline__ void add_row(float (&acc)[8], float w, const uint4& y) {
  acc[0] = fmaf(w, bf16_lo(y.x), acc[0]);
  acc[1] = fmaf(w, bf16_hi(y.x), acc[1]);
  acc[2] = fmaf(w, bf16_lo(y.y), acc[2]);
  acc[3] = fmaf(w, bf16_hi(y.y), acc[3]);
  acc[4] = fmaf(w, bf16_lo(y.z), acc[4]);
  acc[5] = fmaf(w, bf16_hi(y.z), acc[5]);
  acc[6] = fmaf(w, bf16_lo(y.w), acc[6]);
  acc[7] = fmaf(w, bf16_hi(y.w), acc[7]);
}
__device__ __forceinline__ void add_shared(float (&acc)[8], const uint4& s) {
  acc[0] += bf16_lo(s.x);
  acc[1] += bf16_hi(s.x);
  acc[2] += bf16_lo(s.y);
  acc[3] += bf16_hi(s.y);
  acc[4] += bf16_lo(s.z);
  acc[5] += bf16_hi(s.z);
  acc[6] += bf16_lo(s.w);
  acc[7] += bf16_hi(s.w);
}
__device__ __forceinline__ uint4 pack_row(const float (&acc)[8]) {
  return make_uint4(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[2], acc[3]), pack_bf16x2(acc[4], acc[5]),
                    pack_bf16x2(acc[6], acc[7]));
}

constexpr int kCombineThreads = 256;
// CTAs per SM (register cap): one token per CTA, several
constexpr int kCombineCtas = 3, kCombineCtasMany = 4;
constexpr int kSms = 152;

// A CTA of 256 threads takes TOK tokens, 256 / TOK threads each: out[t] = sum_j
// w[t,j] y_perm[perm_dst[t,j]] (+ y_sh[t]), fp32 fused multiply-adds in slot
// order, then the shared row, then bf16.  Bound by HBM reads (k + 1 rows per
// token).
// The body for one token by PER threads, this one the vt-th: w_t, pd_t its k
// weights and positions, y_sh_t its shared-expert row (nullable), out_t its
// output row.
template <int PER>
__device__ __forceinline__ void combine_token(const uint4* y_perm, const uint4* y_sh_t, const float* w_t,
                                              const int32_t* pd_t, int V, int k, uint4* __restrict__ out_t,
                                              uint32_t* status, long long nk, int vt) {
  int p[kMaxTopK];
  float wj[kMaxTopK];
#pragma unroll
  for (int j = 0; j < kMaxTopK; ++j) {
    p[j] = -1;
    wj[j] = 0.f;
    if (j < k) {
      p[j] = pd_t[j];
      wj[j] = w_t[j];
      if (p[j] < 0 || p[j] >= nk) {
        if (vt == 0) record_status(status, ST_BAD_POSITION);
        p[j] = -1;
      }
    }
  }
#pragma unroll(PER == kCombineThreads ? 2 : 1)
  for (int v = vt; v < V; v += PER) {
    uint4 yv[kMaxTopK];
#pragma unroll
    for (int j = 0; j < kMaxTopK; ++j)
      if (p[j] >= 0) yv[j] = ld_dep(y_perm + static_cast<long long>(p[j]) * V + v);
    float acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.f;
#pragma unroll
    for (int j = 0; j < kMaxTopK; ++j)
      if (p[j] >= 0) add_row(acc, wj[j], yv[j]);
    if (y_sh_t) add_shared(acc, ld_dep(y_sh_t + v));
    out_t[v] = pack_row(acc);
  }
}

template <int TOK>
__global__ void __launch_bounds__(kCombineThreads, TOK == 1 ? kCombineCtas : kCombineCtasMany)
    combine_kernel(const uint4* y_perm, const uint4* y_sh, const float* w, const int32_t* perm_dst, int n, int V,
                   int k, uint4* __restrict__ out, uint32_t* status, long long nk) {
  pdl_wait();
  pdl_launch();
  constexpr int kPer = kCombineThreads / TOK;
  const int t = blockIdx.x * TOK + warp_token<TOK>();
  if (t >= n) return;
  const long long tk = static_cast<long long>(t) * k, tv = static_cast<long long>(t) * V;
  combine_token<kPer>(y_perm, y_sh ? y_sh + tv : nullptr, w + tk, perm_dst + tk, V, k, out + tv, status, nk,
                      threadIdx.x % kPer);
}

// The claimed post of a round that holds combined token tg.
__device__ __forceinline__ int mbox_post(const MboxRound* r, int tg) {
  int lo = 0, hi = r->count;  // the last claimed post starting at or before tg
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (r->tok0[mid] <= tg) lo = mid; else hi = mid;
  }
  return lo;
}

// Combine of a mailbox round: CTA b combines the groups of TOK tokens b, b +
// gridDim.x, ... of the round's combined token order (the claimed posts one
// after the other).  A token's post writes into its own output; its weights and
// positions are in its slot's region, its shared-expert row at its place in the
// combined order.
template <int TOK>
__global__ void __launch_bounds__(kCombineThreads, TOK == 1 ? kCombineCtas : kCombineCtasMany)
    combine_mbox_kernel(const MboxRound* r, const MboxGeom g, const uint4* y_perm, const uint4* y_sh, const float* w,
                        const int32_t* perm_dst, uint32_t* status) {
  pdl_wait();
  pdl_launch();
  constexpr int kPer = kCombineThreads / TOK;
  const int n_total = r->n_total;
  const int V = g.H / 8;
  const long long nk = static_cast<long long>(n_total) * g.k;
  for (int tg = blockIdx.x * TOK + warp_token<TOK>(); tg < n_total; tg += gridDim.x * TOK) {
    const int i = mbox_post(r, tg);
    const int t = tg - r->tok0[i];
    const long long tk = (static_cast<long long>(r->slot[i]) * g.slot_tokens + t) * g.k;
    combine_token<kPer>(y_perm, y_sh ? y_sh + static_cast<long long>(tg) * V : nullptr, w + tk, perm_dst + tk, V, g.k,
                        static_cast<uint4*>(r->out[i]) + static_cast<long long>(t) * V, status, nk,
                        threadIdx.x % kPer);
  }
}

// Tile-contiguous weights: 128-byte row pieces grouped per GEMM box.
// dst box (e, nt, kb) = 256 consecutive rows of 128 B: rows nt*256 .. of
// expert e's packed matrix, bytes [kb*128, kb*128 + 128) of each row; one box
// is one contiguous 32 KB read from HBM.  A gate/up tile holds 128 gate (a) and
// the matching 128 up (b) rows, alternating in groups of 1 << log_unit rows.
// R: packed rows per expert; V: 16-byte units per row.
__global__ void retile_kernel(const uint4* __restrict__ a, const uint4* __restrict__ b, int E, int R, int V,
                              bool gate_up, int log_unit, uint4* __restrict__ dst) {
  const int KB = V / 8, NT = R / 256;
  const long long total = static_cast<long long>(E) * R * V;
  for (long long q = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; q < total;
       q += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int v8 = static_cast<int>(q & 7);
    long long t = q >> 3;
    const int r = static_cast<int>(t & 255);
    t >>= 8;
    const int kb = static_cast<int>(t % KB);
    t /= KB;
    const int nt = static_cast<int>(t % NT);
    const long long e = t / NT;
    const uint4* src;
    if (gate_up)
      src = ((r >> log_unit) & 1 ? b : a) +
            (e * (R / 2) + nt * 128 + ((r >> (log_unit + 1)) << log_unit) + (r & ((1 << log_unit) - 1))) * V;
    else
      src = a + (e * R + nt * 256 + r) * V;
    dst[q] = src[kb * 8 + v8];
  }
}

// Tokens per CTA for rows of V vectors.  With one token per CTA a call of many
// tokens is bound by the CTAs' own time (about 1.9 ns a token for dispatch, 4.2
// for combine) where a token moves few bytes: narrow rows, or few experts per
// token.  Measured on a GB300, us with 1 / 2 / 4 / 8 tokens per CTA (one warp per
// token, the form before: last figure):
//   dispatch, 65536 tokens: H 256, k 8 161 / 107 / 79 / 71 (91), H 512 183 / 129 /
//     113 / 116 (128), k 1 126 / 86 / 59 / 47 (55), H 1024, k 8 224 / 200 / 201 / 205
//     (218), H 1536, k 2 165 / 120 / 109 (117), H 2048 175 / 139 / 138 (146), H 4096,
//     k 1 196 / 174 / 175 (187); FP8 H 256 156 / 117 / 74 / 62 (98), H 1024 206 / 161 / 131 / 133 (191);
//     4096 tokens, k 8: H 4096 54 / 55 / 58 (68), H 7168 88 / 91 / 101 (104);
//   combine, 65536 tokens: H 256, k 8 275 / 114 / 69 / 54 (74), H 512 292 / 145 /
//     101 / 99 (116), H 1024 310 / 193 / 183 / 187 (208), H 2048, k 2 291 / 189 / 167
//     (240), H 4096, k 2 452 / 322 / 301 (433), k 4 537 / 423 / 414 (515); 4096 tokens,
//     k 8: H 4096 54 / 52 / 53 (55), H 7168 88 / 86 / 86 (92); 256 tokens: H 2048
//     6.1 / 7.9 / 7.8 (9.9), H 7168 8.8 / 10.4 / 15 (21).
int dispatch_tokens_per_cta(int V) { return V <= 64 ? 8 : V <= 256 ? 4 : V <= 512 ? 2 : 1; }
// (wide rows: one token per CTA while all CTAs are resident at once)
int combine_tokens_per_cta(int V, long long n) {
  return V <= 64 ? 8 : V <= 256 ? 4 : n > kCombineCtas * kSms ? 2 : 1;
}

template <typename F>
cudaError_t by_width(int tokens, F launch) {
  switch (tokens) {
    case 8: return launch(std::integral_constant<int, 8>{});
    case 4: return launch(std::integral_constant<int, 4>{});
    case 2: return launch(std::integral_constant<int, 2>{});
    default: return launch(std::integral_constant<int, 1>{});
  }
}

template <bool FP8>
cudaError_t dispatch(const void* x, int n, int H, int k, int E, const int32_t* idx, const int32_t* chunk_base,
                     void* x_perm, float* xs, uint2* xq_sh, float* xs_sh, int32_t* perm_src, int32_t* perm_dst,
                     uint32_t* status, const DispatchSeg& seg, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  return by_width(dispatch_tokens_per_cta(H / 8), [&](auto tok) {
    constexpr int TOK = decltype(tok)::value;
    return launch_pdl(dispatch_kernel<FP8, TOK>, ceil_div(n, TOK), kDispatchThreads, 0, s, 1,
                      static_cast<const uint4*>(x), n, H / 8, k, E, idx, chunk_base, x_perm, xs, xq_sh, xs_sh,
                      perm_src, perm_dst, status, seg);
  });
}

template <bool FP8>
cudaError_t dispatch_mbox(const MboxRound* r, MboxGeom g, const int32_t* rowmap, const int32_t* idx,
                          const int32_t* chunk_base, const int32_t* offsets, void* x_perm, float* xs, void* x_sh,
                          float* xs_sh, int32_t* perm_src, int32_t* perm_dst, uint32_t* status, cudaStream_t s) {
  return by_width(dispatch_tokens_per_cta(g.H / 8), [&](auto tok) {
    constexpr int TOK = decltype(tok)::value;
    // one post's items; more loop
    return launch_pdl(dispatch_mbox_kernel<FP8, TOK>, g.slot_chunks * (kChunkTokens / TOK), kDispatchThreads, 0, s, 1,
                      r, g, rowmap, idx, chunk_base, offsets, x_perm, xs, x_sh, xs_sh, perm_src, perm_dst, status);
  });
}

}  // namespace

cudaError_t launch_dispatch(const void* x, int n, int H, int k, int E, const int32_t* idx,
                            const int32_t* chunk_base, const int32_t* offsets, void* x_perm, int32_t* perm_src,
                            int32_t* perm_dst, uint32_t* status, cudaStream_t s) {
  DispatchSeg seg{};
  seg.expert_offsets = offsets;
  seg.rows_total = static_cast<long long>(n) * k;
  return launch_dispatch_seg(x, n, H, k, E, idx, chunk_base, x_perm, perm_src, perm_dst, status, seg, s);
}

cudaError_t launch_dispatch_seg(const void* x, int n, int H, int k, int E, const int32_t* idx,
                                const int32_t* chunk_base, void* x_perm, int32_t* perm_src, int32_t* perm_dst,
                                uint32_t* status, const DispatchSeg& seg, cudaStream_t s) {
  return dispatch<false>(x, n, H, k, E, idx, chunk_base, x_perm, nullptr, nullptr, nullptr, perm_src, perm_dst, status,
                         seg, s);
}

cudaError_t launch_dispatch_fp8(const void* x, int n, int H, int k, int E, const int32_t* idx,
                                const int32_t* chunk_base, const int32_t* offsets, void* xq, float* xs,
                                void* xq_sh, float* xs_sh, int32_t* perm_src, int32_t* perm_dst, uint32_t* status,
                                cudaStream_t s) {
  DispatchSeg seg{};
  seg.expert_offsets = offsets;
  seg.rows_total = static_cast<long long>(n) * k;
  return launch_dispatch_fp8_seg(x, n, H, k, E, idx, chunk_base, xq, xs, xq_sh, xs_sh, perm_src, perm_dst, status,
                                 seg, s);
}

cudaError_t launch_dispatch_fp8_seg(const void* x, int n, int H, int k, int E, const int32_t* idx,
                                    const int32_t* chunk_base, void* xq, float* xs, void* xq_sh, float* xs_sh,
                                    int32_t* perm_src, int32_t* perm_dst, uint32_t* status, const DispatchSeg& seg,
                                    cudaStream_t s) {
  return dispatch<true>(x, n, H, k, E, idx, chunk_base, xq, xs, static_cast<uint2*>(xq_sh), xs_sh, perm_src, perm_dst,
                        status, seg, s);
}

cudaError_t launch_quantize_rows(const void* x, int rows, int cols, void* q, float* s, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  return launch_pdl(quantize_rows_kernel, ceil_div(rows, 8), 256, 0, st, 1, static_cast<const uint4*>(x), rows,
                    cols / 8, static_cast<uint2*>(q), s);
}

cudaError_t launch_combine(const void* y_perm, const void* y_shared, const float* w,
                           const int32_t* perm_dst, int n, int H, int k, void* out, uint32_t* status,
                           cudaStream_t s, long long rows_total) {
  if (n <= 0) return cudaSuccess;
  return by_width(combine_tokens_per_cta(H / 8, n), [&](auto tok) {
    constexpr int TOK = decltype(tok)::value;
    return launch_pdl(combine_kernel<TOK>, ceil_div(n, TOK), kCombineThreads, 0, s, 1,
                      static_cast<const uint4*>(y_perm), static_cast<const uint4*>(y_shared), w, perm_dst, n, H / 8, k,
                      static_cast<uint4*>(out), status, rows_total > 0 ? rows_total : static_cast<long long>(n) * k);
  });
}

cudaError_t launch_dispatch_mbox(const MboxRound* r, MboxGeom g, const int32_t* rowmap, const int32_t* idx,
                                 const int32_t* chunk_base, const int32_t* offsets, void* x_perm, int32_t* perm_src,
                                 int32_t* perm_dst, void* x_sh, uint32_t* status, cudaStream_t s) {
  return dispatch_mbox<false>(r, g, rowmap, idx, chunk_base, offsets, x_perm, nullptr, x_sh, nullptr, perm_src,
                              perm_dst, status, s);
}

cudaError_t launch_dispatch_fp8_mbox(const MboxRound* r, MboxGeom g, const int32_t* rowmap, const int32_t* idx,
                                     const int32_t* chunk_base, const int32_t* offsets, void* xq, float* xs,
                                     void* xq_sh, float* xs_sh, int32_t* perm_src, int32_t* perm_dst,
                                     uint32_t* status, cudaStream_t s) {
  return dispatch_mbox<true>(r, g, rowmap, idx, chunk_base, offsets, xq, xs, xq_sh, xs_sh, perm_src, perm_dst, status,
                             s);
}

cudaError_t launch_combine_mbox(const MboxRound* r, MboxGeom g, const void* y_perm, const void* y_shared,
                                const float* w, const int32_t* perm_dst, uint32_t* status, cudaStream_t s) {
  // one post's tokens; more loop
  return by_width(combine_tokens_per_cta(g.H / 8, g.slot_tokens), [&](auto tok) {
    constexpr int TOK = decltype(tok)::value;
    return launch_pdl(combine_mbox_kernel<TOK>, ceil_div(g.slot_tokens, TOK), kCombineThreads, 0, s, 1, r, g,
                      static_cast<const uint4*>(y_perm), static_cast<const uint4*>(y_shared), w, perm_dst, status);
  });
}

cudaError_t launch_retile(const void* a, const void* b, int E, int R, long long row_bytes, bool gate_up, int log_unit,
                          void* dst, cudaStream_t s) {
  if (R % 256 != 0 || row_bytes % 128 != 0) return cudaErrorInvalidValue;
  retile_kernel<<<4096, 256, 0, s>>>(static_cast<const uint4*>(a), static_cast<const uint4*>(b), E, R,
                                     static_cast<int>(row_bytes / 16), gate_up, log_unit, static_cast<uint4*>(dst));
  return cudaGetLastError();
}

}  // namespace asap
