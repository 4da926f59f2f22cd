// Tuning parameters of the grouped GEMMs (ring depths per launch kind and
// the L2 priority of their loads), measured on GB300; build-time defines
// override them.
#pragma once

// Ring depths (stages of A [128 x 64] and B [256 x 64] bf16 boxes).  A k-step
// needs both boxes, so the pipeline depth that counts is that of the
// shallowest ring whose operand comes from HBM.  Measured at 4096 DeepSeek-V3
// tokens with the weights in tile-contiguous order (one 32 KB read per box):
// gate/up (GU) 4 + 4 (2.45 ms; 3 + 5: 2.58, 5 + 3: 2.69, 2 + 6: 3.23); down
// (DN) 4 + 4 (1.34 ms; 3 + 5: 1.36, 2 + 6: 1.64, 3 + 4: 1.37).  router (RT):
// activations from HBM, the 256 x H router weights from L2, 6 + 3 (70.5 ->
// 64.5 us at 16384 tokens).
#ifndef ASAP_RING_GU_A
#define ASAP_RING_GU_A 4
#endif
#ifndef ASAP_RING_GU_B
#define ASAP_RING_GU_B 4
#endif
#ifndef ASAP_RING_DN_A
#define ASAP_RING_DN_A 4
#endif
#ifndef ASAP_RING_DN_B
#define ASAP_RING_DN_B 4
#endif
// paired m-tiles (two 128-row m-tiles per tile sharing the weight boxes; short
// contractions and the down GEMM with the fused combine): A stages of 2 x 128 rows (32 KB) and B
// boxes of 32 KB, 3 + 3 stages.
#ifndef ASAP_RING_PAIR_A
#define ASAP_RING_PAIR_A 3
#endif
#ifndef ASAP_RING_PAIR_B
#define ASAP_RING_PAIR_B 3
#endif
// A launch of those kinds runs paired m-tiles when it has at least this many
// waves of them (estimated, one tile per SM per wave): with fewer the larger tile
// rounds the launch to whole waves more coarsely than it saves.
#ifndef ASAP_PAIR_MIN_WAVES
#define ASAP_PAIR_MIN_WAVES 3
#endif
#ifndef ASAP_RING_RT_A
#define ASAP_RING_RT_A 6
#endif
#ifndef ASAP_RING_RT_B
#define ASAP_RING_RT_B 3
#endif

// CTA pairs: weight and token stages of 16 KB per CTA, 13 in all.  Measured
// (gate/up us at 4096 / 8192 / 16384 DeepSeek-V3 tokens): 8 + 5 2339 / 3171 /
// 5746, 7 + 6 2323 / 3122 / 5642, 6 + 7 2309 / 3185 / 5641.
#ifndef ASAP_RING_CTA2_W
#define ASAP_RING_CTA2_W 7
#endif
#ifndef ASAP_RING_CTA2_X
#define ASAP_RING_CTA2_X 6
#endif

// FP8: weight stages of 32 KB, token stages of 16 KB.
#ifndef ASAP_RING_F8_W
#define ASAP_RING_F8_W 4
#endif
#ifndef ASAP_RING_F8_X
#define ASAP_RING_F8_X 4
#endif

// Tile order of the kernels with a scheduler warp.  Tiles of segments (and the
// shared expert) with several token tiles are tensor-bound, the others wait for
// the weight stream: bursts of ASAP_MIX_BURST of the former are spread evenly
// among the latter.  A burst reads few different weight tiles; with bursts of 1
// to 8 the shared expert's rows and weights were read from HBM again.  Measured
// (layer, us; Zipf 4096 and 8045 tokens, balanced 4096, FP8 Zipf 4096): one kind
// after the other 4110 / 5586 / 3731 / 2615; bursts of 8 3920 / 5332 / 3737 /
// 2538; 32 3846 / 5202 / 3633 / 2470; 128 4100 / 5379 / 3646 / 2487.
#ifndef ASAP_MIX_BURST
#define ASAP_MIX_BURST 32
#endif
// Inside a segment the n-tiles are walked per block of token tiles whose operand
// rows fill this much, so that they are read from HBM once (gate/up GEMM of 8045
// Zipf tokens, whose largest expert has 86 MB of rows: 3458 -> 3308 us; 16 or 64
// MB within 2 %).
#ifndef ASAP_BLOCK_BYTES
#define ASAP_BLOCK_BYTES (32 << 20)
#endif

// L2 priority of the grouped GEMMs' loads (0 normal, 1 evict-first, 2
// evict-last): activations (A) are re-read by every n-tile of their expert
// and stay evict-last; the bf16 weights (B) are read by the m-tiles of one
// expert at about the same time, which find them in L2 only at normal
// priority (measured on GB300 at 4096 DeepSeek-V3 tokens: gate/up 2.90 ->
// 2.59 ms, down 1.78 -> 1.54 ms against evict-first weights).  The FP8 GEMMs
// measured 2 % faster with evict-first weights.
#ifndef ASAP_HINT_BF16_A
#define ASAP_HINT_BF16_A 2
#endif
#ifndef ASAP_HINT_BF16_B
#define ASAP_HINT_BF16_B 0
#endif
// the down GEMM's activations (h), re-read by every n-tile of their expert:
// evict-last as for gate/up (measured: 1.33 ms; normal 1.35, evict-first 1.42)
#ifndef ASAP_HINT_BF16_DN_A
#define ASAP_HINT_BF16_DN_A ASAP_HINT_BF16_A
#endif
#ifndef ASAP_HINT_FP8_A
#define ASAP_HINT_FP8_A 2
#endif
#ifndef ASAP_HINT_FP8_B
#define ASAP_HINT_FP8_B 1
#endif
