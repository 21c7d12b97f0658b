// Shared declarations of the sm_100a routed-MoE library (internal; the public ABI is include/moe_b200.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/moe_b200.h"
#include "../../include/moe_b200_debug.h"

#define MOE_DEVINL __device__ __forceinline__

namespace moe {

// ---- workspace carving (host) ----------------------------------------------------------------
// ws = [ route counters (always first) | act bf16 [S,I] | permute block counts | ffn counters ]
struct WsLayout {
  size_t act_off, route_off, permute_off, ffn_off, total;
};

constexpr int kPermuteChunk = 1024;  // slots per CTA in the multi-CTA permute
constexpr size_t kAlign = 256;

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// native block-scaled FP4 variant (decode-sized batches): on average at most 32 rows per expert (2 passes of 16
// tokens over the weight stream).  Its scratch holds the E2M1 term rows (8 per row) of both projections' inputs:
// [8S, I/2] + [8S, I/32] scale bytes and [8S, H/2] + [8S, H/32]; and one completion counter per expert.
#ifndef MOE_NATIVE_MAX_SLOTS
#define MOE_NATIVE_MAX_SLOTS 6144            // measured crossover to the prefill-sized kernel at the production shape
#endif
#ifndef MOE_NATIVE_MAX_ROWS_PER_EXPERT
#define MOE_NATIVE_MAX_ROWS_PER_EXPERT 32    // on average: two passes of 16 tokens over an expert's weights
#endif
inline bool native_batch_ok(const moe_shape_t& s) {
  const long long S = static_cast<long long>(s.T) * s.k;
  return S <= MOE_NATIVE_MAX_SLOTS && S <= static_cast<long long>(MOE_NATIVE_MAX_ROWS_PER_EXPERT) * s.E;
}
inline size_t native_scratch_bytes(const moe_shape_t& s) {
  const size_t S = static_cast<size_t>(s.T) * s.k;
  return align_up(8 * S * (s.I / 2), kAlign) + align_up(8 * S * (s.I / 32), kAlign) + align_up(8 * S * (s.H / 2), kAlign) +
         align_up(8 * S * (s.H / 32), kAlign) + align_up(static_cast<size_t>(s.E) * 4, kAlign);
}

// beside it, in moe_workspace_bytes() alone: the term rows by token of batches whose front is one launch (see launch_route_sort)
constexpr int kFrontMaxTok = 256, kFrontMaxE = 256;
inline size_t native_token_bytes(const moe_shape_t& s) {
  if (s.T > kFrontMaxTok || s.E > kFrontMaxE) return 0;
  return align_up(static_cast<size_t>(8) * s.T * (s.H / 2), kAlign) + align_up(static_cast<size_t>(8) * s.T * (s.H / 32), kAlign) +
         align_up(static_cast<size_t>(s.T) * s.k * 4, kAlign);
}

// scratch of the quantised-activation variant: one operand row per sorted row (codes and scale bytes of the token rows
// and of the intermediate) and the per-expert counters
inline size_t native_q_scratch_bytes(const moe_shape_t& s) {
  const size_t S = static_cast<size_t>(s.T) * s.k;
  return align_up(S * (s.I / 2), kAlign) + align_up(S * (s.I / 32), kAlign) + align_up(S * (s.H / 2), kAlign) +
         align_up(S * (s.H / 32), kAlign) + align_up(static_cast<size_t>(s.E) * 4, kAlign);
}

// two-term E4M3 variant (moe_ffn_twoterm.cu): pass geometry, scratch and the sizes it is chosen for
struct TwoTermGeometry {
  int max_tok;                     // tokens per pass of an expert
  int sf_step;                     // bytes of token scale factors per pass and K step of 128
};
// By the average rows per expert: shared memory not taken by token rows holds more weight stages (5 at 64 tokens, 4 at 112, 3
// at 224), which is what a batch bound by the weight stream needs (2048 tokens, 64 rows per expert: 0.96 ms with four
// stages, 1.12 with three); larger passes read the weights fewer times.
inline TwoTermGeometry twoterm_geometry(const moe_shape_t& s) {
  const long long S = static_cast<long long>(s.T) * s.k;
  if (S <= 56LL * s.E) return TwoTermGeometry{64, 512};
  if (S <= 96LL * s.E) return TwoTermGeometry{112, 1024};
  return TwoTermGeometry{224, 2048};
}
struct TwoTermScratch {
  size_t xq, aq, sfx, sfa;  // E4M3 pair rows of the tokens [2S, H] and of the intermediate [2S, I], scale factors
  size_t marks, flags;      // what the terms do not hold: a byte per token row and piece of it, an int per expert and one for any
  size_t total;
};
inline TwoTermScratch twoterm_scratch(const moe_shape_t& s) {
  TwoTermScratch L;
  const TwoTermGeometry g = twoterm_geometry(s);
  const size_t S = static_cast<size_t>(s.T) * s.k;
  const size_t passes = (S < static_cast<size_t>(s.E) ? S : static_cast<size_t>(s.E)) + S / g.max_tok;  // at most
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += align_up(bytes, kAlign);
    return o;
  };
  L.xq = take(2 * S * s.H);
  L.aq = take(2 * S * s.I);
  L.sfx = take(passes * (s.H / 128) * g.sf_step);
  L.sfa = take(passes * (s.I / 128) * g.sf_step);
  L.marks = take(S * (s.H / 256));
  L.flags = take((static_cast<size_t>(s.E) + 1) * 4);
  L.total = off;
  return L;
}
// When it is chosen.  Measured on packed weights of 256 experts of 4096 x 2048, top-8, layers in a row: 64 tokens 527 us against
// 446 on the eight-term kernel, 128 tokens 608 and 533, 333 tokens 641 and 886, 768 tokens 743 and 1573 (for the line between
// them see twoterm_chosen); the expert-FFN call against the bf16
// kernel 1024 tokens 0.69 and 1.96 ms, 4096 tokens 1.56 and 2.05, 8192 tokens 2.9 and 3.3; at I = 256 1027 tokens take 0.22
// ms against 2.8 on the streaming kernel.  Below four rows per expert the eight-term kernel reads the weights as fast
// as HBM delivers them, in one launch less; with fewer items than SMs the finer items of the other kernels fill more of the
// chip.
inline bool twoterm_shape_ok(const moe_shape_t& s) { return s.H % 256 == 0 && s.I % 256 == 0; }
inline bool twoterm_batch_ok(const moe_shape_t& s) {
  const long long S = static_cast<long long>(s.T) * s.k;
  const long long groups = S / 224 > s.E ? S / 224 : (S < s.E ? S : s.E);
  const int tiles = s.I / 128 < s.H / 256 ? s.I / 128 : s.H / 256;
  if (!twoterm_shape_ok(s)) return false;
  // at least 128 items of (pass, 128 values of i or 256 output columns), that is 64 gate/up items of 256 i for the 74 CTA
  // pairs.  Where the layer is small as well the launches decide, and the kernels meet (this call / bf16 kernel, L2 cold: 64
  // experts of 512 x 512, 33 rows each 42 us and 42, 64 rows 45 and 48, 96 rows 51 and 50; 128 of them, 64 rows 66 and 81).
  if (S >= 1024 && S >= 4LL * s.E && groups * tiles >= 128) return true;
  // few large experts (a block's shared expert), whatever the number of items: one expert of 4096 x 2048, this call / the kernel
  // that takes it otherwise: 48 rows 51 us and 73 (streaming), 192 rows 84 and 241, 1024 rows 90 and 110 (bf16), 2048 rows 111
  // and 114, 3000 rows 154 and 202.
  return S > 32LL * s.E && tiles >= 16;
}

// quantised-activation variant on CTA pairs (moe_ffn_twoterm.cu): one operand row per sorted row, its scale factors in the order
// tensor memory wants, 2 KB per pass and K step of 256.  For batches that fill the chip with more than
// 64 rows per expert (one launch for both projections up to there).  256 experts of 4096 x 2048, top-8, the call: 2048
// tokens 0.63 ms on either kernel, 4096 tokens 0.74 ms against 1.04, 8192 tokens 1.24 against 1.62, 32768 tokens 3.9
// against 5.4.
constexpr int kQPairTok = 224;
struct QPairScratch {
  size_t xq, aq, sfx, sfa, total;
};
inline QPairScratch q_pair_scratch(const moe_shape_t& s) {
  QPairScratch L;
  const size_t S = static_cast<size_t>(s.T) * s.k;
  const size_t passes = (S < static_cast<size_t>(s.E) ? S : static_cast<size_t>(s.E)) + S / kQPairTok;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += align_up(bytes, kAlign);
    return o;
  };
  L.xq = take(S * s.H / 2);
  L.aq = take(S * s.I / 2);
  L.sfx = take(passes * (s.H / 256) * 2048);
  L.sfa = take(passes * (s.I / 256) * 2048);
  L.total = off;
  return L;
}
inline bool q_pair_batch_ok(const moe_shape_t& s) { return twoterm_batch_ok(s) && static_cast<long long>(s.T) * s.k > 64LL * s.E; }

inline WsLayout ws_layout(const moe_shape_t& s) {
  WsLayout L;
  const size_t S = static_cast<size_t>(s.T) * s.k;
  size_t off = 0;
  L.route_off = off;  // moe_route is given only (T, E, k): its block must not depend on H or I
  off += align_up((static_cast<size_t>(s.E) + 8) * 4, kAlign);
  L.act_off = off;  // bf16 act[S,I], or the scratch of the native variant
  const size_t act_bytes = align_up(S * s.I * 2, kAlign);
  const size_t nat_bytes = native_batch_ok(s) ? native_scratch_bytes(s) + native_token_bytes(s) : 0;
  const size_t twoterm_bytes = twoterm_batch_ok(s) ? twoterm_scratch(s).total : 0;
  size_t ffn_bytes = act_bytes > nat_bytes ? act_bytes : nat_bytes;
  ffn_bytes = ffn_bytes > twoterm_bytes ? ffn_bytes : twoterm_bytes;
  off += ffn_bytes + kAlign;
  L.permute_off = off;
  const size_t nblk = (S + kPermuteChunk - 1) / kPermuteChunk;
  off += align_up(nblk * s.E * 4, kAlign);
  L.ffn_off = off;
  off += align_up(1024, kAlign);
  L.total = off;
  return L;
}

// ---- expert weights as the kernels see them --------------------------------------------------------
// Either the checkpoint's logical layout (rows of H/2 or I/2 packed bytes, rows of K/32 scale bytes), or the layout
// moe_prepack writes for shapes with H and I multiples of 512: the same bytes in tiles that are contiguous in memory,
//   codes:  tile (row / 128, byte / 128) = [128 rows][128 bytes], tiles of one row block consecutive along K
//   scales: tile (row / 128, byte / 16)  = [128 rows][16 bytes]
// so that what a CTA fetches per pipeline step (128 rows x 128 bytes of codes, 128 rows x 16 scale bytes) is one
// contiguous 16 KB / 2 KB run instead of 128 pieces 2 KB apart: DRAM pages are read whole (the decode_c64 expert-FFN
// call went from 0.516 to 0.48 ms on the same bytes).
struct ExpertWeights {
  const uint8_t *w13, *s13, *w2, *s2;
  bool blocked;
};
inline bool blocked_shape(const moe_shape_t& s) { return s.H % 512 == 0 && s.I % 512 == 0; }
struct PackedLayout {
  size_t w13, s13, w2, s2, total;
};
inline PackedLayout packed_layout(const moe_shape_t& s) {
  PackedLayout L;
  const size_t n = static_cast<size_t>(s.E) * s.H * s.I;  // weights of one projection pair half: E * H * I
  size_t off = 0;
  L.w13 = off;
  off += align_up(n, kAlign);        // E * 2I * H/2
  L.s13 = off;
  off += align_up(n / 16, kAlign);   // E * 2I * H/32
  L.w2 = off;
  off += align_up(n / 2, kAlign);    // E * H * I/2
  L.s2 = off;
  off += align_up(n / 32, kAlign);   // E * H * I/32
  L.total = off;
  return L;
}
int launch_prepack(const uint8_t* w13, const uint8_t* s13, const uint8_t* w2, const uint8_t* s2, const moe_shape_t& s,
                   uint8_t* packed, cudaStream_t st);

// ---- the status word the kernels report through (host) ---------------------------------------------
// The caller's, or - when the caller passed NULL - one word inside the library image per device, so that the rule
// "once one bounded wait has run out, every later wait of the grid gives up after a short spin" holds for every
// call: without a word to look at, one lost signal would cost the full limit in every wait that follows it.
// The library's own word is cleared by the call that uses it (`own` tells the launcher to arrange that: by a kernel
// of the call where one runs before the waits or after them, else by a memset node before the launches); nobody
// reads it on the host.  Calls that pass NULL and overlap on the GPU share it: a timeout in one may cut short the
// waits of the other, whose results are then reported nowhere - pass a status word to know.
struct StatusRef {
  int* word;
  bool own;
};
int resolve_status(int32_t* user_word, StatusRef* out);  // MOE_OK or MOE_ERR_CUDA

// ---- per-thread call record (host) -----------------------------------------------------------
void note_kernel(const char* name, int launches);

// ---- launchers implemented in the .cu files --------------------------------------------------
int launch_route(const float* logits, int T, int E, int k, int* ids, float* w, int* offsets, int* counters,
                 cudaStream_t st);
// Routing and stable sort in one launch, for batches that one thread-block cluster routes; beside it, where `split` is given, the
// tokens' rows are split into E2M1 term rows, stored by token (split->n_done counters are cleared).  inv_perm null: the routing
// alone; perm, offsets2 ({0, T}) may be null; `late`: the kernel in front may be the one that writes the logits.
struct FrontSplit {
  const __nv_bfloat16* x;
  uint8_t *aq, *sf;   // [T * 8, H / 2], [T * 8, H / 32]
  int* done;
  int n_done, H;
  int* status_clear;  // the library's own status word, or null
  int* tok;           // token of every sorted row, the top bit set where its expert has more than `most` rows
  int most;
};
bool route_sort_ok(int T, int E);
int launch_route_sort(const float* logits, int T, int E, int k, int* ids, float* w, int* offsets, int* perm, int* inv_perm, int* offsets2,
                      const FrontSplit* split, bool late, cudaStream_t st);
// the rows alone, in the order of a sort that is done (perm: slot of every sorted row)
int launch_gather_rows(const __nv_bfloat16* x, const int* perm, const moe_shape_t& s, __nv_bfloat16* x_perm, cudaStream_t st);
// (x_perm null: the sort alone, no rows are copied)
int launch_permute(const __nv_bfloat16* x, const int* ids, const int* offsets, const moe_shape_t& s,
                   __nv_bfloat16* x_perm, int* perm, int* inv_perm, int* block_counts, cudaStream_t st,
                   const int* range_lo = nullptr, const int* range_hi = nullptr);
// routing and sort of batches that no cluster routes, in a call that makes both (x_perm null: no rows).  offsets is written by the
// sort, and up to 4096 slots by its last CTA after the launch has let its dependents go: whatever is launched next is told so
// (offsets_late) or is a plain launch
bool route_permute_ok(const moe_shape_t& s);
int launch_route_permute(const float* logits, const __nv_bfloat16* x, const moe_shape_t& s, int* ids, float* w, int* offsets,
                         __nv_bfloat16* x_perm, int* perm, int* inv_perm, int* block_counts, cudaStream_t st);
// weight-streaming variant (any shape; the one for decode-sized batches)
int launch_expert_ffn_stream(const __nv_bfloat16* x_perm, const int* offsets, const uint8_t* w13, const uint8_t* s13,
                             const uint8_t* w2, const uint8_t* s2, const moe_shape_t& s, __nv_bfloat16* act, float* y_perm,
                             int* status_word, cudaStream_t st, float* const* row_dst = nullptr, const int* only = nullptr);
bool stream_shape_ok(const moe_shape_t& s);
// (`only`, in this one and the next: null, or device flags [E + 1] of an earlier kernel - experts whose flag is zero are left
// alone, and nothing is done where flag E is zero)
// tcgen05 grouped-GEMM variant (prefill-sized batches); umma_shape_ok says whether it applies
bool umma_shape_ok(const moe_shape_t& s);
int launch_expert_ffn_umma(const __nv_bfloat16* x_perm, const int* offsets, const ExpertWeights& w, const moe_shape_t& s,
                           __nv_bfloat16* act, float* y_perm, int* status_word, cudaStream_t st, float* const* row_dst = nullptr,
                           const int* only = nullptr);
// two-term E4M3 variant: packed codes and bf16 rows as two 8-bit terms on the block-scaled tensor-core path.  `choice` is the
// shape that fixes the pass geometry and the scratch layout (`s`, or the unsharded shape of an expert-parallel rank).
// `guard`: experts with blocks that two terms hold too little of are done again by a kernel that holds every bf16 value (see
// kTtLossyTokens); set where such a kernel would take the shape without this one.
bool twoterm_weights_ok(const void* w13, const void* w2);
struct TwoTermInput {
  const __nv_bfloat16* x;  // rows in sorted order; or, with the two tables of the routing, the tokens' rows
  const int* ids;          // [T, k] expert of every slot
  const int* inv_perm;     // [T, k] sorted row of every slot
  __nv_bfloat16* x_sorted; // with the tables: room for the rows in sorted order, of the experts that `guard` does again
  bool offsets_late;       // with the tables: the kernel in front is the one that writes the offsets (likewise in launch_expert_ffn_native)
  bool write_rows;         // with the tables: x_sorted is the caller's and receives all rows
};
// `again_later`: the launches of `guard` that do experts again are left to launch_twoterm_again, before anything reads y_perm.
// `finished` (may be null), here and in launch_expert_ffn_native: every CTA of the last launch adds one when it is through; the
// grid's size in *n_cta.
int launch_expert_ffn_twoterm(const TwoTermInput& in, const int* offsets, const ExpertWeights& w, const moe_shape_t& s,
                           const moe_shape_t& choice, bool guard, void* scratch, float* y_perm, int* status_word, cudaStream_t st,
                           float* const* row_dst = nullptr, bool again_later = false, int* finished = nullptr, int* n_cta = nullptr);
int launch_twoterm_again(const TwoTermInput& in, const int* offsets, const ExpertWeights& w, const moe_shape_t& s, void* scratch, float* y_perm,
                         int* status_word, cudaStream_t st);
// chosen by the batch and the weights' alignment, where another kernel takes the shape as well: what one of those refuses
// (rows too long for the streaming kernel, its only one) stays refused
bool twoterm_chosen(const moe_shape_t& choice, const ExpertWeights& w);
bool twoterm_guarded(const moe_shape_t& choice, const ExpertWeights& w);
// quantised activations, batches that fill the chip; scratch of q_pair_scratch
int launch_expert_ffn_q_pair(const __nv_bfloat16* x_perm, const int* offsets, const ExpertWeights& w, const moe_shape_t& s,
                             void* scratch, float* y_perm, int* status_word, cudaStream_t st);
// the whole layer in one launch of one cluster, for layers whose weights fit its shared memory; the streaming kernel's bits
struct SmallLayerOut {
  int *ids, *offsets, *perm, *inv_perm;
  float *w, *y_perm;
  __nv_bfloat16 *x_perm, *out;
};
bool layer_small_ok(const moe_shape_t& s);
int launch_layer_small(const float* logits, const __nv_bfloat16* x, const ExpertWeights& w, const moe_shape_t& s, const SmallLayerOut& o,
                       cudaStream_t st);
int launch_combine(const float* y_perm, const int* inv_perm, const float* w, const moe_shape_t& s,
                   __nv_bfloat16* out, cudaStream_t st);
int launch_validate_scales(const uint8_t* scales, size_t n, int* bad, cudaStream_t st);

// native block-scaled FP4 variant; scratch of native_scratch_bytes
bool native_shape_ok(const moe_shape_t& s, const void* w13, const void* w2);
// the quantised-activation variant of the same kernel: any batch size; scratch of native_q_scratch_bytes
bool native_q_shape_ok(const moe_shape_t& s, const void* w13, const void* w2);
int launch_expert_ffn_native_q(const __nv_bfloat16* x_perm, const int* offsets, const ExpertWeights& w, const moe_shape_t& s,
                               void* scratch, float* y_perm, StatusRef status, cudaStream_t st, float* const* row_dst = nullptr);
int launch_expert_ffn_native(const __nv_bfloat16* x_perm, const int* offsets, const ExpertWeights& w, const moe_shape_t& s,
                             void* scratch, float* y_perm, StatusRef status, cudaStream_t st, float* const* row_dst = nullptr,
                             int* finished = nullptr, int* n_cta = nullptr, bool offsets_late = false);

// the native variant behind launch_route_sort: token rows by token (native_front_split says where that launch leaves them).  H a
// multiple of 512.
FrontSplit native_front_split(const __nv_bfloat16* x, const moe_shape_t& s, void* scratch, StatusRef status);
int launch_expert_ffn_native_tokens(const int* offsets, const ExpertWeights& w, const moe_shape_t& s, void* scratch,
                                    float* y_perm, StatusRef status, cudaStream_t st);

// the whole layer in one launch, for a handful of tokens on shapes the native variant takes (moe_forward);
// `sync` is the zeroed block of kForwardSyncBytes, `scratch` holds forward_fused_scratch_bytes
constexpr size_t kForwardSyncBytes = 8192;
// int indices inside that block (both one-launch kernels): [0, E) per-expert counters of the general kernel, then
constexpr int kSyncDone2 = 1024;      // per column tile of the output: warps that have stored their rows of a down item
constexpr int kSyncExit = 1024 + 64;  // CTAs that are through with the counters; the last one clears the block
constexpr int kSyncSplit = 1024 + 65; // general kernel: CTAs that have written their share of the tokens' term rows
// two words that no kernel ever writes: a call that finds one of them non-zero was given a block that was never
// cleared, reports MOE_ERR_WORKSPACE through the status word and does nothing (every CTA takes the same decision)
constexpr int kSyncCanary0 = 1024 + 66, kSyncCanary1 = 2047;
bool forward_fused_ok(const moe_shape_t& s, const void* w13, const void* w2);  // the kernel can take the shape
bool forward_fused_preferred(const moe_shape_t& s);                             // and is the faster choice (measured)
size_t forward_fused_scratch_bytes(const moe_shape_t& s);
int launch_forward_fused(const float* logits, const __nv_bfloat16* x, const ExpertWeights& w, const moe_shape_t& s,
                         __nv_bfloat16* out, int* ids_out, float* w_out, int* sync, void* scratch, StatusRef status,
                         cudaStream_t st);

// the whole layer for one token in one launch with the down projection split along K over pairs of CTAs (moe_forward
// at T = 1 where the shape allows it); `sync` as above, `scratch` holds decode_one_scratch_bytes
bool decode_one_ok(const moe_shape_t& s, const void* w13, const void* w2, int n_shared = 0);
size_t decode_one_scratch_bytes(const moe_shape_t& s, int n_shared = 0);
int launch_decode_one(const float* logits, const __nv_bfloat16* x, const ExpertWeights& w, const moe_shape_t& s,
                      __nv_bfloat16* out, int* ids_out, float* w_out, int* sync, void* scratch, StatusRef status,
                      cudaStream_t st, const ExpertWeights* shared = nullptr);

// router projection, join with the shared expert, and the shared expert's offsets {0, T} (moe_block.cu)
// Where the router projection stands in its stream.  kAlone: whatever comes next may read the logits as it starts.  kFront: what
// comes next is this library's and waits before it reads them, so it may set up meanwhile.  kBeside: likewise, and the logits
// are computed beside the launches in front, without waiting for them; x and w_router are complete.
enum class RouterOrder : int { kAlone, kFront, kBeside };
int launch_router_logits(const __nv_bfloat16* x, const __nv_bfloat16* w_router, int T, int H, int E, float* logits, int* status,
                         cudaStream_t st, RouterOrder order);
// expert-parallel sharding: the table of output rows (see moe_ep_row_table)
int launch_ep_row_table(const int* perm, const int* offsets, int k, int H, int e_begin, int e_end, float* const* owner_y, int world,
                        int tokens_per_rank, float** row_dst, cudaStream_t st, int max_rows);
int launch_combine_shared(const float* y_perm, const int* inv_perm, const float* w, const float* y_shared, const moe_shape_t& s,
                          __nv_bfloat16* out, cudaStream_t st);
int launch_shared_offsets(int* offsets2, int T, cudaStream_t st);  // offsets2: {0, T} and a counter, 0
int launch_shared_join(const int* finished, int n_cta, int* status, cudaStream_t st);

int sm_count();  // of the current device

// ---- per-device one-time set-up (host) ---------------------------------------------------------------
// cudaFuncSetAttribute and the SM count belong to a device, not to the process: a process that drives several GPUs
// through this library sets each kernel's attributes once on every device it calls from.
constexpr int kMaxDevices = 64;
int current_device();  // -1 if the runtime cannot tell
struct PerDeviceFlag {
  bool done[kMaxDevices] = {};
};
template <typename F>
inline bool once_per_device(PerDeviceFlag& f, F&& set) {
  const int d = current_device();
  if (d < 0 || d >= kMaxDevices) return false;
  if (!f.done[d]) {
    if (!set()) return false;
    f.done[d] = true;
  }
  return true;
}

// ---- programmatic dependent launch (host) ------------------------------------------------------
// The kernel may start while its predecessor in the stream is still running; it must execute
// griddepcontrol.wait before it reads anything the predecessor writes, and before it writes anything at all to
// global memory.  Most kernels here wait first and then release their own dependent; route_kernel, route_sort_kernel, layer_small_kernel,
// native_split_kernel, native_quant_rows_kernel, native_expand_kernel, twoterm_scatter_kernel and the expert-FFN kernels
// release theirs BEFORE they wait, so three or four neighbours of a chain (route, permute, split, expert FFN) can be
// resident together.  That is safe because of the rule above: whatever a kernel does before its wait only reads buffers
// that no kernel of the chain still in flight writes (logits, the weights, expert_offsets once the kernel that writes them has
// been waited for by one that had not let its dependents go: see offsets_late), and every
// global write comes after the wait, i.e. after everything launched earlier on the stream has completed - for the wait is
// for the launch in front only, and that has waited in its turn, whether it had work or not.  shared_offsets_kernel and
// shared_join_kernel release by ending; so does router_gemv_kernel but inside moe_ffn_block (see RouterOrder).
// One launch waits for nothing: the router projection beside the shared expert (RouterOrder::kBeside).  It starts when all
// CTAs of the launches in front have, the first of which ended before the next began; what it reads is complete by then,
// and it writes the logits, which only the launch behind it reads.  But its end says nothing of the launches in front, so
// those count their CTAs out and the join waits for the count.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ---- small device helpers ---------------------------------------------------------------------
MOE_DEVINL void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
MOE_DEVINL void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

MOE_DEVINL int warp_excl_scan(int v, int lane, int* total) {
  int incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += n;
  }
  *total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - v;
}

}  // namespace moe
