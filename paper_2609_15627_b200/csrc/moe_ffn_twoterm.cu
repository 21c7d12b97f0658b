// Expert FFN on the 8-bit block-scaled tensor-core path (tcgen05 kind::mxf8f6f4, CTA pairs): a persistent grouped GEMM
// that takes the packed E2M1 weights and their E8M0 scales as they are and the bf16 activations as two E4M3 terms.
//
// A bf16 value has 8 significant bits, an E4M3 value 4, so with one scale 2^s per 32 consecutive elements
//   x = 2^s * hi + 2^(s-5) * lo,   hi = e4m3(x / 2^s),   lo = e4m3((x / 2^s - hi) * 32),   block maximum in [2^7, 2^8) * 2^s
// is exact for every element within 2^14 of its block's maximum and off by at most 2^-22 of that maximum otherwise -
// below what one fp32 addition of a 4096-long sum rounds away, as long as that maximum is in the sum.  It need not be: its
// weight may be zero, and where one element of a block is 2^12 (2^14, 2^18) times the others they then carry a relative error
// of 3e-4 (7e-3, 0.5).  So where a kernel that holds every value would take the shape (twoterm_guarded), such blocks are
// found where they are split, and their experts are done again by that kernel, in launches that end at once when there are none
// (kTtLossyTokens, launch_again).  E2M1 x E4M3 products are exact and accumulate in fp32 in
// tensor memory, so the result is that of the bf16 x expanded-weight product up to summation order, at the same
// tensor-core time (two 8-bit MMAs of K = 32 take what two bf16 MMAs of K = 16 take) and without any expansion of
// weights: what the bf16 kernel spends on that (about 1.9 ms for 256 experts of 4096 x 2048, whatever the batch) is
// gone, and a batch that touches every expert runs at the rate its weights arrive from HBM.
//
// Two CTAs (a thread-block cluster, one TPC) work on one tile with cta_group::2 MMAs: M = 256 weight rows, 128 in either
// CTA's shared memory and accumulator lanes; N = the rows of one expert's tokens, of which either CTA holds half.  That
// halves what shared memory serves for the token operand and the number of instructions to issue: for 128 tokens, per
// K = 32 and M tile, 12 KB are read and 8 KB written per CTA in the 128 cycles of its two MMAs; with one CTA per tile it
// would be 16 and 12 KB, 219 of the 128 bytes a cycle that shared memory delivers.
//   gate/up: item = (expert, pass of tokens, 256 values of i): one M tile of gate rows, one of the matching up rows, so
//            gate and up of one i share a lane of the two accumulators and SwiGLU is local to a thread.
//   down:    item = (expert, pass, 256 rows) with two accumulators taking turns, or 512 rows in the narrow geometry.
// An MMA takes max(64, N/2) cycles on the tensor core, or what its issue takes, about 40.  Hence two forms of a pass:
//   stacked    (up to 112 tokens): one token operand of N = 2n rows, the n hi rows (the first CTA's half) and the n lo rows
//              (the second's); the epilogue adds column j and column n + j.
//   separate   (up to 224): hi and lo operands of N = n rows each, both accumulated into the same columns.
// Where half of the accumulator columns are enough the halves take turns, and the epilogue runs beside the next item.
//
// Warp roles (20 warps, one CTA per SM, persistent):
//   warp 0       weight producer: TMA with a 4-bit tensor map that unpacks codes to the operand's 8-bit containers; scale bytes
//   warp 1       first CTA: copies scale factors to tensor memory (tcgen05.cp), issues the MMAs, commits to both CTAs
//   warp 2       token producer: TMA of the E4M3 rows and of their scale factors (stored by the producing kernel in the
//                order tensor memory wants)
//   warp 3       weight scale bytes into tensor-memory order, in place in shared memory
//   warps 4..19  epilogue, four warps per lane quadrant taking column chunks in turn
// Every mbarrier wait is bounded and reports through the status word.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "moe_mxf4_device.cuh"
#include "moe_sm100_primitives.cuh"
#include "moe_tmap.cuh"

namespace moe {

namespace {

constexpr int kTtK = 128;                    // K per stage: one 128-byte swizzled row of 8-bit containers
constexpr int kTtTile = 128 * 128;           // a CTA's rows of one M tile of a stage
constexpr int kTtEpiWarps = 16;
constexpr int kTtFirstEpi = 4;
constexpr int kTtThreads = (kTtFirstEpi + kTtEpiWarps) * 32;
constexpr int kTtSfSlots = 3;                // weight scale ring: one slot = 128 rows x 16 bytes per M tile (4 K steps)
constexpr uint32_t kTtTmemCols = 512;
constexpr uint32_t kTtHalf = 112;            // columns of an accumulator in a small pass of two M tiles
constexpr uint32_t kTtFull = 224;            //   and in any other
constexpr uint32_t kTtColSf = 448;           // scale factors: two sets (K step parity) of 2 x 4 (weights), 8 (hi), 8 (lo)
constexpr uint32_t kTtSfSet = 24;
constexpr uint32_t kTtSfSetQ = 32;           //   quantised activations: 2 x 2 x 4 (weights: M tile, word), 2 x 8 (tokens)
constexpr int kTtMaxStages = 8;

// token operand boxes: 64, 32 and 16 rows
constexpr int kTtBoxes = 3;
struct alignas(64) TtTokMaps {
  CUtensorMap box[kTtBoxes];
  CUtensorMap sf;  // their scale factors, [pass][K / 128][sf_step] bytes as rows of 128: box of 4 rows
};

struct TtArgs {
  const uint8_t* sc;       // weight scale bytes (see sf_mode)
  uint8_t* aq;             // gate/up: output, E4M3 terms of the intermediate, hi rows [S, I] then lo rows [S, I]
  uint8_t* sfa;            //   and their scale factors [pass][I / 128][sf_step]
  float* y;                // down: output [S, H]
  float* const* row_dst;   // or null; else output row p goes to row_dst[p] (see y_row)
  const int* offsets;      // [E + 1]
  int* status;
  const uint4* marks;      // gate/up, guarded (else flags is null): bytes of the split kernel, `parts` per sorted row
  int* flags;              //   [E + 1] out: experts to be done again
  int parts;
  int E, K, R, I, S;       // R weight rows per expert (2I or H)
  int blocked;             // weights in moe_prepack's tile-contiguous layout (see ExpertWeights)
  int max_tok, sf_step;    // of the pass geometry (see TwoTermGeometry)
  int* finished;           // or null; every CTA adds one when its work is done
  int stages, t_bytes, sf_off;  // ring depth; token part of a stage, and where its scale factors begin (see tt_launch)
};

// A stage: kM weight tiles, then the token part (rows of hi and, in a separate pass, of lo; their scale factors)
struct TtSmem {
  uint32_t ring, stage, sf, bars, misc, prefix, total;
};
__host__ __device__ inline TtSmem tt_smem(int E, int nm, int stages, int t_bytes) {
  TtSmem m;
  uint32_t off = 0;
  m.ring = off;
  m.stage = static_cast<uint32_t>(nm * kTtTile + t_bytes);
  off += static_cast<uint32_t>(stages) * m.stage;
  m.sf = off;
  off += static_cast<uint32_t>(kTtSfSlots * nm) * 2048;
  m.bars = off;
  off += 64 * 8;
  m.misc = off;
  off += 64;
  m.prefix = off;  // passes of the experts before e, then expert_offsets
  off += 2 * (static_cast<uint32_t>(E) + 2) * 4;
  m.total = off;
  return m;
}

MOE_DEVINL int tt_find_expert(const int* prefix, int E, int g) {  // prefix[e] <= g < prefix[e + 1]
  int lo = 0, hi = E;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (prefix[mid] <= g) lo = mid; else hi = mid;
  }
  return lo;
}

// One pass: rows [row0, row0 + n) of the sorted order.  N is a multiple of 32 (M = 256 takes no other): an expert's
// passes are equal up to the rounding to 16 rows (stacked) or 32 (separate), and what is left for the last one is stacked if
// that form can take it - it rounds to half as many rows (272 columns for 257 to 272 rows instead of 288).
struct TtPass {
  int row0, n, nr, N;  // nr: rows of a term in a stacked operand; N: columns of one accumulator
  bool stacked;
};
template <bool kQ>
MOE_DEVINL int tt_pass_rows(int m, int max_tok) {
  const int np = (m + max_tok - 1) / max_tok;
  const int t = (m + np - 1) / np;
  return !kQ && t <= static_cast<int>(kTtHalf) ? (t + 15) & ~15 : (t + 31) & ~31;
}
template <bool kQ>
MOE_DEVINL TtPass tt_pass(int r_begin, int r_end, int pass, int max_tok) {
  TtPass p;
  const int m = r_end - r_begin;
  const int tp = tt_pass_rows<kQ>(m, max_tok);
  p.row0 = r_begin + pass * tp;
  p.n = min(tp, m - pass * tp);
  p.nr = (p.n + 15) & ~15;
  p.stacked = !kQ && p.n <= static_cast<int>(kTtHalf);
  p.N = p.stacked ? 2 * p.nr : (p.n + 31) & ~31;
  return p;
}
// Where the K steps in flight lie in the ring, and their barriers.  Usually in stages as large as the largest pass needs.  kFifo
// (passes of at most 64 tokens, few rows per expert): in KB, one behind the other, as large as their own pass needs, or at the
// start where the end has no room - with 16 rows of a term six steps instead of five (layers in a row, 333 tokens, 10 rows per
// expert: tiles 659.5 -> 645 us, weights in rows 729 -> 706; 210 tokens 642 -> 633).
// All roles of both CTAs step through the same sequence; step n of a fifo uses barrier n % kTtMaxStages.
MOE_DEVINL int tt_fifo_kb(const TtPass& p, int kM) { return (kM * kTtTile + p.nr * 128 + 512 + 1023) >> 10; }
template <bool kFifo>
struct TtRing {
  uint32_t stage;    // bytes of a stage
  int stages, size;  // stages; KB (kFifo)
  int s, off, n, free, freed;
  uint32_t ph;
  uint64_t taken;    // KB of the last eight steps, with what was skipped in front of them, the newest in the low byte
  uint32_t addr;     // of the step that `take` or `next` found
  int bar;
  uint32_t parity;
  MOE_DEVINL TtRing(uint32_t stage_bytes, int n_stages)
      : stage(stage_bytes), stages(n_stages), size(static_cast<int>(stage_bytes * n_stages >> 10)), s(0), off(0), n(0), free(size), freed(0), ph(0),
        taken(0), addr(0), bar(0), parity(0) {}
  MOE_DEVINL void next(int kb) {  // consumer
    if constexpr (kFifo) {
      const int at = off + kb > size ? 0 : off;
      off = at + kb;
      addr = static_cast<uint32_t>(at) << 10;
      bar = n & (kTtMaxStages - 1);
      parity = static_cast<uint32_t>(n / kTtMaxStages) & 1u;
      ++n;
    } else {
      addr = s * stage;
      bar = s;
      parity = ph;
      if (++s == stages) { s = 0; ph ^= 1u; }
    }
  }
  MOE_DEVINL void take(int kb, uint64_t* empty, int* status) {  // producer: the same, once it is free
    if constexpr (kFifo) {
      const int at = off + kb > size ? 0 : off, need = at == 0 && off != 0 ? size - off + kb : kb;
      free -= need;
      while (free < 0 || n - freed == kTtMaxStages) {
        const int f = freed++;
        free += static_cast<int>(taken >> (8 * (n - f - 1))) & 0xFF;
        mbar_wait_warp(&empty[f & (kTtMaxStages - 1)], static_cast<uint32_t>(f / kTtMaxStages) & 1u, status);
      }
      taken = (taken << 8) | static_cast<uint64_t>(need);
      next(kb);
    } else {
      mbar_wait_warp(&empty[s], ph ^ 1u, status);
      next(kb);
    }
  }
};
// passes of experts < e, for all e: one warp
MOE_DEVINL void tt_prefix(const int* offsets, int E, int max_tok, int* prefix, int lane) {
  int run = 0;
  for (int e0 = 0; e0 < E; e0 += 32) {
    const int e = e0 + lane;
    const int rows = (e < E) ? __ldg(offsets + e + 1) - __ldg(offsets + e) : 0;
    int tot;
    const int ex = warp_excl_scan((rows + max_tok - 1) / max_tok, lane, &tot);
    if (e < E) prefix[e] = run + ex;
    run += tot;
  }
  if (lane == 0) prefix[E] = run;
}
// byte of operand row r, K block k32 (0..3) inside a step's scale factors: 128-row chunks of [32 lanes][4 words]
MOE_DEVINL int tt_sf_byte(int r, int k32) { return (r >> 7) * 512 + (r & 31) * 16 + ((r >> 5) & 3) * 4 + k32; }

// Scale byte of a block (biased exponent of the block's maximum minus 7; at least 5, so that the lo terms' byte, 5 less,
// exists) and 1 / 2^s.  Blocks whose maximum is below 2^-115 lose bits at the bottom instead.
MOE_DEVINL uint32_t tt_scale(uint32_t amax_bits) { return max(amax_bits >> 23, 12u) - 7u; }
MOE_DEVINL float tt_inv(uint32_t sb) { return __uint_as_float((254u - sb) << 23); }
// Smallest magnitude (bits of a float, at least 1) that is certain to be held exactly in a block with this maximum: the last bit
// of a bf16 value 2^14 below the maximum's power of two is the lo term's last.  Smaller values lose their lowest
// bits, 2^-22 of the maximum at most.
MOE_DEVINL uint32_t tt_lossy_below(uint32_t amax_bits) {
  constexpr uint32_t k14 = (14u << 23) + 1u;
  return max(amax_bits & 0x7F800000u, k14) - k14 + 1u;
}
// Which experts are done again: those with a token block of at least kTtLossyTokens values below that bound, or a block of the
// intermediate with at least kTtLossyInter of them and no more than kTtLarge that reach 2^-10 of the maximum; or with a value that is
// not finite.  Batches of ordinary values have none: of normal values one in 10^4 is below the bound, of the products a
// SwiGLU makes of them one in 10^3 (six, eight in one block: less than 1e-14 of the blocks), and where gates in the tens leave
// half of a block next to zero the rest of it is large (four or fewer: 1e-6, so a block or so of a large batch).  With
// one element of every block 2^10 times the others half a percent of the token blocks are found, 4 % of the
// intermediate's; at 2^14 most.  What is left to the terms in an expert that is not done again is thus
// an error of 1e-5 of a block's norm without its few largest elements, at most 2^-22 of its maximum per element.
constexpr int kTtLossyTokens = 6, kTtLossyInter = 8, kTtLarge = 3;
// The decision for eight blocks of the intermediate, value t of a lane in half t & 1 of word t / 2, of which the first n count
// (the others are columns beyond the pass).  By a whole warp, after a cheaper look has found one of the eight suspect.
MOE_DEVINL bool tt_again(const uint32_t (&pk)[4], int n) {
  bool again = false;
#pragma unroll 1
  for (int t = 0; t < 8 && t < n; ++t) {
    const uint32_t w = t < 2 ? pk[0] : t < 4 ? pk[1] : t < 6 ? pk[2] : pk[3];
    const uint32_t v = ((t & 1) ? w & 0xFFFF0000u : w << 16) & 0x7FFFFFFFu;
    const uint32_t amax = __reduce_max_sync(0xffffffffu, v);
    const int lossy = __popc(__ballot_sync(0xffffffffu, v - 1u < tt_lossy_below(amax) - 1u));
    // (with an inexact value in it the maximum is above 2^-112)
    const int large = lossy > 0 ? __popc(__ballot_sync(0xffffffffu, v >= (amax & 0x7F800000u) - (10u << 23))) : 32;
    again |= amax >= 0x7F800000u || (lossy >= kTtLossyInter && large <= kTtLarge);
  }
  return again;
}
// Four values over their blocks' scales, as halves y (exact down to 2^-24, below the lo term's last bit) -> four hi and four lo
// codes, one per byte.  E4M3 is a half without its last seven mantissa bits and 8 less of exponent bias, subnormals
// included: the code of v is the half v / 2^8, rounded (half away from zero) by adding 0x40 to its bits, less the low
// seven.  So no conversion instruction is needed (the split kernel was bound by them: they kept their pipe 99.8 % busy).
// Values that are not finite come out as anything: where a block's maximum shows one, tt_nan_codes makes both infinity, which the 8-bit
// format has not, and NaN a NaN, so that a token with such a value gives non-finite outputs.
MOE_DEVINL __half2 tt_bits_half2(uint32_t u) { return *reinterpret_cast<const __half2*>(&u); }
MOE_DEVINL uint32_t tt_half2_bits(__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); }
MOE_DEVINL uint32_t tt_high_bytes(uint32_t u) { return ((u << 1) & 0x7F007F00u) | (u & 0x80FF80FFu); }  // a rounded half -> its code in the upper byte
MOE_DEVINL void tt_codes(__half2 y01, __half2 y23, uint32_t* hi, uint32_t* lo) {
  const __half2 k256 = __float2half2_rn(1.0f / 256.0f), k8 = __float2half2_rn(0.125f), km32 = __float2half2_rn(-32.0f);
  const uint32_t u0 = tt_half2_bits(__hmul2(y01, k256)) + 0x00400040u, u1 = tt_half2_bits(__hmul2(y23, k256)) + 0x00400040u;
  // (y - hi) * 32 / 2^8
  const __half2 r0 = __hfma2(tt_bits_half2(u0 & 0xFF80FF80u), km32, __hmul2(y01, k8));
  const __half2 r1 = __hfma2(tt_bits_half2(u1 & 0xFF80FF80u), km32, __hmul2(y23, k8));
  const uint32_t v0 = tt_half2_bits(r0) + 0x00400040u, v1 = tt_half2_bits(r1) + 0x00400040u;
  *hi = __byte_perm(tt_high_bytes(u0), tt_high_bytes(u1), 0x7531);
  *lo = __byte_perm(tt_high_bytes(v0), tt_high_bytes(v1), 0x7531);
}
MOE_DEVINL uint32_t tt_nan_codes(uint32_t hi, float a, float b, float c, float d) {  // NaN where the value is not finite
  auto bad = [](float v, uint32_t byte) { return (__float_as_uint(v) & 0x7F800000u) == 0x7F800000u ? 0xFFu << (8 * byte) : 0u; };
  const uint32_t m = bad(a, 0) | bad(b, 1) | bad(c, 2) | bad(d, 3);
  return (hi & ~m) | (0x7F7F7F7Fu & m);
}

// The same by conversion instructions, two values at a time (low byte: the first): fewer instructions, for the gate/up epilogue,
// which is not bound by their pipe but adds to the power of the MMAs beside it (whole layer at 8192 tokens against
// the bf16 kernel's: 1.29 with these, 1.25 with the integer form)
MOE_DEVINL void tt_codes_cvt(__half2 y, uint32_t* hi, uint32_t* lo) {
  const __nv_fp8x2_storage_t h = __nv_cvt_halfraw2_to_fp8x2(*reinterpret_cast<const __half2_raw*>(&y), __NV_SATFINITE, __NV_E4M3);
  const __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2(h, __NV_E4M3);
  const __half2 r = __hmul2(__hsub2(y, *reinterpret_cast<const __half2*>(&hr)), __float2half2_rn(32.0f));
  *hi = static_cast<uint32_t>(h);
  *lo = static_cast<uint32_t>(__nv_cvt_halfraw2_to_fp8x2(*reinterpret_cast<const __half2_raw*>(&r), __NV_SATFINITE, __NV_E4M3));
}

// ---- cta_group::2 forms of the primitives.  The issuing ones are called by a whole convergent warp and issued by one
// elected lane, always the same: operands then live in uniform registers.  Issued inside an `if (lane == 0)` every operand
// is moved there anew for each instruction, and a block-scaled MMA takes 63 to 115 cycles to issue, whatever its size ----
MOE_DEVINL uint32_t tt_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
MOE_DEVINL void tt_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
MOE_DEVINL void tt_tmem_alloc(uint32_t* holder_smem, uint32_t ncols) {  // one whole warp in either CTA
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder_smem)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
MOE_DEVINL void tt_tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// arrive on the same barrier of both CTAs when every MMA and copy issued so far has completed
MOE_DEVINL void tt_commit(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
      "h"(static_cast<unsigned short>(3))
      : "memory");
}
// Arrive on the first CTA's copy of a barrier, at CTA scope: the arrival says that something is over and carries no data from one
// CTA to the other.  Scale factors: the first CTA reads none of the second's; tcgen05.cp and the MMAs of cta_group::2 read either
// CTA's operands in that CTA, through its own asynchronous proxy, for which every writing lane's fence.proxy.async has
// completed its shared-memory writes before the warp meets and one lane arrives.  Accumulators: what tcgen05.wait::ld has
// returned is in registers, and nothing of it is left to be seen elsewhere.  So no release at cluster scope, which would order
// memory between the CTAs, is needed; it is not free either: with it (and the acquire at the other end) a call takes
// 8 to 13 % longer (mixed batch of 333 tokens 667 -> 763 us), whether the warp that writes the scale factors does it or one that
// does nothing else.
MOE_DEVINL void tt_arrive_first(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .b32 ra;\n\t"
      "mapa.shared::cluster.u32 ra, %0, 0;\n\t"
      "mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}" ::"r"(smem_u32(bar))
      : "memory");
}
// address of the first CTA's copy of a barrier
MOE_DEVINL uint32_t tt_first_addr(const void* p) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(ra) : "r"(smem_u32(p)));
  return static_cast<uint32_t>(warp_uniform(static_cast<int>(ra)));
}
// Tensor-map load into this CTA's shared memory that counts its bytes on a barrier of either CTA of the pair.  (A warp of
// the second CTA that passed its own barriers' phases on to the first took 700 cycles per remote arrival.)
MOE_DEVINL void tt_load_2d(uint32_t dst, const void* tmap, int x, int y, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4}], [%2];\n\t}" ::"r"(
          dst),
      "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
MOE_DEVINL void tt_load_2d_hint(uint32_t dst, const void* tmap, int x, int y, uint32_t bar, uint64_t policy) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2.L2::cache_hint [%0], [%1, {%3, %4}], "
      "[%2], %5;\n\t}" ::"r"(dst),
      "l"(tmap), "r"(bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}
MOE_DEVINL void tt_bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
MOE_DEVINL void tt_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar), "r"(bytes)
      : "memory");
}
// instruction descriptor without the scale byte index: A E2M1, B E4M3, UE8M0 scales, M = 256
MOE_DEVINL uint32_t tt_idesc(int N) { return (5u << 7) | (static_cast<uint32_t>(N >> 3) << 17) | (1u << 23) | (2u << 27); }
// One K step of 128: D[tmem] (+)= A[smem, E2M1 in 8-bit containers] * B[smem, E4M3]^T, K = 32 per instruction, one UE8M0
// scale per row and 32 elements (byte j of the scale words), descriptors advancing 32 bytes along the swizzled rows.
// kM M tiles share the token operand.
template <int kM>
MOE_DEVINL void tt_mma_step(uint32_t d0, uint32_t d1, uint64_t a0, uint64_t a1, uint64_t b, uint32_t idesc, uint32_t sfa0,
                            uint32_t sfa1, uint32_t sfb, uint32_t accumulate) {
  if constexpr (kM == 2)
    asm volatile(
        "{\n\t.reg .pred q, p, t;\n\t.reg .b64 a, b;\n\t.reg .b32 id;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.b32 p, %9, 0;\n\t"
        "setp.eq.b32 t, 0, 0;\n\t"
        "add.s64 a, %2, 0;\n\tadd.s64 b, %4, 0;\n\tadd.u32 id, %5, 0x00000000;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], p;\n\t"
        "add.s64 a, %3, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%1], a, b, id, [%7], [%8], p;\n\t"
        "add.s64 a, %2, 2;\n\tadd.s64 b, %4, 2;\n\tadd.u32 id, %5, 0x20000010;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], t;\n\t"
        "add.s64 a, %3, 2;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%1], a, b, id, [%7], [%8], t;\n\t"
        "add.s64 a, %2, 4;\n\tadd.s64 b, %4, 4;\n\tadd.u32 id, %5, 0x40000020;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], t;\n\t"
        "add.s64 a, %3, 4;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%1], a, b, id, [%7], [%8], t;\n\t"
        "add.s64 a, %2, 6;\n\tadd.s64 b, %4, 6;\n\tadd.u32 id, %5, 0x60000030;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], t;\n\t"
        "add.s64 a, %3, 6;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%1], a, b, id, [%7], [%8], t;\n\t"
        "}" ::"r"(d0), "r"(d1), "l"(a0), "l"(a1), "l"(b), "r"(idesc), "r"(sfa0), "r"(sfa1), "r"(sfb), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred q, p, t;\n\t.reg .b64 a, b;\n\t.reg .b32 id;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.b32 p, %9, 0;\n\t"
        "setp.eq.b32 t, 0, 0;\n\t"
        "add.s64 a, %2, 0;\n\tadd.s64 b, %4, 0;\n\tadd.u32 id, %5, 0x00000000;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], p;\n\t"
        "add.s64 a, %2, 2;\n\tadd.s64 b, %4, 2;\n\tadd.u32 id, %5, 0x20000010;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], t;\n\t"
        "add.s64 a, %2, 4;\n\tadd.s64 b, %4, 4;\n\tadd.u32 id, %5, 0x40000020;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], t;\n\t"
        "add.s64 a, %2, 6;\n\tadd.s64 b, %4, 6;\n\tadd.u32 id, %5, 0x60000030;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], a, b, id, [%6], [%8], t;\n\t"
        "}" ::"r"(d0), "r"(d1), "l"(a0), "l"(a1), "l"(b), "r"(idesc), "r"(sfa0), "r"(sfa1), "r"(sfb), "r"(accumulate)
        : "memory");
}
// The same for dense 4-bit operands, a K step of 256: K = 64 per instruction, two of a row's eight scales (one half of word j / 2,
// the words 4 columns apart for the weights, 8 for the tokens)
MOE_DEVINL uint32_t tt_idesc_mxf4(int N) { return (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) | (1u << 23) | (2u << 27); }
template <int kM>
MOE_DEVINL void tt_mma_step_mxf4(uint32_t d0, uint32_t d1, uint64_t a0, uint64_t a1, uint64_t b, uint32_t idesc, uint32_t sfa0,
                                 uint32_t sfa1, uint32_t sfb, uint32_t accumulate) {
  if constexpr (kM == 2)
    asm volatile(
        "{\n\t.reg .pred q, p, t;\n\t.reg .b64 a, b;\n\t.reg .b32 id, sa, sb;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.b32 p, %9, 0;\n\t"
        "setp.eq.b32 t, 0, 0;\n\t"
        "add.s64 a, %2, 0;\n\tadd.s64 b, %4, 0;\n\tadd.u32 id, %5, 0x00000000;\n\tadd.u32 sa, %6, 0;\n\tadd.u32 sb, %8, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], p;\n\t"
        "add.s64 a, %3, 0;\n\tadd.u32 sa, %7, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%1], a, b, id, [sa], [sb], p;\n\t"
        "add.s64 a, %2, 2;\n\tadd.s64 b, %4, 2;\n\tadd.u32 id, %5, 0x40000020;\n\tadd.u32 sa, %6, 0;\n\tadd.u32 sb, %8, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
        "add.s64 a, %3, 2;\n\tadd.u32 sa, %7, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%1], a, b, id, [sa], [sb], t;\n\t"
        "add.s64 a, %2, 4;\n\tadd.s64 b, %4, 4;\n\tadd.u32 id, %5, 0x00000000;\n\tadd.u32 sa, %6, 4;\n\tadd.u32 sb, %8, 8;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
        "add.s64 a, %3, 4;\n\tadd.u32 sa, %7, 4;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%1], a, b, id, [sa], [sb], t;\n\t"
        "add.s64 a, %2, 6;\n\tadd.s64 b, %4, 6;\n\tadd.u32 id, %5, 0x40000020;\n\tadd.u32 sa, %6, 4;\n\tadd.u32 sb, %8, 8;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
        "add.s64 a, %3, 6;\n\tadd.u32 sa, %7, 4;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%1], a, b, id, [sa], [sb], t;\n\t"
        "}" ::"r"(d0), "r"(d1), "l"(a0), "l"(a1), "l"(b), "r"(idesc), "r"(sfa0), "r"(sfa1), "r"(sfb), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred q, p, t;\n\t.reg .b64 a, b;\n\t.reg .b32 id, sa, sb;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.b32 p, %9, 0;\n\t"
        "setp.eq.b32 t, 0, 0;\n\t"
        "add.s64 a, %2, 0;\n\tadd.s64 b, %4, 0;\n\tadd.u32 id, %5, 0x00000000;\n\tadd.u32 sa, %6, 0;\n\tadd.u32 sb, %8, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], p;\n\t"
        "add.s64 a, %2, 2;\n\tadd.s64 b, %4, 2;\n\tadd.u32 id, %5, 0x40000020;\n\tadd.u32 sa, %6, 0;\n\tadd.u32 sb, %8, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
        "add.s64 a, %2, 4;\n\tadd.s64 b, %4, 4;\n\tadd.u32 id, %5, 0x00000000;\n\tadd.u32 sa, %6, 4;\n\tadd.u32 sb, %8, 8;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
        "add.s64 a, %2, 6;\n\tadd.s64 b, %4, 6;\n\tadd.u32 id, %5, 0x40000020;\n\tadd.u32 sa, %6, 4;\n\tadd.u32 sb, %8, 8;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
        "}" ::"r"(d0), "r"(d1), "l"(a0), "l"(a1), "l"(b), "r"(idesc), "r"(sfa0), "r"(sfa1), "r"(sfb), "r"(accumulate)
        : "memory");
}
// 512 bytes of scale factors in shared memory, [32 lanes][4 words], -> 4 columns of tensor memory, in all four lane
// quadrants, in either CTA from its own shared memory; ordered with the MMAs that the same lane issues before and after
MOE_DEVINL void tt_cp_sf(uint32_t taddr, uint32_t smem_addr) {
  const uint64_t desc = static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(128 >> 4) << 32) |
                        (static_cast<uint64_t>(1) << 46);  // no swizzle, 8-row groups 128 bytes apart
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;\n\t}" ::"r"(taddr), "l"(desc)
      : "memory");
}
MOE_DEVINL void tt_tmem_ld_32x8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}

MOE_DEVINL float tt_silu_mul(float g, float u) { return __fdividef(g, 1.0f + __expf(-g)) * u; }

// 4 x 4 byte transpose over lanes 4a..4a+3: in, byte t of lane l is (token t, row l); out, byte l of lane t
MOE_DEVINL uint32_t transpose_4x4(uint32_t w, int lane) {
  uint32_t p = __shfl_xor_sync(0xffffffffu, w, 1);
  w = (lane & 1) ? __byte_perm(w, p, 0x3715) : __byte_perm(w, p, 0x6240);
  p = __shfl_xor_sync(0xffffffffu, w, 2);
  return (lane & 2) ? __byte_perm(w, p, 0x3276) : __byte_perm(w, p, 0x5410);
}

}  // namespace

// Where a sorted row's scale factors go: bytes from the start of the buffer to the hi word of its first K step, and from
// there to the lo word (quantised activations: to the step's second word)
struct TtSfPlace {
  size_t hi;
  int lo;
};
// What it takes to know, per expert, in shared memory (tt_tables fills it): first row, passes before, rows per pass
struct TtTables {
  int *prefix, *off, *tp;
};
constexpr int kTtTableInts = 3;
template <bool kQ>
MOE_DEVINL TtTables tt_tables(int* smem, const int* offsets, int E, int max_tok) {  // whole block
  const TtTables t{smem, smem + E + 1, smem + 2 * (E + 1)};
  if (threadIdx.x < 32) tt_prefix(offsets, E, max_tok, t.prefix, static_cast<int>(threadIdx.x));
  for (int e = threadIdx.x; e <= E; e += blockDim.x) {
    const int lo = __ldg(offsets + e), hi = e < E ? __ldg(offsets + e + 1) : lo;
    t.off[e] = lo;
    t.tp[e] = hi > lo ? tt_pass_rows<kQ>(hi - lo, max_tok) : 1;
  }
  __syncthreads();
  return t;
}
template <bool kQ>
MOE_DEVINL TtSfPlace tt_sf_place(int p, int e, const TtTables& t, int H, int sf_step) {
  const int d = p - t.off[e], tp = t.tp[e];
  int pass = static_cast<int>(__fdividef(static_cast<float>(d), static_cast<float>(tp)));
  pass -= pass * tp > d;  // (the quotient is off by less than one)
  pass += (pass + 1) * tp <= d;
  const int r = d - pass * tp, hi = tt_sf_byte(r, 0);
  TtSfPlace at{static_cast<size_t>(t.prefix[e] + pass) * (H / (kQ ? 256 : 128)) * sf_step + hi, 1024};
  const int n = min(tp, t.off[e + 1] - t.off[e] - pass * tp);
  if (!kQ && n <= static_cast<int>(kTtHalf)) at.lo = tt_sf_byte(((n + 15) & ~15) + r, 0) - hi;  // stacked
  return at;
}
// A warp's 256 consecutive values of a row, 16 bytes per lane -> 8 hi and 8 lo codes per lane, and the scale word of the K
// step its half warp holds.  Four lanes share a block of 32.  Bound by issue where its input is in L2: the block maximum on
// 16-bit pairs and the terms on pairs of halves.
// kGuard: says whether one of the eight blocks is to be done again (the same in all lanes).
template <bool kGuard>
MOE_DEVINL bool tt_split_256(const uint4& v, int lane, uint2* hi, uint2* lo, uint32_t* word) {
  uint32_t w[4] = {v.x, v.y, v.z, v.w};
  constexpr uint32_t kAbs = 0x7FFF7FFFu;
  uint32_t m2 = __vmaxu2(__vmaxu2(w[0] & kAbs, w[1] & kAbs), __vmaxu2(w[2] & kAbs, w[3] & kAbs));
  m2 = __vmaxu2(m2, __shfl_xor_sync(0xffffffffu, m2, 1));
  m2 = __vmaxu2(m2, __shfl_xor_sync(0xffffffffu, m2, 2));
  const uint32_t amax = max(m2 & 0xFFFFu, m2 >> 16) << 16;
  const uint32_t sb = tt_scale(amax);
  const float inv = tt_inv(sb);
  uint32_t h[2], l[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float f[4] = {__uint_as_float(w[2 * j] << 16), __uint_as_float(w[2 * j] & 0xFFFF0000u), __uint_as_float(w[2 * j + 1] << 16),
                        __uint_as_float(w[2 * j + 1] & 0xFFFF0000u)};
    tt_codes(__floats2half2_rn(f[0] * inv, f[1] * inv), __floats2half2_rn(f[2] * inv, f[3] * inv), &h[j], &l[j]);
    if (amax >= 0x7F800000u) h[j] = tt_nan_codes(h[j], f[0], f[1], f[2], f[3]);
  }
  *hi = make_uint2(h[0], h[1]);
  *lo = make_uint2(l[0], l[1]);
  uint32_t sw = sb << (8 * ((lane >> 2) & 3));
  sw |= __shfl_xor_sync(0xffffffffu, sw, 4);
  sw |= __shfl_xor_sync(0xffffffffu, sw, 8);
  *word = sw;
  if constexpr (!kGuard) return false;
  // magnitudes less one, so that zeros are the largest: the smallest against the bound, and a count only where it is below
  uint32_t least = 0xFFFFFFFFu;
#pragma unroll
  for (int j = 0; j < 4; ++j) least = __viaddmin_u16x2(w[j] & kAbs, 0xFFFFFFFFu, least);
  const uint32_t below = (tt_lossy_below(amax) - 1u) >> 16;  // (a value v of 1 .. bound - 1: v - 1 < below)
  const bool finite = amax < 0x7F800000u;
  if (!__any_sync(0xffffffffu, min(least & 0xFFFFu, least >> 16) < below || !finite)) return false;
  int n = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) n += ((w[j] & 0x7FFFu) - 1u < below) + (((w[j] >> 16) & 0x7FFFu) - 1u < below);
  n += __shfl_xor_sync(0xffffffffu, n, 1);
  n += __shfl_xor_sync(0xffffffffu, n, 2);
  return __any_sync(0xffffffffu, n >= kTtLossyTokens || !finite);
}

// ---- bf16 rows of the sorted order -> two E4M3 rows and their scale factors.  Warp task: (row, `chunks` pieces of 256 values; eight -
// enough for the look-up of the row's place not to count, few enough for a short last round of the resident warps).  Bound by
// issue (2 bytes read and 2 written per element; 12288 rows of 4096: 41 us; 54 with a look-up per four pieces, 49 with
// conversion instructions, which kept their pipe 99.8 % busy). ----
// kGuard: a byte per task into `marks` (see tt_split_256), and the experts' flags start at zero.
template <bool kGuard>
__global__ void __launch_bounds__(256, 4) twoterm_split_kernel(const __nv_bfloat16* __restrict__ x, const int* __restrict__ offsets,
                                                              uint8_t* __restrict__ xq, uint8_t* __restrict__ sfx, int S, int H, int E,
                                                              int max_tok, int sf_step, uint8_t* __restrict__ marks, int* __restrict__ flags, int chunks) {
  extern __shared__ int s_tt_tables[];
  // The first launch of a public call, so the kernel in front of it may be the one that writes expert_offsets: wait before
  // they are read here, and before the gate/up grid, which reads them as it starts, may start (it waits again before it
  // reads rows).
  pdl_wait();
  pdl_launch_dependents();
  const TtTables tab = tt_tables<false>(s_tt_tables, offsets, E, max_tok);
  if (kGuard && blockIdx.x == 0)
    for (int e = threadIdx.x; e <= E; e += blockDim.x) flags[e] = 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int n_chunk = H / 256, parts = (n_chunk + chunks - 1) / chunks;
  const int p_begin = tab.off[0], n_task = (tab.off[E] - p_begin) * parts;
  const bool sf_lane = (lane & 15) < 2, sf_is_lo = (lane & 1) != 0;  // in either half warp one lane stores the hi word, one the lo word
  const uint32_t sf_less = sf_is_lo ? 0x05050505u : 0u;
  for (int task = static_cast<int>(blockIdx.x) * 8 + wid; task < n_task; task += static_cast<int>(gridDim.x) * 8) {
    const int row = parts == 1 ? task : (parts == 2 ? task >> 1 : task / parts);
    const int p = p_begin + row, c0 = (task - row * parts) * chunks, left = min(n_chunk - c0, chunks);
    // the expert: off[e] <= p < off[e + 1] (empty experts share a value with their successor)
    const int e = tt_find_expert(tab.off, E, p);
    const TtSfPlace at = tt_sf_place<false>(p, e, tab, H, sf_step);
    const uint4* src = reinterpret_cast<const uint4*>(x + static_cast<size_t>(p) * H) + c0 * 32 + lane;
    uint2* dst_hi = reinterpret_cast<uint2*>(xq + static_cast<size_t>(p) * H) + c0 * 32 + lane;
    uint2* dst_lo = dst_hi + static_cast<size_t>(S) * H / 8;
    uint8_t* sf = sfx + at.hi + (sf_is_lo ? at.lo : 0) + static_cast<size_t>(2 * c0 + (lane >> 4)) * sf_step;
    bool again = false;
#pragma unroll 1
    for (int cb = 0; cb < 8 && cb < left; cb += 4) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (cb + u < left) v[u] = __ldcg(src + u * 32);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (cb + u < left) {
          uint32_t word;
          uint2 hi, lo;
          again |= tt_split_256<kGuard>(v[u], lane, &hi, &lo, &word);
          dst_hi[u * 32] = hi;
          dst_lo[u * 32] = lo;
          if (sf_lane) *reinterpret_cast<uint32_t*>(sf) = word - sf_less;
          sf += 2 * sf_step;
        }
      src += 128;
      dst_hi += 128;
      dst_lo += 128;
    }
    if (kGuard && lane == 0) marks[static_cast<size_t>(p) * parts + (task - row * parts)] = again;
  }
}

// ---- quantised activations (moe_expert_ffn_q): bf16 rows of the sorted order -> one E2M1 row of H / 2 bytes, two scale words per K
// step of 256.  Warp task: (row, four pieces of 512 values), all their loads issued before the row's place is looked up, 16
// values a lane so that a block is two lanes.  4096 tokens of 4096, top-8, in a row of layers: 84 -> 77 us (as a form of the kernel
// above, eight values a lane); the 0.34 GB take 51 at the copy rate. ----
// The quantised-activation variant's counterpart: 16 E2M1 codes per lane (native_quant_rows_kernel's arithmetic), scale word likewise
MOE_DEVINL uint32_t max_bf16x2(uint32_t a, uint32_t b) {  // the larger of each pair, the number where the other is a NaN (as fmaxf)
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
MOE_DEVINL uint2 tt_quant_512(const uint4 (&v)[2], int lane, uint32_t* word) {
  const uint32_t w[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
  constexpr uint32_t kAbs = 0x7FFF7FFFu;
  uint32_t m2 = 0u;
#pragma unroll
  for (int j = 0; j < 8; ++j) m2 = max_bf16x2(m2, w[j] & kAbs);
  m2 = max_bf16x2(m2, __shfl_xor_sync(0xffffffffu, m2, 1));
  const uint32_t amax = max(m2 & 0xFFFFu, m2 >> 16) << 16;
  const int se = amax != 0u ? term_exp(__uint_as_float(amax)) : 0;
  const float inv = pow2f(-se);
  uint32_t codes[2] = {0u, 0u};
#pragma unroll
  for (int j = 0; j < 8; ++j)
    codes[j >> 2] |= static_cast<uint32_t>(__nv_cvt_float2_to_fp4x2(make_float2(__uint_as_float(w[j] << 16) * inv, __uint_as_float(w[j] & 0xFFFF0000u) * inv),
                                                                    __NV_E2M1, cudaRoundNearest)) << (8 * (j & 3));
  uint32_t sw = static_cast<uint32_t>(se + 127) << (8 * ((lane >> 1) & 3));
  sw |= __shfl_xor_sync(0xffffffffu, sw, 2);
  sw |= __shfl_xor_sync(0xffffffffu, sw, 4);
  *word = sw;
  return make_uint2(codes[0], codes[1]);
}

__global__ void __launch_bounds__(256, 4) twoterm_quant_kernel(const __nv_bfloat16* __restrict__ x, const int* __restrict__ offsets,
                                                              uint8_t* __restrict__ xq, uint8_t* __restrict__ sfx, int H, int E, int max_tok,
                                                              int sf_step) {
  extern __shared__ int s_tt_tables[];
  pdl_wait();  // (as twoterm_split_kernel)
  pdl_launch_dependents();
  const TtTables tab = tt_tables<true>(s_tt_tables, offsets, E, max_tok);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int parts = (H + 2047) / 2048;
  const int p_begin = tab.off[0], n_task = (tab.off[E] - p_begin) * parts;
  for (int task = static_cast<int>(blockIdx.x) * 8 + wid; task < n_task; task += static_cast<int>(gridDim.x) * 8) {
    const int row = parts == 1 ? task : (parts == 2 ? task >> 1 : task / parts);
    const int p = p_begin + row, c0 = (task - row * parts) * 4;
    const int left = H - c0 * 512 - lane * 16;  // values of the row from this lane's first on (a multiple of 16)
    const uint4* src = reinterpret_cast<const uint4*>(x + static_cast<size_t>(p) * H) + c0 * 64 + lane * 2;
    uint4 v[4][2];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int i = 0; i < 2; ++i) v[u][i] = left > u * 512 ? __ldcg(src + u * 64 + i) : make_uint4(0u, 0u, 0u, 0u);
    // the expert: off[e] <= p < off[e + 1] (empty experts share a value with their successor)
    const TtSfPlace at = tt_sf_place<true>(p, tt_find_expert(tab.off, E, p), tab, H, sf_step);
    uint2* dst = reinterpret_cast<uint2*>(xq + static_cast<size_t>(p) * (H / 2)) + c0 * 32 + lane;
    uint8_t* sf = sfx + at.hi + ((lane >> 3) & 1) * at.lo + static_cast<size_t>(2 * c0 + (lane >> 4)) * sf_step;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      uint32_t word;
      const uint2 codes = tt_quant_512(v[u], lane, &word);
      if (left > u * 512) {  // (of a last half piece, half of the lanes: words in whole eights)
        dst[u * 32] = codes;
        if ((lane & 7) == 0) *reinterpret_cast<uint32_t*>(sf + static_cast<size_t>(2 * u) * sf_step) = word;
      }
    }
  }
}

// ---- the same from the unsorted rows, where a call holds the routing (moe_forward, moe_ffn_block): a token's row is split
// once and stored at its k sorted places, so the bf16 copy in sorted order is neither written nor read and a value is
// converted once, not k times.  Warp task: (token, `chunks` pieces of 256 values).  It writes k * H * 2 bytes per token and is
// bound by issuing them, 8 bytes a lane with the row and scale places shuffled out per slot: 8192 tokens of 4096, top-8,
// 166 us for 0.61 GB, 0.56 of the copy rate.  (A warp's part collected in shared memory and sent with one bulk copy per slot and
// term: 181 us.)
// It writes at 3.9 TB/s, which is what torch's fill_ writes at - the only kernel of stores alone that was timed beside it; a copy
// reaches 6.5 with the half that it reads.
// kRows: into `rows` the bf16 rows in sorted order as well, for a caller whose buffer they are (moe_layer): 11 us less than the
// copy and a split from it (8216 slots of 4096: the layer 238 -> 227 us; 12288 slots 1123 -> 1108).  (Asked at run time, slot by
// slot, it took the form without it from 40 to 48 registers and made that of moe_forward's prompts spill: 8192 tokens 160 us
// and 158, 32768 skewed 610 and 604.) ----
template <bool kGuard, bool kRows>
__global__ void __launch_bounds__(256) twoterm_scatter_kernel(const __nv_bfloat16* __restrict__ x, const int* __restrict__ ids,
                                                             const int* __restrict__ inv_perm, const int* __restrict__ offsets,
                                                             uint8_t* __restrict__ xq, uint8_t* __restrict__ sfx, int T, int k, int H,
                                                             int E, int max_tok, int sf_step, int chunks, uint8_t* __restrict__ marks,
                                                             int* __restrict__ flags, int offsets_late, __nv_bfloat16* __restrict__ rows) {
  extern __shared__ int s_tt_tables[];
  // expert_offsets is read here and, as it starts, by the gate/up grid: complete where the sort of the same call waited for
  // the router before it let this kernel start, to be waited for where one kernel routes and sorts
  if (offsets_late) pdl_wait();
  pdl_launch_dependents();
  const TtTables tab = tt_tables<false>(s_tt_tables, offsets, E, max_tok);
  pdl_wait();
  if (kGuard && blockIdx.x == 0)
    for (int e = threadIdx.x; e <= E; e += blockDim.x) flags[e] = 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const size_t S = static_cast<size_t>(T) * k;
  const int n_chunk = H / 256, parts = (n_chunk + chunks - 1) / chunks;
  const int n_task = T * parts;
  for (int task = static_cast<int>(blockIdx.x) * 8 + wid; task < n_task; task += static_cast<int>(gridDim.x) * 8) {
    const int t = task / parts, c0 = (task % parts) * chunks, c1 = min(c0 + chunks, n_chunk);
    int p = 0, sf_lo = 0;
    size_t sf_hi = 0;
    if (lane < k) {  // lane j looks up slot j
      p = __ldg(inv_perm + static_cast<size_t>(t) * k + lane);
      const TtSfPlace at = tt_sf_place<false>(p, __ldg(ids + static_cast<size_t>(t) * k + lane), tab, H, sf_step);
      sf_hi = at.hi;
      sf_lo = at.lo;
    }
    __syncwarp();
    const uint4* src = reinterpret_cast<const uint4*>(x + static_cast<size_t>(t) * H);
    bool again = false;
#pragma unroll 2
    for (int c = c0; c < c1; ++c) {
      uint2 hi, lo;
      uint32_t word;
      const uint4 v = __ldg(src + c * 32 + lane);
      again |= tt_split_256<kGuard>(v, lane, &hi, &lo, &word);
      const size_t step = static_cast<size_t>(2 * c + (lane >> 4)) * sf_step;
      for (int j = 0; j < k; ++j) {
        const size_t row = static_cast<size_t>(__shfl_sync(0xffffffffu, p, j));
        reinterpret_cast<uint2*>(xq + row * H)[c * 32 + lane] = hi;
        reinterpret_cast<uint2*>(xq + (S + row) * H)[c * 32 + lane] = lo;
        if (kRows) reinterpret_cast<uint4*>(rows + row * H)[c * 32 + lane] = v;
        const size_t at = __shfl_sync(0xffffffffu, static_cast<unsigned long long>(sf_hi), j);
        const int d = __shfl_sync(0xffffffffu, sf_lo, j);
        if ((lane & 15) == 0) *reinterpret_cast<uint32_t*>(sfx + at + step) = word;
        if ((lane & 15) == 1) *reinterpret_cast<uint32_t*>(sfx + at + step + d) = word - 0x05050505u;
      }
    }
    if (kGuard && lane < k) marks[static_cast<size_t>(p) * parts + task % parts] = again;
  }
}

// Rows in sorted order of the experts that are done again, where the split above left them where they were
__global__ void __launch_bounds__(256) twoterm_gather_kernel(const __nv_bfloat16* __restrict__ x, const int* __restrict__ ids,
                                                            const int* __restrict__ inv_perm, const int* only, int T, int k, int H,
                                                            int E, __nv_bfloat16* __restrict__ x_sorted) {
  pdl_wait();
  if (__ldcg(only + E) == 0) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (size_t s = static_cast<size_t>(blockIdx.x) * 8 + wid; s < static_cast<size_t>(T) * k; s += static_cast<size_t>(gridDim.x) * 8) {
    if (__ldcg(only + __ldg(ids + s)) == 0) continue;
    const uint4* src = reinterpret_cast<const uint4*>(x + s / k * H);
    uint4* dst = reinterpret_cast<uint4*>(x_sorted + static_cast<size_t>(__ldg(inv_perm + s)) * H);
    for (int i = lane; i < H / 8; i += 32) dst[i] = __ldg(src + i);
  }
}

// kM: M tiles per item (gate/up: always 2)
// kQ: quantised activations (moe_expert_ffn_q), one E2M1 term per value: dense 4-bit operands (kind::mxf4, K = 64), K steps of
// 256, two scale words per row and step; every pass is of the separate form with one operand
// kGuard (gate/up): blocks that the terms hold too little of are looked for
template <bool STAGE1, int kM, bool kQ, bool kGuard, bool kFifo>
__global__ void __launch_bounds__(kTtThreads, 1)
ffn_twoterm_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_sc,
                   const __grid_constant__ TtTokMaps tmap_t, const TtArgs a) {
  static_assert(!STAGE1 || kM == 2, "gate and up");
  static_assert(!kGuard || (STAGE1 && !kQ), "gate/up on two terms");
  static_assert(!kFifo || !kQ, "stacked passes");
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  const TtSmem sm = tt_smem(a.E, kM, a.stages, a.t_bytes);
  unsigned char* sSf = smem + sm.sf;
  const uint32_t ring = smem_u32(smem + sm.ring);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + sm.bars);
  // What the MMAs wait for is counted in the first CTA: its own loads and the second CTA's, scale bytes of both
  uint64_t* full = bars;                         // [kTtMaxStages] both producers' TMA -> MMA
  uint64_t* empty = full + kTtMaxStages;         // MMA done -> producers, in both CTAs
  uint64_t* full_sf = empty + kTtMaxStages;      // [kTtSfSlots] scale bytes in order -> MMA
  uint64_t* empty_sf = full_sf + kTtSfSlots;
  uint64_t* raw_sf = empty_sf + kTtSfSlots;      // scale bytes as they lie in memory -> scale warp
  uint64_t* acc_full = raw_sf + kTtSfSlots;      // [2] MMA -> epilogue, in both CTAs
  uint64_t* acc_empty = acc_full + 2;            // [2] both CTAs' epilogues -> MMA
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + sm.misc);
  int* prefix = reinterpret_cast<int*>(smem + sm.prefix);
  int* s_off = prefix + a.E + 2;

  const int tid = threadIdx.x, lane = tid & 31, wid = warp_uniform(tid >> 5);
  const int rank = warp_uniform(static_cast<int>(tt_ctarank()));
  constexpr int step_k = kQ ? 256 : 128;
  const int K = a.K, n_steps = K / step_k;
  const int tiles = STAGE1 ? a.I / 256 : a.R / (256 * kM);
  // scale bytes of 128 rows per M tile and group: 16 bytes a row (K = 512) by TMA; 8 bytes (256) in one contiguous
  // piece where that is all a row has; 8 bytes by plain loads where a row's bytes are no multiple of 16
  const bool sf_tma = (K % 512) == 0, sf_bulk = K == 256;
  const int grp_steps = (sf_tma ? 512 : 256) / step_k;

  // ---- setup ----  (expert_offsets was complete before the split kernel let this chain start)
  if (wid == 2) tt_prefix(a.offsets, a.E, a.max_tok, prefix, lane);
  if (wid >= kTtFirstEpi)
    for (int e = tid - kTtFirstEpi * 32; e <= a.E; e += kTtEpiWarps * 32) s_off[e] = __ldg(a.offsets + e);
  if (tid == 0) {
    for (int s = 0; s < kTtMaxStages; ++s) {
      mbar_init(&full[s], 2);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < kTtSfSlots; ++s) {
      mbar_init(&full_sf[s], 2);
      mbar_init(&empty_sf[s], 1);
      mbar_init(&raw_sf[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], 2 * kTtEpiWarps);
    }
    mbar_fence_init();
  }
  if (wid == 1) tt_tmem_alloc(tmem_holder, kTtTmemCols);
  tc_fence_before_sync();
  __syncthreads();
  tt_cluster_sync();
  tc_fence_after_sync();
  // (see warp_uniform)
  const uint32_t tmem_base = static_cast<uint32_t>(warp_uniform(static_cast<int>(*tmem_holder)));
  // Items go round-robin to the CTA pairs in blocks of consecutive tiles of one pass: of one tile, so that the pairs work on
  // few passes at a time whose token rows stay in L2; of four where an item is a few K steps long, so that what an item costs
  // beside them (looking up its pass) is paid once per block.
  const int tb = n_steps <= 4 && (tiles & 3) == 0 ? 4 : 1, tb_shift = tb == 4 ? 2 : 0;
  const int total = warp_uniform(prefix[a.E]) * tiles;
  const int pair = static_cast<int>(blockIdx.x) >> 1, pairs = static_cast<int>(gridDim.x) >> 1;
  const int first = pair << tb_shift;
  auto next_item = [&](int w) { return (w & (tb - 1)) != tb - 1 ? w + 1 : w + 1 + ((pairs - 1) << tb_shift); };
  pdl_launch_dependents();  // the next kernel waits for this grid before it reads what it writes

  // first weight row of this CTA in M tile t of an item
  auto weight_row = [&](int e, int rt, int t) {
    return STAGE1 ? e * a.R + t * a.I + rt * 256 + rank * 128 : e * a.R + (rt * kM + t) * 256 + rank * 128;
  };

  auto uniform_pass = [&](int g) {
    const int e = tt_find_expert(prefix, a.E, g);
    TtPass p = tt_pass<kQ>(s_off[e], s_off[e + 1], g - prefix[e], a.max_tok);
    p.row0 = warp_uniform(p.row0);
    p.n = warp_uniform(p.n);
    p.nr = warp_uniform(p.nr);
    p.N = warp_uniform(p.N);
    p.stacked = warp_uniform(static_cast<int>(p.stacked)) != 0;
    return p;
  };

  if (wid == 0) {
    // =========================== weights (all lanes; the instructions are issued by an elected one) ===========================
    int fs = 0, kb = 0;
    uint32_t fph = 0;
    TtRing<kFifo> r(sm.stage, a.stages);
    const uint32_t sf_base = smem_u32(sSf), raw_bar = smem_u32(raw_sf), full_own = smem_u32(full), full_first = tt_first_addr(full);
    const uint64_t pol_once = l2_policy_evict_first(), pol_again = l2_policy_evict_normal();
    int g_known = -1, e = 0;
    bool once = true;
    for (int w = first; w < total; w = next_item(w)) {
      const int g = w / tiles, rt = w % tiles;
      if (g != g_known) {
        e = warp_uniform(tt_find_expert(prefix, a.E, g));
        once = warp_uniform(prefix[e + 1] - prefix[e]) == 1;  // an expert of one pass is read once per call
        if (kFifo) kb = warp_uniform(tt_fifo_kb(tt_pass<kQ>(s_off[e], s_off[e + 1], g - prefix[e], a.max_tok), kM));
        g_known = g;
      }
      const uint64_t pol = once ? pol_once : pol_again;
      for (int ks = 0; ks < n_steps; ++ks) {
        if ((sf_tma || sf_bulk) && (ks & (grp_steps - 1)) == 0) {
          mbar_wait_warp(&empty_sf[fs], fph ^ 1u, a.status);
          tt_expect_tx(raw_bar + fs * 8, static_cast<uint32_t>(kM * 128 * (sf_tma ? 16 : 8)));
#pragma unroll
          for (int t = 0; t < kM; ++t) {
            const int row = weight_row(e, rt, t);
            const uint32_t dst = sf_base + (fs * kM + t) * 2048;
            if (sf_tma && a.blocked)  // 128 rows in one piece
              bulk_g2s_hint_elect(dst, a.sc + static_cast<size_t>((row >> 7) * (K / 512) + ks * step_k / 512) * 2048, 2048u, raw_bar + fs * 8, pol);
            else if (sf_tma)
              tt_load_2d_hint(dst, &tmap_sc, ks * (step_k / 32), row, raw_bar + fs * 8, pol);
            else
              tt_bulk_g2s(dst, a.sc + static_cast<size_t>(row) * 8, 1024u, raw_bar + fs * 8);
          }
          if (++fs == kTtSfSlots) { fs = 0; fph ^= 1u; }
        }
        r.take(kb, empty, a.status);
        if (rank == 0) tt_expect_tx(full_own + r.bar * 8, 2 * kM * (kQ ? kTtTile : kTtTile / 2));  // both CTAs' (transactions count the packed bytes)
#pragma unroll
        for (int t = 0; t < kM; ++t) {
          // 128 rows x 128 codes; tile-contiguous layout: half of the rows of tile (row / 128, ks / 2)
          const int row = weight_row(e, rt, t);
          if constexpr (kQ)  // packed rows as they are: 128 rows x 128 bytes
            tt_load_2d_hint(ring + r.addr + t * kTtTile, &tmap_w, a.blocked ? 0 : ks * 128,
                            a.blocked ? ((row >> 7) * n_steps + ks) * 128 : row, full_first + r.bar * 8, pol);
          else
            tt_load_2d_hint(ring + r.addr + t * kTtTile, &tmap_w, a.blocked ? (ks & 1) * kTtK : ks * kTtK,
                            a.blocked ? ((row >> 7) * (n_steps >> 1) + (ks >> 1)) * 128 : row, full_first + r.bar * 8, pol);
        }
      }
    }
  } else if (wid == 2) {
    // =========================== tokens (likewise) ===========================
    // The rows and scale factors are complete.  (A CTA without items leaves at once: kernels further down the stream may be waiting
    // for its SM to start beside this one, see moe_ffn_block.  Where no CTA has any - an expert-parallel rank without rows -
    // one pair waits all the same: each kernel of a stream waits for the one in front only, which must therefore not
    // end before those in front of it.)
    if (first < total || (total == 0 && pair == 0)) pdl_wait();
    TtRing<kFifo> r(sm.stage, a.stages);
    const uint32_t full_own = smem_u32(full), full_first = tt_first_addr(full);
    const int sf_pitch = a.sf_step >> 7;  // scale factors as rows of 128 bytes: a box is one 512-byte chunk
    int g_known = -1;
    TtPass p = {};
    for (int w = first; w < total; w = next_item(w)) {
      const int g = w / tiles;
      if (g != g_known) p = uniform_pass(g);
      g_known = g;
      const int chunks = p.N <= 128 ? 1 : 2;
      const int rows = p.N >> 1;  // this CTA's half of the operand
      const int row_hi = p.stacked ? p.row0 + rank * a.S : p.row0 + rank * rows;
      const int kb = kFifo ? tt_fifo_kb(p, kM) : 0, sf_off = kFifo ? p.nr * 128 : a.sf_off;
      for (int ks = 0; ks < n_steps; ++ks) {
        const int terms = kQ || p.stacked ? 1 : 2;  // operands of this CTA: one term of a stacked pass, hi and lo of a separate one
        const int words = kQ ? 2 : terms;          // sets of scale factor chunks
        r.take(kb, empty, a.status);
        const uint32_t part = ring + r.addr + kM * kTtTile, bar = full_first + r.bar * 8;
        if (rank == 0) tt_expect_tx(full_own + r.bar * 8, static_cast<uint32_t>(2 * (terms * rows * 128 + words * chunks * 512)));
        for (int t = 0; t < words; ++t)
          for (int c = 0; c < chunks; ++c)
            tt_load_2d(part + sf_off + t * 1024 + c * 512, &tmap_t.sf, 0, (g * n_steps + ks) * sf_pitch + t * 8 + c * 4, bar);
        for (int t = 0; t < terms; ++t) {
          uint32_t dst = part + t * (rows * 128);
          int row = row_hi + t * a.S;
          if (rows & 64) {
            tt_load_2d(dst, &tmap_t.box[0], ks * 128, row, bar);
            row += 64;
            dst += 64 * 128;
          }
          if (rows & 32) {
            tt_load_2d(dst, &tmap_t.box[1], ks * 128, row, bar);
            row += 32;
            dst += 32 * 128;
          }
          if (rows & 16) tt_load_2d(dst, &tmap_t.box[2], ks * 128, row, bar);
        }
      }
    }
  } else if (wid == 1) {
    int fs = 0, tog = 0;
    uint32_t fph = 0, acc_ph[2] = {0u, 0u};
    int g_known = -1;
    TtPass p = {};
    TtRing<kFifo> r(sm.stage, a.stages);
    if (rank == 0) {
      // =========================== first CTA: MMA issuer, all lanes ===========================
      for (int w = first; w < total; w = next_item(w)) {
        const int g = w / tiles;
        if (g != g_known) p = uniform_pass(g);
        g_known = g;
        const bool small = kM == 1 || p.N <= static_cast<int>(kTtHalf);
        const uint32_t idesc = kQ ? tt_idesc_mxf4(p.N) : tt_idesc(p.N);
        const int half = small ? tog : 0;
        mbar_wait_warp(&acc_empty[half], acc_ph[half] ^ 1u, a.status);
        if (!small) mbar_wait_warp(&acc_empty[1], acc_ph[1] ^ 1u, a.status);
        const uint32_t d0 = tmem_base + static_cast<uint32_t>(half) * kTtFull;
        const uint32_t d1 = d0 + (small ? kTtHalf : kTtFull);
        tc_fence_after_sync();
        const int kb = kFifo ? tt_fifo_kb(p, kM) : 0, sf_off = kFifo ? p.nr * 128 : a.sf_off;
        for (int ks = 0; ks < n_steps; ++ks) {
          const uint32_t sf_col = tmem_base + kTtColSf + static_cast<uint32_t>(ks & 1) * (kQ ? kTtSfSetQ : kTtSfSet);
          const int si = ks & (grp_steps - 1);
          if (si == 0) mbar_wait_warp(&full_sf[fs], fph, a.status);
          r.next(kb);
          mbar_wait_warp(&full[r.bar], r.parity, a.status);
          tc_fence_after_sync();
          const uint32_t w_addr = ring + r.addr, t_addr = w_addr + kM * kTtTile;
          const uint32_t sfw = smem_u32(sSf) + static_cast<uint32_t>((fs * 4 + si * (kQ ? 2 : 1)) * kM) * 512, sft = t_addr + sf_off;
          if constexpr (kQ) {
#pragma unroll
            for (uint32_t w = 0; w < 2; ++w) {  // scale words of the step
              tt_cp_sf(sf_col + w * 4, sfw + w * (kM * 512));
              if (kM == 2) tt_cp_sf(sf_col + 8 + w * 4, sfw + w * (kM * 512) + 512);
              tt_cp_sf(sf_col + 16 + w * 8, sft + w * 1024);
              if (p.N > 128) tt_cp_sf(sf_col + 20 + w * 8, sft + w * 1024 + 512);
            }
            tt_mma_step_mxf4<kM>(d0, d1, umma_desc_k_sw128(w_addr), umma_desc_k_sw128(w_addr + kTtTile), umma_desc_k_sw128(t_addr),
                                 idesc, sf_col, sf_col + 8, sf_col + 16, ks != 0 ? 1u : 0u);
          } else {
            tt_cp_sf(sf_col, sfw);
            if (kM == 2) tt_cp_sf(sf_col + 4, sfw + 512);
            tt_cp_sf(sf_col + 8, sft);
            if (p.N > 128) tt_cp_sf(sf_col + 12, sft + 512);
            tt_mma_step<kM>(d0, d1, umma_desc_k_sw128(w_addr), umma_desc_k_sw128(w_addr + kTtTile), umma_desc_k_sw128(t_addr), idesc,
                            sf_col, sf_col + 4, sf_col + 8, ks != 0 ? 1u : 0u);
            if (!p.stacked) {  // the lo terms, into the same columns
              tt_cp_sf(sf_col + 16, sft + 1024);
              if (p.N > 128) tt_cp_sf(sf_col + 20, sft + 1536);
              tt_mma_step<kM>(d0, d1, umma_desc_k_sw128(w_addr), umma_desc_k_sw128(w_addr + kTtTile),
                              umma_desc_k_sw128(t_addr + (p.N >> 1) * 128), idesc, sf_col, sf_col + 4, sf_col + 16, 1u);
            }
          }
          tt_commit(&empty[r.bar]);
          if (si == grp_steps - 1) {
            tt_commit(&empty_sf[fs]);
            if (++fs == kTtSfSlots) { fs = 0; fph ^= 1u; }
          }
        }
        tt_commit(&acc_full[half]);
        acc_ph[half] ^= 1u;
        if (!small) {
          tt_commit(&acc_full[1]);
          acc_ph[1] ^= 1u;
          tog = 0;
        } else {
          tog ^= 1;
        }
      }
    }
  } else if (wid == 3) {
    // =========================== weight scale bytes -> tensor-memory order ===========================
    // Per M tile and K step a chunk of [32 lanes][4 words]: lane l, word c = the four scale bytes of row 32c + l.  A slot's
    // bytes are read whole before the chunks are written over them.  (No load from global memory is in flight across the
    // proxy fence: with prefetched plain loads the fence waited for them, 1100 cycles per group.)
    int fs = 0;
    uint32_t fph = 0;
    for (int w = first; w < total; w = next_item(w)) {
      const int g = w / tiles, rt = w % tiles;
      const int e = tt_find_expert(prefix, a.E, g);
      for (int ks = 0; ks < n_steps; ks += grp_steps) {
        unsigned char* slot = sSf + fs * kM * 2048;
        uint4 r[kM][4];
        if (sf_tma || sf_bulk) {
          mbar_wait(&raw_sf[fs], fph, a.status);
          __syncwarp();
#pragma unroll
          for (int t = 0; t < kM; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              if (sf_tma) {
                r[t][c] = *reinterpret_cast<const uint4*>(slot + t * 2048 + (32 * c + lane) * 16);
              } else {
                const uint2 v = *reinterpret_cast<const uint2*>(slot + t * 2048 + (32 * c + lane) * 8);
                r[t][c] = make_uint4(v.x, v.y, 0u, 0u);
              }
            }
          __syncwarp();
        } else {
#pragma unroll
          for (int t = 0; t < kM; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint2 v = __ldg(reinterpret_cast<const uint2*>(a.sc + static_cast<size_t>(weight_row(e, rt, t) + 32 * c + lane) * (K / 32) + ks * (step_k / 32)));
              r[t][c] = make_uint4(v.x, v.y, 0u, 0u);
            }
          mbar_wait(&empty_sf[fs], fph ^ 1u, a.status);
          __syncwarp();
        }
#pragma unroll
        for (int t = 0; t < kM; ++t) {
          uint4* dst = reinterpret_cast<uint4*>(slot + t * 512) + lane;
          constexpr int step = kM * 32;
          dst[0] = make_uint4(r[t][0].x, r[t][1].x, r[t][2].x, r[t][3].x);
          dst[step] = make_uint4(r[t][0].y, r[t][1].y, r[t][2].y, r[t][3].y);
          if (sf_tma) {
            dst[2 * step] = make_uint4(r[t][0].z, r[t][1].z, r[t][2].z, r[t][3].z);
            dst[3 * step] = make_uint4(r[t][0].w, r[t][1].w, r[t][2].w, r[t][3].w);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) tt_arrive_first(&full_sf[fs]);
        if (++fs == kTtSfSlots) { fs = 0; fph ^= 1u; }
      }
    }
  } else {
    // =========================== epilogue ===========================
    const int q = wid & 3, sub = (wid - kTtFirstEpi) >> 2;
    const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
    int tog = 0, g_known = -1;
    TtPass p = {};
    uint32_t acc_ph[2] = {0u, 0u};
    if constexpr (kGuard) {
      // the split kernel's marks -> flags of their experts, 16 at a time, while the first MMAs run
      pdl_wait();  // the marks are complete and the flags zero
      const size_t n_marks = (static_cast<size_t>(a.S) * a.parts + 15) / 16;
      for (size_t i = static_cast<size_t>(blockIdx.x) * (kTtEpiWarps * 32) + (tid - kTtFirstEpi * 32); i < n_marks;
           i += static_cast<size_t>(gridDim.x) * (kTtEpiWarps * 32)) {
        const uint4 v = __ldcg(a.marks + i);
        if ((v.x | v.y | v.z | v.w) == 0u) continue;
        const uint32_t m[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int b = 0; b < 16; ++b) {
          if (((m[b >> 2] >> (8 * (b & 3))) & 0xFFu) == 0u) continue;
          const int row = static_cast<int>((i * 16 + b) / a.parts);
          if (row < s_off[0] || row >= s_off[a.E]) continue;  // (rows of other ranks' experts: their marks are not written)
          a.flags[tt_find_expert(s_off, a.E, row)] = 1;
          a.flags[a.E] = 1;
        }
      }
      __syncwarp();
    }
    int e = 0;
    for (int w = first; w < total; w = next_item(w)) {
      const int g = w / tiles, rt = w % tiles;
      if (g != g_known) {
        e = tt_find_expert(prefix, a.E, g);
        p = tt_pass<kQ>(s_off[e], s_off[e + 1], g - prefix[e], a.max_tok);
        g_known = g;
      }
      const bool small = kM == 1 || p.N <= static_cast<int>(kTtHalf);
      const int half = small ? tog : 0;
      mbar_wait(&acc_full[half], acc_ph[half], a.status);
      acc_ph[half] ^= 1u;
      if (!small) {
        mbar_wait(&acc_full[1], acc_ph[1], a.status);
        acc_ph[1] ^= 1u;
        tog = 0;
      } else {
        tog ^= 1;
      }
      __syncwarp();  // tcgen05.ld is warp-collective
      tc_fence_after_sync();
      const uint32_t d0 = tmem_base + lane_base + static_cast<uint32_t>(half) * kTtFull;
      const uint32_t d1 = d0 + (small ? kTtHalf : kTtFull);
      auto release = [&]() {
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) {
          if (rank == 0) {
            mbar_arrive(&acc_empty[half]);
            if (!small) mbar_arrive(&acc_empty[1]);
          } else {
            tt_arrive_first(&acc_empty[half]);
            if (!small) tt_arrive_first(&acc_empty[1]);
          }
        }
      };
      if constexpr (STAGE1) {
        // lane = i inside the tile, columns = tokens, gate in the first accumulator and up in the second.  First SwiGLU and
        // the rounding to bf16 of this warp's columns (8 in turn with the other three warps of the quadrant), two values
        // per register, so that the accumulators are free again early.
        constexpr int kChunks = 7;
        uint32_t pk[kChunks][4];
#pragma unroll
        for (int ch = 0; ch < kChunks; ++ch) {
          const int c0 = ch * 32 + sub * 8;
          if (c0 < p.n) {
            uint32_t gv[8], uv[8];
            tt_tmem_ld_32x8(d0 + static_cast<uint32_t>(c0), gv);
            tt_tmem_ld_32x8(d1 + static_cast<uint32_t>(c0), uv);
            if (p.stacked) {
              uint32_t gl[8], ul[8];
              tt_tmem_ld_32x8(d0 + static_cast<uint32_t>(p.nr + c0), gl);
              tt_tmem_ld_32x8(d1 + static_cast<uint32_t>(p.nr + c0), ul);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                gv[j] = __float_as_uint(__uint_as_float(gv[j]) + __uint_as_float(gl[j]));
                uv[j] = __float_as_uint(__uint_as_float(uv[j]) + __uint_as_float(ul[j]));
              }
            } else {
              tmem_ld_wait();
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const __nv_bfloat162 h = __floats2bfloat162_rn(tt_silu_mul(__uint_as_float(gv[2 * j]), __uint_as_float(uv[2 * j])),
                                                             tt_silu_mul(__uint_as_float(gv[2 * j + 1]), __uint_as_float(uv[2 * j + 1])));
              pk[ch][j] = *reinterpret_cast<const uint32_t*>(&h);
            }
          }
        }
        release();
        if constexpr (kQ) {
          // One E2M1 term: the warp's 32 lanes are one scale block.  A lane's codes of eight tokens are the nibbles of a word;
          // transposed over eight lanes, a lane holds four bytes - eight consecutive values - of one token.
          uint8_t* sf = a.sfa + (static_cast<size_t>(g) * (a.I / 256) + rt) * a.sf_step + rank * 1024;
#pragma unroll
          for (int ch = 0; ch < kChunks; ++ch) {
            const int c0 = ch * 32 + sub * 8;
            if (c0 < p.n) {
              uint32_t codes = 0u, my_se = 0u;
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                float y[2];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                  const uint32_t vb = t ? pk[ch][j] & 0xFFFF0000u : pk[ch][j] << 16;
                  // (finite by this variant's domain: the integer maximum is the maximum of the magnitudes)
                  const uint32_t amax = __reduce_max_sync(0xffffffffu, vb & 0x7FFFFFFFu);
                  const int se = amax > 0u ? term_exp(__uint_as_float(amax)) : 0;
                  y[t] = __uint_as_float(vb) * pow2f(-se);
                  if (lane == 2 * j + t) my_se = static_cast<uint32_t>(se + 127);
                }
                codes |= static_cast<uint32_t>(__nv_cvt_float2_to_fp4x2(make_float2(y[0], y[1]), __NV_E2M1, cudaRoundNearest)) << (8 * j);
              }
              codes = transpose_8x8_nibbles(codes, lane);
              const int tok = c0 + (lane & 7);
              if (tok < p.n)
                *reinterpret_cast<uint32_t*>(a.aq + static_cast<size_t>(p.row0 + tok) * (a.I / 2) + (rt * 256 + rank * 128 + q * 32) / 2 +
                                             4 * (lane >> 3)) = codes;
              if (lane < 8 && c0 + lane < p.n) sf[tt_sf_byte(c0 + lane, q)] = static_cast<uint8_t>(my_se);
            }
          }
        } else {
          // Then the two terms: the warp's 32 lanes are one scale block; the bytes of four tokens are transposed over four
          // lanes so that a store writes four rows of the block at a time.
          const int kstep = rt * 2 + rank;
          const int i0 = kstep * 128 + q * 32 + 4 * (lane >> 2);
          uint8_t* sf = a.sfa + (static_cast<size_t>(g) * (a.I / kTtK) + kstep) * a.sf_step;
          bool again = false;  // (kGuard) a block of this item that the terms hold too little of
  #pragma unroll
          for (int ch = 0; ch < kChunks; ++ch) {
            const int c0 = ch * 32 + sub * 8;
            if (c0 < p.n) {
              uint32_t my_sb = 0u;
              int lossy = 0;           // most inexact values in one of the eight blocks
              bool not_finite = false;
  #pragma unroll
              for (int jj = 0; jj < 8; jj += 4) {
                float v[4], inv[4];
                bool bad = false;
  #pragma unroll
                for (int t = 0; t < 4; ++t) {
                  const uint32_t pw = pk[ch][(jj + t) >> 1];
                  const uint32_t vb = (t & 1) ? pw & 0xFFFF0000u : pw << 16;
                  const uint32_t amax = __reduce_max_sync(0xffffffffu, vb & 0x7FFFFFFFu);
                  const uint32_t sb = tt_scale(amax);
                  v[t] = __uint_as_float(vb);
                  inv[t] = tt_inv(sb);
                  bad |= amax >= 0x7F800000u;
                  if (kGuard) lossy = max(lossy, __popc(__ballot_sync(0xffffffffu, (vb & 0x7FFFFFFFu) - 1u < tt_lossy_below(amax) - 1u)));
                  if (lane == jj + t) my_sb = sb;
                }
                uint32_t hw, lw, h1, l1;
                tt_codes_cvt(__floats2half2_rn(v[0] * inv[0], v[1] * inv[1]), &hw, &lw);
                tt_codes_cvt(__floats2half2_rn(v[2] * inv[2], v[3] * inv[3]), &h1, &l1);
                hw |= h1 << 16;
                lw |= l1 << 16;
                if (bad) hw = tt_nan_codes(hw, v[0], v[1], v[2], v[3]);
                not_finite |= bad;
                hw = transpose_4x4(hw, lane);
                lw = transpose_4x4(lw, lane);
                const int tok = c0 + jj + (lane & 3);
                if (tok < p.n) {
                  uint8_t* dst = a.aq + static_cast<size_t>(p.row0 + tok) * a.I + i0;
                  *reinterpret_cast<uint32_t*>(dst) = hw;
                  *reinterpret_cast<uint32_t*>(dst + static_cast<size_t>(a.S) * a.I) = lw;
                }
              }
              if (lane < 8 && c0 + lane < p.n) {
                const int r = c0 + lane;
                sf[tt_sf_byte(r, q)] = static_cast<uint8_t>(my_sb);
                sf[p.stacked ? tt_sf_byte(p.nr + r, q) : 1024 + tt_sf_byte(r, q)] = static_cast<uint8_t>(my_sb - 5u);
              }
              if (kGuard && (lossy >= kTtLossyInter || not_finite)) again |= tt_again(pk[ch], p.n - c0);
            }
          }
          if (kGuard && again && lane == 0) {
            a.flags[e] = 1;
            a.flags[a.E] = 1;
          }
        }
      } else {
#pragma unroll 1
        for (int t = 0; t < kM; ++t) {
          const uint32_t d = t == 0 ? d0 : d1;
          const int n = (rt * kM + t) * 256 + rank * 128 + q * 32 + lane;
#pragma unroll 1
          for (int c0 = sub * 16; c0 < p.n; c0 += 64) {
            uint32_t v[16];
            tmem_ld_32x16(d + static_cast<uint32_t>(c0), v);
            if (p.stacked) {
              uint32_t l[16];
              tmem_ld_32x16(d + static_cast<uint32_t>(p.nr + c0), l);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(l[j]));
            } else {
              tmem_ld_wait();
            }
            if (a.row_dst == nullptr) {
              float* dst = a.y + static_cast<size_t>(p.row0 + c0) * a.R + n;
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                if (c0 + j < p.n) *dst = __uint_as_float(v[j]);
                dst += a.R;
              }
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (c0 + j < p.n) y_row(a.y, a.row_dst, static_cast<size_t>(p.row0 + c0 + j), a.R)[n] = __uint_as_float(v[j]);
            }
          }
        }
        release();
      }
    }
  }

  // ---- teardown: neither CTA leaves while the other's MMAs may read its shared memory or arrive on its barriers ----
  tc_fence_before_sync();
  __syncthreads();
  if (tid == 0 && a.finished != nullptr) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.finished) : "memory");
  tt_cluster_sync();
  if (wid == 1) {
    tc_fence_after_sync();
    tt_tmem_dealloc(tmem_base, kTtTmemCols);
  }
}

// ---- host side ---------------------------------------------------------------------------------------
bool twoterm_weights_ok(const void* w13, const void* w2) {  // the 4-bit tensor map wants 32-byte aligned addresses
  return ((reinterpret_cast<uintptr_t>(w13) | reinterpret_cast<uintptr_t>(w2)) & 31u) == 0;
}

namespace {

template <bool STAGE1, int kM, bool kQ, bool kGuard = false, bool kFifo = false>
bool tt_launch(const CUtensorMap& tm_w, const CUtensorMap& tm_sc, const TtTokMaps& tm_t, TtArgs a, cudaStream_t st) {
  a.stages = 1;
  if (kFifo) {
    // the whole ring is one stage of `kb` KB, whose nominal token part is what the weight tiles leave (TtRing only takes its size from it)
    const int kb = (227 * 1024 - 1024 - static_cast<int>(tt_smem(a.E, 0, 0, 0).total) - kTtSfSlots * kM * 2048) >> 10;
    a.t_bytes = kb * 1024 - kM * kTtTile;
  }
  while (!kFifo && a.stages < kTtMaxStages && tt_smem(a.E, kM, a.stages + 1, a.t_bytes).total + 1024 <= 227 * 1024) ++a.stages;
  static PerDeviceFlag flag;
  if (!once_per_device(flag, [] {
        return cudaFuncSetAttribute(ffn_twoterm_kernel<STAGE1, kM, kQ, kGuard, kFifo>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess;
      }))
    return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(sm_count() & ~1));
  cfg.blockDim = dim3(kTtThreads);
  cfg.dynamicSmemBytes = tt_smem(a.E, kM, a.stages, a.t_bytes).total + 1024;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, ffn_twoterm_kernel<STAGE1, kM, kQ, kGuard, kFifo>, tm_w, tm_sc, tm_t, a) == cudaSuccess;
}

}  // namespace

bool twoterm_chosen(const moe_shape_t& choice, const ExpertWeights& w) {
  const long long S = static_cast<long long>(choice.T) * choice.k;
  // Few rows per expert of large ones: the eight-term kernel is ahead up to six, on weights in rows and in moe_prepack's tiles
  // (256 experts of 4096 x 2048, top-8, layers in a row, 4 / 5 / 6 / 7 / 8 rows, eight terms and two: tiles 532 us and 602,
  // 555 and 609, 574 and 615, 672 and 625, 672 and 631; rows 583 and 645, 615 and 670, 632 and 685, 733 and 694, 736 and 699).
  // With H = 2048 the two meet about 5 (2048 x 2048, 4 / 5 / 6 / 8 rows: tiles 307 and 318, 311 and 314, 347 and 317, 396 and
  // 334; rows 323 and 335, 329 and 338, 367 and 346, 424 and 350; after a pause, at higher clocks, two terms are ahead at 4 as
  // well, 310 and 300): they stay with the line at 4 of twoterm_batch_ok.  One line for both layouts, so that they give
  // the same bits.
  if (choice.H >= 4096 && choice.I >= 1024 && S <= 6LL * choice.E && native_shape_ok(choice, w.w13, w.w2)) return false;
  // A layer of small experts is done in a few rounds of either kernel, and the launches that look for experts to be done again
  // decide (L2 cold, this call / bf16 kernel: 64 experts of 512 x 512, 128 rows 59 us and 56, 200 rows 74 and 65; 32 of 1024 x
  // 512, 128 rows 57 and 50; with fewer rows or more experts the other way: 64 of 512 x 512, 64 rows 45 and 48, 128 of them,
  // 128 rows 79 and 97).
  const long long expert = static_cast<long long>(choice.H) * choice.I;
  if (umma_shape_ok(choice) && !native_shape_ok(choice, w.w13, w.w2) && S > 112LL * choice.E && expert <= (1 << 19) &&
      expert * choice.E < (1 << 25))
    return false;
  return twoterm_batch_ok(choice) && twoterm_weights_ok(w.w13, w.w2) &&
         (native_shape_ok(choice, w.w13, w.w2) || umma_shape_ok(choice) || w.blocked || stream_shape_ok(choice));
}
bool twoterm_guarded(const moe_shape_t& choice, const ExpertWeights& w) { return !native_shape_ok(choice, w.w13, w.w2); }

// The experts that `flags` names, by the kernel that would take the shape without this one; their rows of the output are
// written again.  The bf16 intermediate lies over the two-term one, which no kernel reads any more.
static int launch_again(const TwoTermInput& in, const int* offsets, const ExpertWeights& w, const moe_shape_t& sh, const moe_shape_t& choice,
                        void* act, float* y_perm, int* status_word, cudaStream_t st, float* const* row_dst, const int* flags) {
  const __nv_bfloat16* rows = in.x;
  if (in.write_rows) {
    rows = in.x_sorted;
  } else if (in.inv_perm != nullptr) {
    if (launch_pdl(twoterm_gather_kernel, dim3(static_cast<unsigned>(sm_count()) * 8), dim3(256), 0, st, in.x, in.ids, in.inv_perm, flags,
                   sh.T, sh.k, sh.H, sh.E, in.x_sorted) != cudaSuccess)
      return MOE_ERR_CUDA;
    rows = in.x_sorted;
  }
  __nv_bfloat16* a = static_cast<__nv_bfloat16*>(act);
  if (umma_shape_ok(choice) || w.blocked) return launch_expert_ffn_umma(rows, offsets, w, sh, a, y_perm, status_word, st, row_dst, flags);
  return launch_expert_ffn_stream(rows, offsets, w.w13, w.s13, w.w2, w.s2, sh, a, y_perm, status_word, st, row_dst, flags);
}

int launch_expert_ffn_twoterm(const TwoTermInput& in, const int* offsets, const ExpertWeights& w, const moe_shape_t& sh,
                              const moe_shape_t& choice, bool guard, void* scratch, float* y_perm, int* status_word, cudaStream_t st,
                              float* const* row_dst, bool again_later, int* finished, int* n_cta) {
  const TwoTermGeometry geo = twoterm_geometry(choice);
  const bool two = geo.max_tok == 64 && sh.H % 512 == 0;  // M tiles of a down item
  const TwoTermScratch L = twoterm_scratch(choice);
  uint8_t* base = static_cast<uint8_t*>(scratch);
  const uint64_t S = static_cast<uint64_t>(sh.T) * sh.k;
  CUtensorMap tm_w13, tm_w2, tm_s13, tm_s2, unused13, unused2;
  TtTokMaps tm_x, tm_a;
  if (!weight_maps(w, sh, &unused13, &tm_s13, &unused2, &tm_s2) ||
      !codes_map_u4(&tm_w13, w.w13, sh.H, static_cast<uint64_t>(sh.E) * 2 * sh.I, w.blocked) ||
      !codes_map_u4(&tm_w2, w.w2, sh.I, static_cast<uint64_t>(sh.E) * sh.H, w.blocked))
    return MOE_ERR_CUDA;
  for (int b = 0; b < kTtBoxes; ++b)
    if (!term_row_map(&tm_x.box[b], base + L.xq, sh.H, 2 * S, 64u >> b) || !term_row_map(&tm_a.box[b], base + L.aq, sh.I, 2 * S, 64u >> b))
      return MOE_ERR_CUDA;
  if (!byte_map_2d(&tm_x.sf, base + L.sfx, 128, (L.sfa - L.sfx) / 128, 128, 4) || !byte_map_2d(&tm_a.sf, base + L.sfa, 128, (L.marks - L.sfa) / 128, 128, 4))
    return MOE_ERR_CUDA;
  uint8_t* marks = base + L.marks;
  int* flags = reinterpret_cast<int*>(base + L.flags);
  const int n_chunk = sh.H / 256;
  int parts = (n_chunk + 7) / 8;  // pieces of a row, a mark each
  const size_t most = static_cast<size_t>(sm_count()) * 8;  // CTAs of the scatter kernel at most (five or six of a SM's eight run at a time)
  const size_t table_bytes = static_cast<size_t>(kTtTableInts * (sh.E + 1)) * 4;
  cudaError_t rc;
  if (in.inv_perm != nullptr) {
    // whole rows per warp where there are tokens enough to fill the chip, pieces of them otherwise
    const size_t per_token = most * 8 / static_cast<size_t>(sh.T);
    const int chunks = per_token >= static_cast<size_t>(n_chunk) ? 1 : (per_token <= 1 ? n_chunk : (n_chunk + static_cast<int>(per_token) - 1) / static_cast<int>(per_token));
    parts = (n_chunk + chunks - 1) / chunks;
    const size_t want = (static_cast<size_t>(sh.T) * parts + 7) / 8;
    const auto scatter = in.write_rows ? (guard ? twoterm_scatter_kernel<true, true> : twoterm_scatter_kernel<false, true>)
                                       : (guard ? twoterm_scatter_kernel<true, false> : twoterm_scatter_kernel<false, false>);
    rc = launch_pdl(scatter, dim3(static_cast<unsigned>(want < most ? want : most)), dim3(256), table_bytes, st, in.x,
                    in.ids, in.inv_perm, offsets, base + L.xq, base + L.sfx, sh.T, sh.k, sh.H, sh.E, geo.max_tok, geo.sf_step, chunks,
                    marks, flags, in.offsets_late ? 1 : 0, in.x_sorted);
  } else {
    // few rows (a block's shared expert, whose chain of launches the block waits for): shorter tasks, more warps.  The call on one expert of
    // 4096 x 2048 with pieces of eight and of two: 40 rows 30.2 us and 28.6, 120 rows 44.3 and 42.8, 225 rows 44.9 and 44.6; 256 rows 45.5
    // and 46.1, 400 rows 64.9 and 67.6, 512 rows 61.2 and 61.7, 1024 rows 76.1 and 77.8 (of 7168 x 2048: 40 rows 36.2 and 34.3, 225 rows 59.2
    // and 58.6, 256 rows 60.4 and 61.1; there 300 rows are the other way, 72.8 and 70.9).  Block of 48 tokens 372.2 and 370.2, of 120 tokens 550 and 548.
    const int chunks = S < 256 ? 2 : 8;
    parts = (n_chunk + chunks - 1) / chunks;
    const size_t want = (S * parts + 7) / 8, resident = static_cast<size_t>(sm_count()) * 4;
    rc = launch_pdl(guard ? twoterm_split_kernel<true> : twoterm_split_kernel<false>, dim3(static_cast<unsigned>(want < resident ? want : resident)), dim3(256), table_bytes, st, in.x,
                    offsets, base + L.xq, base + L.sfx, static_cast<int>(S), sh.H, sh.E, geo.max_tok, geo.sf_step, marks, flags, chunks);
  }
  if (rc != cudaSuccess) return MOE_ERR_CUDA;
  TtArgs a = {};
  a.offsets = offsets;
  a.y = y_perm;
  a.row_dst = row_dst;
  a.status = status_word;
  a.E = sh.E;
  a.I = sh.I;
  a.S = static_cast<int>(S);
  a.blocked = w.blocked ? 1 : 0;
  a.max_tok = geo.max_tok;
  a.sf_step = geo.sf_step;
  // token part of a stage: this CTA's rows of both terms (up to 112 tokens: of one, the passes are all stacked) and their
  // scale factors; a stage is a multiple of 1 KB
  a.sf_off = geo.max_tok * 128;
  a.t_bytes = a.sf_off + (geo.sf_step > 1024 ? 2048 : 1024);
  a.aq = base + L.aq;
  a.sfa = base + L.sfa;
  if (guard) {
    a.marks = reinterpret_cast<const uint4*>(marks);
    a.flags = flags;
    a.parts = parts;
  }
  a.sc = w.s13;
  a.K = sh.H;
  a.R = 2 * sh.I;
  // Up to 16 rows per expert on average, where most passes have 16 or 32 rows (512 tokens, 16 rows: 703 -> 699 us); with 48 rows no step more
  // fits and finding its place costs 1 % (2048 tokens 986 -> 999).  Where no other kernel does experts again: the kernel that does
  // is for more rows, or small layers.
  const bool fifo = !guard && two && S <= 16ull * choice.E;
  if (!(guard  ? tt_launch<true, 2, false, true>(tm_w13, tm_s13, tm_x, a, st)
        : fifo ? tt_launch<true, 2, false, false, true>(tm_w13, tm_s13, tm_x, a, st)
               : tt_launch<true, 2, false>(tm_w13, tm_s13, tm_x, a, st)))
    return MOE_ERR_CUDA;
  a.finished = finished;
  if (n_cta != nullptr) *n_cta = sm_count() & ~1;
  a.sc = w.s2;
  a.K = sh.I;
  a.R = sh.H;
  if (!(fifo  ? tt_launch<false, 2, false, false, true>(tm_w2, tm_s2, tm_a, a, st)
        : two ? tt_launch<false, 2, false>(tm_w2, tm_s2, tm_a, a, st)
              : tt_launch<false, 1, false>(tm_w2, tm_s2, tm_a, a, st)))
    return MOE_ERR_CUDA;
  if (guard && !again_later) {
    const int again = launch_again(in, offsets, w, sh, choice, base + L.aq, y_perm, status_word, st, row_dst, flags);
    if (again != MOE_OK) return again;
  }
  note_kernel("ffn_mxf8_two_term_cta_pair", 3 + (guard && in.inv_perm != nullptr && !in.write_rows ? 1 : 0));
  return MOE_OK;
}

int launch_twoterm_again(const TwoTermInput& in, const int* offsets, const ExpertWeights& w, const moe_shape_t& sh, void* scratch, float* y_perm,
                         int* status_word, cudaStream_t st) {
  const TwoTermScratch L = twoterm_scratch(sh);
  uint8_t* base = static_cast<uint8_t*>(scratch);
  return launch_again(in, offsets, w, sh, sh, base + L.aq, y_perm, status_word, st, nullptr, reinterpret_cast<const int*>(base + L.flags));
}

int launch_expert_ffn_q_pair(const __nv_bfloat16* x_perm, const int* offsets, const ExpertWeights& w, const moe_shape_t& sh,
                             void* scratch, float* y_perm, int* status_word, cudaStream_t st) {
  const QPairScratch L = q_pair_scratch(sh);
  uint8_t* base = static_cast<uint8_t*>(scratch);
  const uint64_t S = static_cast<uint64_t>(sh.T) * sh.k;
  CUtensorMap tm_w13, tm_w2, tm_s13, tm_s2;
  TtTokMaps tm_x, tm_a;
  if (!weight_maps(w, sh, &tm_w13, &tm_s13, &tm_w2, &tm_s2)) return MOE_ERR_CUDA;
  for (int b = 0; b < kTtBoxes; ++b)
    if (!term_row_map(&tm_x.box[b], base + L.xq, sh.H / 2, S, 64u >> b) || !term_row_map(&tm_a.box[b], base + L.aq, sh.I / 2, S, 64u >> b))
      return MOE_ERR_CUDA;
  if (!byte_map_2d(&tm_x.sf, base + L.sfx, 128, (L.sfa - L.sfx) / 128, 128, 4) || !byte_map_2d(&tm_a.sf, base + L.sfa, 128, (L.total - L.sfa) / 128, 128, 4))
    return MOE_ERR_CUDA;
  const size_t want = (S * ((sh.H + 2047) / 2048) + 7) / 8, resident = static_cast<size_t>(sm_count()) * 4;
  if (launch_pdl(twoterm_quant_kernel, dim3(static_cast<unsigned>(want < resident ? want : resident)), dim3(256),
                 static_cast<size_t>(kTtTableInts * (sh.E + 1)) * 4, st, x_perm, offsets, base + L.xq, base + L.sfx, sh.H, sh.E, kQPairTok,
                 2048) != cudaSuccess)
    return MOE_ERR_CUDA;
  TtArgs a = {};
  a.offsets = offsets;
  a.y = y_perm;
  a.status = status_word;
  a.E = sh.E;
  a.I = sh.I;
  a.S = static_cast<int>(S);
  a.blocked = w.blocked ? 1 : 0;
  a.max_tok = kQPairTok;
  a.sf_step = 2048;
  a.sf_off = kQPairTok / 2 * 128;
  a.t_bytes = a.sf_off + 2048;
  a.aq = base + L.aq;
  a.sfa = base + L.sfa;
  a.sc = w.s13;
  a.K = sh.H;
  a.R = 2 * sh.I;
  if (!tt_launch<true, 2, true>(tm_w13, tm_s13, tm_x, a, st)) return MOE_ERR_CUDA;
  a.sc = w.s2;
  a.K = sh.I;
  a.R = sh.H;
  if (!tt_launch<false, 1, true>(tm_w2, tm_s2, tm_a, a, st)) return MOE_ERR_CUDA;
  note_kernel("ffn_mxf4_quantised_cta_pair", 3);
  return MOE_OK;
}

}  // namespace moe
