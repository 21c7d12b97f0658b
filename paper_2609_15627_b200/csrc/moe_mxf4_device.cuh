// Device routines shared by the kernels that feed the block-scaled FP4 tensor-core instruction (kind::mxf4): the MMA
// itself with its instruction descriptor, tensor-memory stores for scale factors, the split of a bf16 activation row
// into E2M1 term rows with per-32 block scales, and the bounded wait on a global counter.
#pragma once

#include <cuda_fp4.h>

#include "moe_sm100_primitives.cuh"

namespace moe {

constexpr int kTerms = 8;  // E2M1 terms per activation value: x = sum_t 2^(s_t) * q_t, residual below 2^-16 of the block's maximum

MOE_DEVINL void tmem_st_32x8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
MOE_DEVINL void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// One K step of 256: D[tmem] (+)= A[smem, E2M1] * B[smem, E2M1]^T, K = 64 per instruction, descriptors advancing 32 bytes
// along the swizzled rows.  A row's eight UE8M0 scales of the step are two words, kSfa (kSfb) columns of tensor memory apart,
// of which an instruction takes one half.  By a whole convergent warp, issued by an elected lane (see umma_commit_elect).
template <int kSfa, int kSfb>
MOE_DEVINL void umma_mxf4_step(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t sfa, uint32_t sfb,
                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred q, p, t;\n\t.reg .b64 a, b;\n\t.reg .b32 id, sa, sb;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "setp.eq.b32 t, 0, 0;\n\t"
      "add.s64 a, %1, 0;\n\tadd.s64 b, %2, 0;\n\tadd.u32 id, %3, 0x00000000;\n\tadd.u32 sa, %4, 0;\n\tadd.u32 sb, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], p;\n\t"
      "add.s64 a, %1, 2;\n\tadd.s64 b, %2, 2;\n\tadd.u32 id, %3, 0x40000020;\n\tadd.u32 sa, %4, 0;\n\tadd.u32 sb, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
      "add.s64 a, %1, 4;\n\tadd.s64 b, %2, 4;\n\tadd.u32 id, %3, 0x00000000;\n\tadd.u32 sa, %4, %7;\n\tadd.u32 sb, %5, %8;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
      "add.s64 a, %1, 6;\n\tadd.s64 b, %2, 6;\n\tadd.u32 id, %3, 0x40000020;\n\tadd.u32 sa, %4, %7;\n\tadd.u32 sb, %5, %8;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], a, b, id, [sa], [sb], t;\n\t"
      "}" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(sfa), "r"(sfb), "r"(accumulate), "n"(kSfa), "n"(kSfb)
      : "memory");
}
// instruction descriptor: A and B E2M1, UE8M0 scales, M = 128, N = 256 (or n_cols), bytes 0,1 of the scale words
MOE_DEVINL uint32_t idesc_mxf4(uint32_t n_cols = 256u) {
  return (1u << 7) | (1u << 10) | ((n_cols >> 3) << 17) | (1u << 23) | ((128u >> 4) << 24);
}

// Bounded wait until *p >= need (acquire at GPU scope); same give-up rules as mbar_wait
MOE_DEVINL void counter_wait_ge(const int* p, int need, int* status) {
  const long long t0 = clock64();
  int spins = 0;
  while (true) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if (v >= need) return;
    const long long waited = clock64() - t0;
    if (waited > kWaitLimitCycles) {
      if (status != nullptr) atomicExch(status, static_cast<int>(MOE_ERR_TIMEOUT));
      return;
    }
    if (((++spins) & 63) == 0 && waited > 2000000 && status != nullptr && *reinterpret_cast<volatile int*>(status) != 0) return;
    __nanosleep(64);
  }
}
// The same by a whole convergent warp (see mbar_wait_warp)
MOE_DEVINL void counter_wait_ge_warp(const int* p, int need, int* status) {
  const long long t0 = clock64();
  int spins = 0;
  while (true) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if (__all_sync(0xffffffffu, v >= need)) return;
    const long long waited = clock64() - t0;
    if (__any_sync(0xffffffffu, waited > kWaitLimitCycles)) {
      if (status != nullptr) atomicExch(status, static_cast<int>(MOE_ERR_TIMEOUT));
      return;
    }
    if (((++spins) & 63) == 0 &&
        __any_sync(0xffffffffu, waited > 2000000 && status != nullptr && *reinterpret_cast<volatile int*>(status) != 0))
      return;
    __nanosleep(64);
  }
}
// orders this thread's generic-proxy accesses with its asynchronous-proxy (TMA) accesses, global memory included
MOE_DEVINL void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
MOE_DEVINL void prefetch_tmap(const void* tmap) { asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory"); }

MOE_DEVINL float pow2f(int e) { return __uint_as_float(static_cast<uint32_t>(e + 127) << 23); }  // e in [-126, 127]
// Block exponent of a term: the smallest s with amax <= 6 * 2^s (amax > 0), kept inside the UE8M0 range
MOE_DEVINL int term_exp(float amax) {
  const uint32_t u = __float_as_uint(amax);
  const int e = static_cast<int>((u >> 23) & 0xFFu) - 127;
  const int s = ((u & 0x7FFFFFu) <= 0x400000u) ? e - 2 : e - 1;  // 1.5 * 2^e = 6 * 2^(e-2)
  return max(-126, min(s, 126));
}
// Two values (already divided by the block scale) -> one byte of two E2M1 codes (a in the low nibble) and their
// decoded values.  (A version in plain float and integer instructions - step chosen by two compares, the multiple by
// the round-to-nearest-even of one float addition - gives the same codes and was slower: decode_c64 call +4 %.)
MOE_DEVINL uint32_t e2m1_pair(float a, float b, float* qa, float* qb) {
  const __nv_fp4x2_storage_t c = __nv_cvt_float2_to_fp4x2(make_float2(a, b), __NV_E2M1, cudaRoundNearest);
  const __half2_raw h = __nv_cvt_fp4x2_to_halfraw2(c, __NV_E2M1);
  const float2 q = __half22float2(*reinterpret_cast<const __half2*>(&h));
  *qa = q.x;
  *qb = q.y;
  return static_cast<uint32_t>(c);
}

// 8 x 8 nibble transpose over lanes 8a..8a+7: in, nibble t of lane l is (token t, row l); out, nibble l of lane t
MOE_DEVINL uint32_t transpose_8x8_nibbles(uint32_t w, int lane) {
  uint32_t p = __shfl_xor_sync(0xffffffffu, w, 4);
  w = (lane & 4) ? __byte_perm(w, p, 0x3276) : __byte_perm(w, p, 0x5410);
  p = __shfl_xor_sync(0xffffffffu, w, 2);
  w = (lane & 2) ? __byte_perm(w, p, 0x3715) : __byte_perm(w, p, 0x6240);
  p = __shfl_xor_sync(0xffffffffu, w, 1);
  return (lane & 1) ? ((p >> 4) & 0x0F0F0F0Fu) | (w & 0xF0F0F0F0u) : (w & 0x0F0F0F0Fu) | ((p & 0x0F0F0F0Fu) << 4);
}

// Eight threads (consecutive lanes) share one 32-element block, four consecutive values each: the 8-term split,
// for NB independent blocks at once (their dependency chains interleave).  `store(nb, t, bytes, se)` receives
// term t's two bytes of codes (values 0,1 and 2,3 of this thread) and the block exponent.  All 32 lanes must call
// it together.  (With NB > 1 the chains overlap little: the exchanges and the stores keep their program order.)
template <int NB, typename Store>
MOE_DEVINL void split_terms(float (&r)[NB][4], Store store) {
#pragma unroll 1
  for (int t = 0; t < kTerms; ++t) {
#pragma unroll
    for (int nb = 0; nb < NB; ++nb) {
      float amax = fmaxf(fmaxf(fabsf(r[nb][0]), fabsf(r[nb][1])), fmaxf(fabsf(r[nb][2]), fabsf(r[nb][3])));
      amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
      amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
      amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 4));
      const int se = (amax > 0.0f) ? term_exp(amax) : 0;
      const float inv = pow2f(-se), sc = pow2f(se);
      float q0, q1, q2, q3;
      const uint32_t bytes =
          e2m1_pair(r[nb][0] * inv, r[nb][1] * inv, &q0, &q1) | (e2m1_pair(r[nb][2] * inv, r[nb][3] * inv, &q2, &q3) << 8);
      r[nb][0] = fmaf(-q0, sc, r[nb][0]);
      r[nb][1] = fmaf(-q1, sc, r[nb][1]);
      r[nb][2] = fmaf(-q2, sc, r[nb][2]);
      r[nb][3] = fmaf(-q3, sc, r[nb][3]);
      store(nb, t, bytes, se);
    }
  }
}

// Rows [0, n_rows) of bf16 -> 8 E2M1 term rows each with their scale bytes; thread gt of the grid, 8 threads per 32-element block
// (whole warps call it together)
MOE_DEVINL void split_row_blocks(const __nv_bfloat16* __restrict__ x, uint8_t* __restrict__ aq, uint8_t* __restrict__ aq_sf, int n_rows, int H,
                                 long long gt) {
  const int n_blk = H / 32;
  const long long task = gt >> 3;  // (row, block); the grid is padded to whole warps, so whole tasks are in or out
  const int sub = static_cast<int>(gt & 7);
  const bool live = task < static_cast<long long>(n_rows) * n_blk;
  const int p = live ? static_cast<int>(task / n_blk) : 0, b = live ? static_cast<int>(task % n_blk) : 0;
  const uint2 v = __ldcg(reinterpret_cast<const uint2*>(x + static_cast<size_t>(p) * H + b * 32 + sub * 4));
  float r[1][4] = {{__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16),
                   __uint_as_float(v.y & 0xFFFF0000u)}};
  split_terms<1>(r, [&](int, int t, uint32_t bytes, int se) {
    if (live) {
      const size_t row = static_cast<size_t>(p) * kTerms + t;
      *reinterpret_cast<uint16_t*>(aq + row * (H / 2) + b * 16 + sub * 2) = static_cast<uint16_t>(bytes);
      if (sub == 0) aq_sf[row * n_blk + b] = static_cast<uint8_t>(se + 127);
    }
  });
}

}  // namespace moe
