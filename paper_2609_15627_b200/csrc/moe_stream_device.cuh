// The register-expansion arithmetic of the expert FFN, shared by the streaming kernel and the one-cluster layer: 128 elements of K
// of a tile of 16 weight rows times up to eight rows of activations.
#pragma once

#include "moe_sm100_primitives.cuh"

namespace moe {

MOE_DEVINL void mma_bf16_16x8x16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// eight consecutive activations -> the pairs that the expansion of eight codes makes
MOE_DEVINL void stream_activations(const uint4& v, uint32_t* b) {
  b[0] = __byte_perm(v.x, v.z, 0x5410);  // elements (0,4)
  b[1] = __byte_perm(v.x, v.z, 0x7632);  // elements (1,5)
  b[2] = __byte_perm(v.y, v.w, 0x5410);  // elements (2,6)
  b[3] = __byte_perm(v.y, v.w, 0x7632);  // elements (3,7)
}
// 32 codes of either half of the tile's rows per lane, their scales, the activations of the lane's row; c2: a second chain, so that
// consecutive MMAs do not wait on each other
MOE_DEVINL void stream_group(float (&c)[4], float (&c2)[4], const uint4& wa, const uint4& wb, uint32_t ma, uint32_t mb, const uint32_t (&breg)[16],
                             uint32_t k1, uint32_t k2) {
  const uint32_t wav[4] = {wa.x, wa.y, wa.z, wa.w};
  const uint32_t wbv[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t pa[4], pb[4];
    dequant8(wav[q], ma, k1, k2, pa);
    dequant8(wbv[q], mb, k1, k2, pb);
    mma_bf16_16x8x16(c, pa[0], pb[0], pa[1], pb[1], breg[4 * q + 0], breg[4 * q + 1]);
    mma_bf16_16x8x16(c2, pa[2], pb[2], pa[3], pb[3], breg[4 * q + 2], breg[4 * q + 3]);
  }
}
MOE_DEVINL __nv_bfloat16 stream_swiglu(float g, float u) { return __float2bfloat16_rn((g / (1.0f + __expf(-g))) * u); }

}  // namespace moe
