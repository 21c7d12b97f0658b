// The whole layer in one launch, for layers that fit the shared memory of one thread-block cluster: a few experts of a few
// hundred rows, a few tokens.  Such a layer's kernels each last 3 to 6 us, nearly all of it launch and memory latency, so what
// counts is how many of them follow one another.  Here every CTA of a cluster of eight keeps some experts' weights whole: while
// they are copied into shared memory every CTA routes all tokens (a warp per token) and sorts
// the slots (a thread per slot, by counting), so nothing is exchanged; a CTA then runs its own experts' rows through both
// projections, the intermediate staying in its shared memory; the rows of y_perm meet at one cluster barrier, behind which
// all CTAs reduce them.  Everything the four calls write is written.
// 16 tokens, 8 experts of 256 x 128, top-2, layers in a row: 21.0 us in five launches -> 8.0 (in a graph 13.8 -> 7.6).  Copies of the
// weights that started before the kernel in front had ended gave 7.35 (7.0); but that kernel may be the one that writes them, as it may
// in front of the streaming kernel.
//
// The arithmetic is the streaming kernel's (moe_ffn_stream.cu), K group by K group in its order, so that the rows have the
// same bits: there warp w holds the 128-element groups w, w + 16, .. of K and the warps' sums are added in order; up to
// K = 2048 that is one group a warp, so a warp that goes through the groups and adds their sums does the same additions.
#include "moe_route_device.cuh"
#include "moe_stream_device.cuh"

namespace moe {

namespace {

constexpr int kSmallCluster = 8;
constexpr int kSmallThreads = 512;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallMaxTok = 32, kSmallMaxSlots = 128, kSmallMaxK = 2048, kSmallMaxE = 256;
constexpr size_t kSmallSmem = 220 * 1024;

struct SmallArgs {
  const float* logits;
  const __nv_bfloat16* x;
  const uint8_t *w13, *s13, *w2, *s2;
  int *ids, *offsets, *perm, *inv_perm;
  float *w, *y;
  __nv_bfloat16 *x_perm, *out;
  uint32_t k1, k2;  // multipliers of the E2M1 expansion, kept opaque to the compiler
  int T, H, I, E, k;
};

// Shared memory of a CTA: its experts' weights, each [w13 | s13 | w2 | s2]; the tokens' rows and the rows of the intermediate, padded by
// 16 bytes so that the eight rows of an MMA lie in different banks; the tables of the sort
struct SmallSmem {
  size_t w13, s13, w2, s2, expert, x, act, ids, wt, pos, slot, off, total;
  int x_pitch, a_pitch;  // elements
};
__host__ __device__ inline SmallSmem small_smem(int T, int H, int I, int E, int k) {
  SmallSmem m;
  const size_t n = static_cast<size_t>(H) * I;
  m.w13 = 0;
  m.s13 = n;
  m.w2 = m.s13 + n / 16;
  m.s2 = m.w2 + n / 2;
  m.expert = m.s2 + n / 32;
  m.x_pitch = H + 8;
  m.a_pitch = I + 8;
  const int mine = (E + kSmallCluster - 1) / kSmallCluster;
  size_t off = mine * m.expert;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 15) / 16 * 16;
    return o;
  };
  m.x = take(static_cast<size_t>(T) * m.x_pitch * 2);
  m.act = take(static_cast<size_t>(T) * m.a_pitch * 2);  // one expert's rows at a time: a token chooses it once at most
  m.ids = take(static_cast<size_t>(T) * k * 4);
  m.wt = take(static_cast<size_t>(T) * k * 4);
  m.pos = take(static_cast<size_t>(T) * k * 4);
  m.slot = take(static_cast<size_t>(T) * k * 4);
  m.off = take((static_cast<size_t>(E) + 1) * 4);
  m.total = off;
  return m;
}

MOE_DEVINL void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
MOE_DEVINL void copy_async(unsigned char* dst, const uint8_t* src, size_t bytes) {  // whole block, in 16-byte pieces
  for (size_t i = threadIdx.x * 16; i < bytes; i += kSmallThreads * 16) cp_async16(dst + i, src + i);
}

// One tile of 16 weight rows times up to eight rows of activations: rows tile_a + 0..7 and tile_b + 0..7 of codes and scale bytes,
// activations of rows row(0..7) of `act`.  Sums in the order described above: v[0], v[1] row tile_a + g, activations 2t and 2t + 1;
// v[2], v[3] row tile_b + g.
template <typename Row>
MOE_DEVINL void small_tile(const unsigned char* codes, const unsigned char* scales, int tile_a, int tile_b, int K, const __nv_bfloat16* act,
                           Row row, int n_rows, uint32_t k1, uint32_t k2, float (&v)[4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const unsigned char* ca = codes + static_cast<size_t>(tile_a + g) * (K / 2) + t * 16;
  const unsigned char* cb = codes + static_cast<size_t>(tile_b + g) * (K / 2) + t * 16;
  const unsigned char* sa = scales + static_cast<size_t>(tile_a + g) * (K / 32) + t;
  const unsigned char* sb = scales + static_cast<size_t>(tile_b + g) * (K / 32) + t;
  const bool live = g < n_rows;
  const uint4* src = reinterpret_cast<const uint4*>(act + (live ? row(g) : 0) + t * 32);
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = 0.0f;
  for (int sc = 0; sc < K / 128; ++sc) {
    uint32_t breg[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 b = live ? src[sc * 16 + q] : make_uint4(0u, 0u, 0u, 0u);
      stream_activations(b, breg + 4 * q);
    }
    float c[4] = {0.0f, 0.0f, 0.0f, 0.0f}, c2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    stream_group(c, c2, *reinterpret_cast<const uint4*>(ca + sc * 64), *reinterpret_cast<const uint4*>(cb + sc * 64), scale_mult(sa[sc * 4]),
                 scale_mult(sb[sc * 4]), breg, k1, k2);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] += c[i] + c2[i];
  }
}

}  // namespace

__global__ void __launch_bounds__(kSmallThreads, 1) layer_small_kernel(const SmallArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const SmallSmem m = small_smem(a.T, a.H, a.I, a.E, a.k);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, rank = static_cast<int>(blockIdx.x);  // (one cluster)
  const int S = a.T * a.k;
  __nv_bfloat16* s_x = reinterpret_cast<__nv_bfloat16*>(smem + m.x);
  __nv_bfloat16* s_act = reinterpret_cast<__nv_bfloat16*>(smem + m.act);
  int* s_ids = reinterpret_cast<int*>(smem + m.ids);
  float* s_w = reinterpret_cast<float*>(smem + m.wt);
  int* s_pos = reinterpret_cast<int*>(smem + m.pos);    // sorted row of a slot
  int* s_slot = reinterpret_cast<int*>(smem + m.slot);  // slot of a sorted row
  int* s_off = reinterpret_cast<int*>(smem + m.off);
  pdl_launch_dependents();  // (whatever comes next waits before it reads)
  pdl_wait();  // the kernel in front may write the weights, the logits and the rows, and may still read what is written here
  const size_t n = static_cast<size_t>(a.H) * a.I;
  for (int e = rank, j = 0; e < a.E; e += kSmallCluster, ++j) {
    unsigned char* dst = smem + j * m.expert;
    copy_async(dst + m.w13, a.w13 + e * n, n);
    copy_async(dst + m.s13, a.s13 + e * (n / 16), n / 16);
    copy_async(dst + m.w2, a.w2 + e * (n / 2), n / 2);
    copy_async(dst + m.s2, a.s2 + e * (n / 32), n / 32);
  }
  const int per_row = a.H / 8;
  for (int i = tid; i < a.T * per_row; i += kSmallThreads) {
    const int t = i / per_row, c = i - t * per_row;
    cp_async16(s_x + static_cast<size_t>(t) * m.x_pitch + c * 8, a.x + static_cast<size_t>(t) * a.H + c * 8);
  }
  // ---- routing: a warp per token ----
  for (int t = wid; t < a.T; t += kSmallWarps) {
    int my_id;
    float my_v;
    warp_topk_256(a.logits + static_cast<size_t>(t) * a.E, a.E, a.k, lane, &my_id, &my_v);
    const float wt = warp_softmax_selected(my_v, a.k, lane);
    if (lane < a.k) {
      s_ids[t * a.k + lane] = my_id;
      s_w[t * a.k + lane] = wt;
      if (rank == 0) {
        a.ids[t * a.k + lane] = my_id;
        a.w[t * a.k + lane] = wt;
      }
    }
  }
  __syncthreads();
  // ---- sort: slots of smaller experts, then earlier slots of the same one ----
  if (tid < S) {
    const int e = s_ids[tid];
    int p = 0;
    for (int s = 0; s < S; ++s) p += s_ids[s] < e || (s_ids[s] == e && s < tid);
    s_pos[tid] = p;
    s_slot[p] = tid;
    if (rank == 0) {
      a.inv_perm[tid] = p;
      a.perm[p] = tid;
    }
  } else if (tid >= kSmallMaxSlots && tid - kSmallMaxSlots <= a.E) {
    for (int e = tid - kSmallMaxSlots; e <= a.E; e += kSmallThreads - kSmallMaxSlots) {
      int p = 0;
      for (int s = 0; s < S; ++s) p += s_ids[s] < e;
      s_off[e] = p;
      if (rank == 0) a.offsets[e] = p;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // ---- this CTA's experts ----
  for (int e = rank, j = 0; e < a.E; e += kSmallCluster, ++j) {
    const unsigned char* we = smem + j * m.expert;
    const int p0 = s_off[e], rows = s_off[e + 1] - p0;
    for (int i = tid; i < rows * per_row; i += kSmallThreads) {
      const int r = i / per_row, c = i - r * per_row;
      *reinterpret_cast<uint4*>(a.x_perm + static_cast<size_t>(p0 + r) * a.H + c * 8) =
          *reinterpret_cast<const uint4*>(s_x + static_cast<size_t>(s_slot[p0 + r] / a.k) * m.x_pitch + c * 8);
    }
    const int blocks = (rows + 7) / 8, g = lane >> 2, t = lane & 3;
    for (int u = wid; u < a.I / 8 * blocks; u += kSmallWarps) {  // 8 gate rows and the matching 8 up rows
      const int r0 = u % blocks * 8, i0 = u / blocks * 8;
      float v[4];
      small_tile(we + m.w13, we + m.s13, i0, a.I + i0, a.H, s_x, [&](int r) { return s_slot[p0 + r0 + r] / a.k * m.x_pitch; }, rows - r0, a.k1,
                 a.k2, v);
      const int ra = r0 + 2 * t;
      if (ra < rows) s_act[ra * m.a_pitch + i0 + g] = stream_swiglu(v[0], v[2]);
      if (ra + 1 < rows) s_act[(ra + 1) * m.a_pitch + i0 + g] = stream_swiglu(v[1], v[3]);
    }
    __syncthreads();
    for (int u = wid; u < a.H / 16 * blocks; u += kSmallWarps) {
      const int r0 = u % blocks * 8, n0 = u / blocks * 16;
      float v[4];
      small_tile(we + m.w2, we + m.s2, n0, n0 + 8, a.I, s_act, [&](int r) { return (r0 + r) * m.a_pitch; }, rows - r0, a.k1, a.k2, v);
      const int ra = r0 + 2 * t;
      float* ya = a.y + static_cast<size_t>(p0 + ra) * a.H + n0 + g;
      if (ra < rows) {
        ya[0] = v[0];
        ya[8] = v[2];
      }
      if (ra + 1 < rows) {
        ya[a.H] = v[1];
        ya[a.H + 8] = v[3];
      }
    }
    __syncthreads();  // (the next expert's intermediate takes the place of this one's)
  }
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  // ---- combine: moe_combine's arithmetic, four columns a thread ----
  const int groups = a.H / 4;
  for (int i = rank * kSmallThreads + tid; i < a.T * groups; i += kSmallCluster * kSmallThreads) {
    const int t = i / groups, c = (i - t * groups) * 4;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
    for (int j = 0; j < a.k; ++j) {
      const float4 v = __ldcg(reinterpret_cast<const float4*>(a.y + static_cast<size_t>(s_pos[t * a.k + j]) * a.H + c));
      const float w = s_w[t * a.k + j];
      acc[0] = __fmaf_rn(w, v.x, acc[0]);
      acc[1] = __fmaf_rn(w, v.y, acc[1]);
      acc[2] = __fmaf_rn(w, v.z, acc[2]);
      acc[3] = __fmaf_rn(w, v.w, acc[3]);
    }
    __nv_bfloat162 o[2] = {__floats2bfloat162_rn(acc[0], acc[1]), __floats2bfloat162_rn(acc[2], acc[3])};
    *reinterpret_cast<uint2*>(a.out + static_cast<size_t>(t) * a.H + c) = *reinterpret_cast<uint2*>(o);
  }
}

// (Where the streaming kernel would take the layer: the caller asks for that.)  What fits shared memory and, since the eight CTAs go
// through all rows where the streaming kernel's 148 would, up to 128 slots (this / five launches, in a graph: one token of 8 experts
// of 1024 x 128, top-8 13.8 us and 16.5, 8 tokens of 32 of 256 x 128, top-8 18.6 and 19.8; 32 tokens, 256 slots, of 8 of 256 x 128 24.1
// and 21.5.  With seven or eight experts a CTA and 64 slots or more it is ahead only without a graph: 16 tokens of 64 of 128 x 128,
// top-4 22.4 and 24.9, in a graph 22.1 and 20.5).  And up to 2^20 weights times rows per CTA that has an expert (launched, and in a graph: 32
// tokens of 8 of 512 x 128, top-4, which is that, 22.8 us and 25.9, 22.5 and 21.7; of 8 of 384 x 256, top-4, one and a half times that, 28.9 and
// 28.2, 28.5 and 24.3; of 4 of 512 x 128, top-4, twice that, 27.2 and 24.6, 27.1 and 21.1).
bool layer_small_ok(const moe_shape_t& s) {
  return s.T <= kSmallMaxTok && s.T * s.k <= kSmallMaxSlots && s.E <= kSmallMaxE && s.H <= kSmallMaxK && s.I <= kSmallMaxK &&
         static_cast<long long>(s.T) * s.k * s.H * s.I <= (1LL << 20) * (s.E < kSmallCluster ? s.E : kSmallCluster) &&
         small_smem(s.T, s.H, s.I, s.E, s.k).total <= kSmallSmem;
}

int launch_layer_small(const float* logits, const __nv_bfloat16* x, const ExpertWeights& w, const moe_shape_t& s, const SmallLayerOut& o,
                       cudaStream_t st) {
  static PerDeviceFlag flag;
  if (!once_per_device(flag, [] {
        return cudaFuncSetAttribute(layer_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmallSmem)) == cudaSuccess;
      }))
    return MOE_ERR_CUDA;
  const SmallArgs a{logits, x, w.w13, w.s13, w.w2, w.s2, o.ids, o.offsets, o.perm, o.inv_perm, o.w, o.y_perm, o.x_perm, o.out, 0x1040u, 0x0104u,
                    s.T, s.H, s.I, s.E, s.k};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kSmallCluster);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = small_smem(s.T, s.H, s.I, s.E, s.k).total;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = kSmallCluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, layer_small_kernel, a) != cudaSuccess) return MOE_ERR_CUDA;
  note_kernel("layer_one_cluster", 1);
  return MOE_OK;
}

}  // namespace moe
