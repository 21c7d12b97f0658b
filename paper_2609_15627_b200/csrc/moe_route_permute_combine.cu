// Router top-k, route production (stable expert sort + row gather) and the fixed-order fp32 combine.
// All three are integer / bandwidth work: warp shuffles, shared-memory histograms, prefix scans and
// 16-byte vector copies.  Results are bit-defined (see include/moe_b200.h).
#include "moe_common.cuh"
#include "moe_mxf4_device.cuh"
#include "moe_route_device.cuh"

namespace moe {

// =================================================================================================
// moe_route
// =================================================================================================

// Exclusive scan of counts[0..E) into offsets[0..E], offsets[E] = total.  Whole block takes part.
__device__ void block_offsets_scan(const int* counts, int E, int* offsets, int* warp_tot /* smem [32] */) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  const int per = (E + blockDim.x - 1) / blockDim.x;
  const int base = tid * per;
  int sum = 0;
  for (int i = 0; i < per; ++i)
    if (base + i < E) sum += counts[base + i];
  int wtotal;
  const int excl = warp_excl_scan(sum, lane, &wtotal);
  if (lane == 0) warp_tot[wid] = wtotal;
  __syncthreads();
  if (wid == 0) {
    const int v = (lane < nw) ? warp_tot[lane] : 0;
    int tot;
    const int ex = warp_excl_scan(v, lane, &tot);
    __syncwarp();
    warp_tot[lane] = ex;
    if (lane == 0) offsets[E] = tot;
  }
  __syncthreads();
  int run = warp_tot[wid] + excl;
  for (int i = 0; i < per; ++i) {
    if (base + i < E) {
      offsets[base + i] = run;
      run += counts[base + i];
    }
  }
}

// kSingle: one CTA handles every token and builds the histogram in shared memory.  Otherwise a warp per token and nothing
// but its ids and weights: the histogram is another launch's (route_offsets_kernel or the sort), which reads the ids back in
// chunks.  (With a global atomic per slot, 256 addresses for all, 8192 tokens took 37 us in a row of layers and 32768 129, with a
// memset in front; without, and with the keys sorted, 17 and 48.)  zero: counters [0, n_zero) that the next launch adds to, or null.  kWide: more than 256 experts.
template <bool kSingle, bool kWide>
__global__ void __launch_bounds__(kSingle ? 1024 : 256, kSingle || kWide ? 1 : 6) route_kernel(const float* __restrict__ logits, int T, int E, int k,
                                                     int* __restrict__ ids, float* __restrict__ w,
                                                     int* __restrict__ offsets, int* zero, int n_zero) {
  extern __shared__ float sm_f[];
  const int nw = blockDim.x >> 5;
  float* rows = sm_f;                                   // [nw][E], more than 256 experts or one CTA
  int* s_counts = reinterpret_cast<int*>(sm_f + nw * E);  // [E], one CTA
  int* s_misc = s_counts + E;                           // [32]
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // Programmatic dependent launch on both sides: what comes next may start and waits before it reads; this kernel may
  // itself have started while the kernel before it (the previous layer call's moe_combine, which still reads the
  // routing weights this kernel is about to overwrite) is running, so it writes nothing to global memory before it waits, and reads the
  // logits before only where one CTA routes (what moe_route promises: up to 32 tokens).
  pdl_launch_dependents();
  bool waited = false;
  if (kSingle) {
    for (int e = tid; e < E; e += blockDim.x) s_counts[e] = 0;
    __syncthreads();
  } else {
    pdl_wait();
    waited = true;
    if (zero != nullptr && blockIdx.x == 0)
      for (int e = tid; e < n_zero; e += blockDim.x) zero[e] = 0;
  }
  float* row = rows + wid * E;
  const int t0 = blockIdx.x * nw + wid;
  const int tstride = gridDim.x * nw;
  for (int t = t0; t < T; t += tstride) {
    int my_id;
    float my_v;
    if (!kSingle && !kWide) {
      warp_topk_256_sorted(logits + static_cast<size_t>(t) * E, E, k, lane, &my_id, &my_v);
    } else {
      for (int e = lane; e < E; e += 32) row[e] = logits[static_cast<size_t>(t) * E + e];
      __syncwarp();
      warp_topk(row, E, k, lane, &my_id, &my_v);
    }
    const float wt = warp_softmax_selected(my_v, k, lane);
    if (!waited) {
      pdl_wait();
      waited = true;
    }
    if (lane < k) {
      ids[static_cast<size_t>(t) * k + lane] = my_id;
      w[static_cast<size_t>(t) * k + lane] = wt;
      if (kSingle && my_id >= 0) atomicAdd(&s_counts[my_id], 1);
    }
    __syncwarp();
  }
  if (!waited) pdl_wait();  // warps without a token
  if (kSingle) {
    __syncthreads();
    block_offsets_scan(s_counts, E, offsets, s_misc);
  }
}

// expert_offsets from the ids: a histogram in shared memory per chunk, added to counts[0..E), which the router cleared; the last CTA
// (ticket in counts[E]) scans them.
constexpr int kOffsetsChunk = 4096;
__global__ void __launch_bounds__(1024) route_offsets_kernel(const int* __restrict__ ids, int S, int E, int* __restrict__ offsets, int* counts) {
  extern __shared__ int s_hist[];  // [E], then the scan's [32] and a flag
  int* s_misc = s_hist + E;
  const int tid = threadIdx.x;
  for (int e = tid; e < E; e += blockDim.x) s_hist[e] = 0;
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();
  const int s0 = blockIdx.x * kOffsetsChunk + 4 * tid;  // (a chunk is four slots a thread)
  int e4[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) e4[j] = s0 + j < S ? __ldg(ids + s0 + j) : -1;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (e4[j] >= 0) atomicAdd(&s_hist[e4[j]], 1);
  __syncthreads();
  for (int e = tid; e < E; e += blockDim.x)
    if (s_hist[e] != 0) atomicAdd(&counts[e], s_hist[e]);
  __threadfence();
  __syncthreads();
  if (tid == 0) s_misc[32] = atomicAdd(&counts[E], 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (s_misc[32] == 0) return;
  __threadfence();
  for (int e = tid; e < E; e += blockDim.x) s_hist[e] = __ldcg(&counts[e]);
  __syncthreads();
  block_offsets_scan(s_hist, E, offsets, s_misc);
}

// the router alone (no offsets), a warp per token
static int launch_route_ids(const float* logits, int T, int E, int k, int* ids, float* w, int* zero, int n_zero, cudaStream_t st) {
  constexpr int nw = 8;
  const size_t smem = E <= 256 ? 0 : (static_cast<size_t>(nw) * E + E + 40) * 4;
  return launch_pdl(E <= 256 ? route_kernel<false, false> : route_kernel<false, true>, dim3((T + nw - 1) / nw), dim3(nw * 32), smem, st, logits, T, E, k, ids, w, static_cast<int*>(nullptr), zero,
                    n_zero) == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}
static bool route_attr_once() {
  static PerDeviceFlag flag;
  return once_per_device(flag, [] {
    return cudaFuncSetAttribute(route_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) == cudaSuccess &&
           cudaFuncSetAttribute(route_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) == cudaSuccess;
  });
}

int launch_route(const float* logits, int T, int E, int k, int* ids, float* w, int* offsets, int* counters,
                 cudaStream_t st) {
  if (route_sort_ok(T, E)) return launch_route_sort(logits, T, E, k, ids, w, offsets, nullptr, nullptr, nullptr, nullptr, false, st);
  if (!route_attr_once()) return MOE_ERR_CUDA;
  // One CTA up to a round of its 32 warps.  (64 tokens: 19 us in two rounds of one CTA, 7 us on eight.)
  if (T <= 32) {
    const size_t smem = (static_cast<size_t>(32) * E + E + 40) * 4;
    if (launch_pdl(route_kernel<true, true>, dim3(1), dim3(1024), smem, st, logits, T, E, k, ids, w, offsets, static_cast<int*>(nullptr), 0) != cudaSuccess)
      return MOE_ERR_CUDA;
    note_kernel("route_topk_single_cta", 1);
    return MOE_OK;
  }
  const int S = T * k, rc = launch_route_ids(logits, T, E, k, ids, w, counters, E + 1, st);
  if (rc != MOE_OK) return rc;
  if (launch_pdl(route_offsets_kernel, dim3((S + kOffsetsChunk - 1) / kOffsetsChunk), dim3(1024), (static_cast<size_t>(E) + 40) * 4, st, ids, S, E,
                 offsets, counters) != cudaSuccess)
    return MOE_ERR_CUDA;
  note_kernel("route_topk_multi_cta", 2);
  return MOE_OK;
}

// ---- routing and sort of batches that one cluster routes (up to 256 tokens and 256 experts), and the split of their rows ----
// A warp per token, tokens in order over the cluster's CTAs (as many as there are eights of tokens: the warps of a CTA share its
// issue slots).  The warps that chose an expert are the bits of a mask, so a CTA's count of it is a population count and
// a slot's rank the one of the bits below its warp's; the counts meet through distributed shared memory.  Latency is all
// there is to it: one launch, where larger batches take a router and a sort (64 tokens and the split of their rows: 9 us until the
// expert FFN's weights start to stream; 26 with a memset, a router whose last CTA scanned, and a sort).  Not for more than a token per
// warp: 333 tokens in two rounds took 12 us, and those three launches 13 to the end of the sort.
// The CTAs behind the first cluster (kSplit) split the token rows, which depends on no routing, meanwhile.
constexpr int kFrontCluster = 8;
static_assert(kFrontMaxTok == 32 * kFrontCluster, "a warp per token");
template <bool kSplit>
__global__ void __launch_bounds__(1024) route_sort_kernel(const float* __restrict__ logits, int T, int E, int k, int* __restrict__ ids,
                                                          float* __restrict__ w, int* __restrict__ offsets, int* __restrict__ perm,
                                                          int* __restrict__ inv_perm, int* __restrict__ offsets2, int late, const FrontSplit f) {
  __shared__ unsigned s_mask[kFrontMaxE];
  __shared__ int s_cnt[kFrontMaxE], s_all[kFrontMaxE], s_base[kFrontMaxE], s_tot[kFrontMaxE / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  unsigned n_cta, rank;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n_cta));
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  pdl_launch_dependents();  // (whatever comes next waits before it reads)
  if (kSplit && blockIdx.x >= n_cta) {
    pdl_wait();
    const long long gt = static_cast<long long>(blockIdx.x - n_cta) * blockDim.x + tid;
    for (long long i = gt; i < f.n_done; i += static_cast<long long>(gridDim.x - n_cta) * blockDim.x) f.done[i] = 0;
    if (gt == 0 && f.status_clear != nullptr) *f.status_clear = 0;
    split_row_blocks(f.x, f.aq, f.sf, T, f.H, gt);
    return;
  }
  // this kernel may have started while the one before it still reads what is about to be overwritten: only the logits are read
  // before the wait, and not where that one may write them (what moe_route promises above 32 tokens)
  if (late) pdl_wait();
  if (tid < kFrontMaxE) s_mask[tid] = 0u;
  __syncthreads();
  const int per_cta = (T + static_cast<int>(n_cta) - 1) / static_cast<int>(n_cta);  // at most 32
  const int t = static_cast<int>(rank) * per_cta + wid;
  const bool live = wid < per_cta && t < T;
  int my_id = -1;
  float wt = 0.0f;
  if (live) {
    float my_v;
    warp_topk_256(logits + static_cast<size_t>(t) * E, E, k, lane, &my_id, &my_v);
    wt = warp_softmax_selected(my_v, k, lane);
  }
  if (!late) pdl_wait();
  const bool mine = live && lane < k;
  if (mine) {
    ids[static_cast<size_t>(t) * k + lane] = my_id;
    w[static_cast<size_t>(t) * k + lane] = wt;
    atomicOr(&s_mask[my_id], 1u << wid);
  }
  __syncthreads();
  if (tid < E) s_cnt[tid] = __popc(s_mask[tid]);
  if (n_cta > 1)
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  int total = 0, before = 0, ex = 0;
  if (tid < kFrontMaxE) {
    if (tid < E) {
      for (unsigned c = 0; c < n_cta; ++c) {
        uint32_t at;
        int v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(&s_cnt[tid])), "r"(c));
        asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
        total += v;
        before += c < rank ? v : 0;
      }
    }
    int warp_total;
    ex = warp_excl_scan(total, lane, &warp_total);
    if (lane == 0) s_tot[wid] = warp_total;
  }
  __syncthreads();
  if (tid < E) {
    for (int i = 0; i < wid; ++i) ex += s_tot[i];
    s_base[tid] = ex + before;
    s_all[tid] = total;
    if (rank == 0) {
      offsets[tid] = ex;
      if (tid == E - 1) offsets[E] = ex + total;
    }
  }
  if (rank == 0 && tid < 2 && offsets2 != nullptr) offsets2[tid] = tid == 0 ? 0 : T;
  if (n_cta > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");  // (the other CTAs' counts have been read)
  __syncthreads();
  if (inv_perm != nullptr && mine) {
    const int p = s_base[my_id] + __popc(s_mask[my_id] & ((1u << wid) - 1u)), slot = t * k + lane;
    inv_perm[slot] = p;
    if (perm != nullptr) perm[p] = slot;
    if (kSplit) f.tok[p] = s_all[my_id] > f.most ? t | static_cast<int>(0x80000000u) : t;
  }
  if (n_cta > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

bool route_sort_ok(int T, int E) { return E <= kFrontMaxE && T <= kFrontMaxTok; }

int launch_route_sort(const float* logits, int T, int E, int k, int* ids, float* w, int* offsets, int* perm, int* inv_perm, int* offsets2,
                      const FrontSplit* split, bool late, cudaStream_t st) {
  int n_cta = 1;
  while (n_cta < kFrontCluster && n_cta * 8 < T) n_cta *= 2;
  long long extra = 0;
  if (split != nullptr) {
    extra = (static_cast<long long>(T) * (split->H / 32) * 8 + 1023) / 1024;
    extra = (extra + n_cta - 1) / n_cta * n_cta;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(n_cta + extra));
  cfg.blockDim = dim3(1024);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(n_cta);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, split != nullptr ? route_sort_kernel<true> : route_sort_kernel<false>, logits, T, E, k, ids, w, offsets, perm,
                         inv_perm, offsets2, late || T > 32 ? 1 : 0, split != nullptr ? *split : FrontSplit{}) != cudaSuccess)
    return MOE_ERR_CUDA;
  note_kernel(inv_perm != nullptr ? "route_topk_and_sort_one_cluster" : "route_topk_one_cluster", 1);
  return MOE_OK;
}

// =================================================================================================
// moe_permute
// =================================================================================================

MOE_DEVINL void warp_copy_row(const __nv_bfloat16* src, __nv_bfloat16* dst, int H, int lane) {
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  const int n = H / 8;
  // four loads in flight per lane: a row is a few KB and one warp moves it, so latency is what counts - in flight and in the
  // number of warps that fit (eight loads take the registers of a third of them)
  for (int i0 = lane; i0 < n; i0 += 32 * 4) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + 32 * u < n) v[u] = __ldg(&s4[i0 + 32 * u]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + 32 * u < n) d4[i0 + 32 * u] = v[u];
  }
}

// Up to permute_direct slots: a CTA takes eight consecutive slots, counts the earlier slots of each one's expert directly
// (an id is loaded once per CTA and compared with the eight experts) and copies their rows, one warp each; the sort is
// stable by construction.  One launch where the chunked sort takes two, and a third for the rows.
// The count is quadratic and the launches are not.  moe_route and moe_permute one after the other in a graph, 256 experts, top-8, direct /
// chunked: H = 256: 4096 slots 12.0 us and 15.4, 6144 14.4 and 15.3, 8192 17.8 and 15.4, 12288 22.5 and 17.0; H = 1024: 8192 slots 17.5 and
// 17.8, 12288 23.1 and 19.8; H = 2048: 8192 slots 18.6 and 20.0, 12288 24.3 and 23.0, 16384 34.2 and 27.5; H = 4096: 8192 slots 23.0 and
// 26.8, 12288 33.6 and 34.1, 16384 42.2 and 41.7, 24576 64.1 and 57.5.  The two lines were set when the chunked sort had a scan between its
// launches; they lie where H = 1024 and H = 4096 meet now, and 256 and 2048 meet earlier, near 6800 and 11000 slots.
constexpr int permute_direct(bool rows, int H) { return rows && H >= 2048 ? 16384 : 8192; }
// kOffsets: expert_offsets is not there yet.  Then the slots of smaller experts are counted as well, and the last CTA writes it.
template <bool kOffsets>
__global__ void __launch_bounds__(256, kOffsets ? 6 : 8) permute_small_kernel(const __nv_bfloat16* __restrict__ x,
                                                            const int* __restrict__ ids,
                                                            int* __restrict__ offsets, int S, int H, int k,
                                                            __nv_bfloat16* __restrict__ x_perm,
                                                            int* __restrict__ perm, int* __restrict__ inv_perm,
                                                            const int* __restrict__ range_lo, const int* __restrict__ range_hi, int E) {
  __shared__ int s_cnt[8][8];  // [warp][slot of the CTA]
  extern __shared__ int s_hist[];  // kOffsets: [E + 32]
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int s0 = blockIdx.x * 8, s = s0 + wid;
  pdl_wait();                // the router's ids and offsets are complete
  pdl_launch_dependents();   // the expert FFN may set up and start its weight stream
  if (kOffsets && s0 >= S) {  // (one CTA more than the slots take)
    for (int e = threadIdx.x; e < E; e += 256) s_hist[e] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < S; i += 256) atomicAdd(&s_hist[__ldg(ids + i)], 1);
    __syncthreads();
    block_offsets_scan(s_hist, E, offsets, s_hist + E);
    return;
  }
  int e8[8], c8[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    e8[j] = s0 + j < S ? __ldg(ids + s0 + j) : -1;
    c8[j] = 0;
  }
  if constexpr (kOffsets) {  // slots of smaller experts, and earlier slots of the same one
    for (int q = 4 * threadIdx.x; q < S; q += 4 * 256) {
      int v[4];
      if (q + 4 <= S) {
        const int4 v4 = __ldg(reinterpret_cast<const int4*>(ids + q));
        v[0] = v4.x, v[1] = v4.y, v[2] = v4.z, v[3] = v4.w;
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = q + u < S ? __ldg(ids + q + u) : 0x7FFFFFFF;
      }
      const int same = q < s0 ? 1 : 0;  // (s0 is a multiple of 8: all four or none)
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int u = 0; u < 4; ++u) c8[j] += v[u] < e8[j] + same;
    }
  } else {
    for (int q = 4 * threadIdx.x; q < s0; q += 4 * 256) {
      const int4 v = __ldg(reinterpret_cast<const int4*>(ids + q));  // (s0 is a multiple of 8)
#pragma unroll
      for (int j = 0; j < 8; ++j) c8[j] += (v.x == e8[j]) + (v.y == e8[j]) + (v.z == e8[j]) + (v.w == e8[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int c = __reduce_add_sync(0xffffffffu, c8[j]);
    if (lane == 0) s_cnt[wid][j] = c;
  }
  __syncthreads();
  if (s >= S) return;
  int e = 0, c = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    c += s_cnt[j][wid];
    if (j == wid) e = e8[j];
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) c += (j < wid && e8[j] == e);
  const int p = kOffsets ? c : offsets[e] + c;
  if (lane == 0) {
    perm[p] = s;
    inv_perm[s] = p;
  }
  if (x_perm == nullptr || (range_lo != nullptr && (p < *range_lo || p >= *range_hi))) return;
  warp_copy_row(x + static_cast<size_t>(s / k) * H, x_perm + static_cast<size_t>(p) * H, H, lane);
}

// Large S, pass 1: per-chunk histogram.
__global__ void __launch_bounds__(256) permute_count_kernel(const int* __restrict__ ids, int S, int E,
                                                            int* __restrict__ block_counts) {
  extern __shared__ int s_hist[];
  pdl_wait();               // each kernel of the chain waits for the one before it, then lets the next one set up
  pdl_launch_dependents();
  for (int e = threadIdx.x; e < E; e += blockDim.x) s_hist[e] = 0;
  __syncthreads();
  const int base = blockIdx.x * kPermuteChunk;
  for (int i = threadIdx.x; i < kPermuteChunk; i += blockDim.x) {
    const int s = base + i;
    if (s < S) atomicAdd(&s_hist[ids[s]], 1);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < E; e += blockDim.x) block_counts[static_cast<size_t>(blockIdx.x) * E + e] = s_hist[e];
}

// Very large S (more than kSortChunks chunks), between the two passes: one warp per expert turns the per-chunk counts into per-chunk
// start positions.
constexpr int kSortChunks = 512;
__global__ void __launch_bounds__(256) permute_scan_kernel(const int* __restrict__ offsets, int E, int nblk,
                                                           int* __restrict__ block_counts) {
  const int lane = threadIdx.x & 31;
  const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  pdl_wait();
  pdl_launch_dependents();
  if (e >= E) return;
  int running = offsets[e];
  for (int b0 = 0; b0 < nblk; b0 += 32) {
    const int b = b0 + lane;
    const int v = (b < nblk) ? block_counts[static_cast<size_t>(b) * E + e] : 0;
    int tot;
    const int ex = warp_excl_scan(v, lane, &tot);
    if (b < nblk) block_counts[static_cast<size_t>(b) * E + e] = running + ex;
    running += tot;
  }
}

// Large S, pass 2: stable ranks inside a chunk, a slot per thread: warps are ordered through a per-warp count table, lanes through a
// match mask.  What comes before the chunk is summed from the counts of pass 1 by every CTA itself, a row of E counts per chunk and
// all rows in L2: one launch less than a scan between the two (in a row of layers, both: 1027 tokens 6.6 -> 4.6 us, 8192 10.4 -> 7.6, 32768
// 14.2 -> 12.1, with the offsets as well).
// offsets_out: expert_offsets is not there yet and written here by the last chunk; else it is read, or, where that is null as well,
// block_counts holds positions already.
__global__ void __launch_bounds__(kPermuteChunk) permute_scatter_kernel(const int* __restrict__ ids, int S, int E,
                                                                       const int* __restrict__ block_counts, const int* __restrict__ offsets,
                                                                       int* __restrict__ offsets_out, int* __restrict__ perm,
                                                                       int* __restrict__ inv_perm) {
  constexpr int kWarps = kPermuteChunk / 32;
  extern __shared__ int s_base[];  // [E] counts before the chunk, then positions; [E] all counts; [32]; [kWarps][E] 16-bit counts
  int* s_tot = s_base + E;
  int* s_misc = s_tot + E;
  unsigned short* s_w = reinterpret_cast<unsigned short*>(s_misc + 32);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, blk = static_cast<int>(blockIdx.x), nblk = static_cast<int>(gridDim.x);
  for (int i = tid; i < 2 * E; i += kPermuteChunk) s_base[i] = 0;
  for (int i = tid; i < kWarps * E; i += kPermuteChunk) s_w[i] = 0;
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();
  const int s = blk * kPermuteChunk + tid;
  const int e = s < S ? ids[s] : E;
  // the counts: thread (four experts, part) sums every parts-th row, sixteen loads in flight
  const int rows = offsets_out != nullptr ? nblk : blk;
  if (offsets_out == nullptr && offsets == nullptr) {
    if (tid < E) s_base[tid] = block_counts[static_cast<size_t>(blk) * E + tid];
  } else if ((E & 3) == 0) {
    const int quads = E >> 2, parts = kPermuteChunk / quads, cq = tid % quads, part = tid / quads;
    if (part < parts) {
      int before[4] = {0, 0, 0, 0}, all[4] = {0, 0, 0, 0};
#pragma unroll 16
      for (int b = part; b < rows; b += parts) {
        const int4 c = __ldcg(reinterpret_cast<const int4*>(block_counts + static_cast<size_t>(b) * E) + cq);
        const int in_front = b < blk ? -1 : 0;
        all[0] += c.x, all[1] += c.y, all[2] += c.z, all[3] += c.w;
        before[0] += c.x & in_front, before[1] += c.y & in_front, before[2] += c.z & in_front, before[3] += c.w & in_front;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (before[j] != 0) atomicAdd(&s_base[4 * cq + j], before[j]);
        if (all[j] != 0) atomicAdd(&s_tot[4 * cq + j], all[j]);
      }
    }
  } else {
    const int parts = kPermuteChunk / E, ce = tid % E, part = tid / E;  // (E is at most 1024)
    if (part < parts) {
      int before = 0, all = 0;
      for (int b = part; b < rows; b += parts) {
        const int c = __ldcg(block_counts + static_cast<size_t>(b) * E + ce);
        all += c;
        before += b < blk ? c : 0;
      }
      if (before != 0) atomicAdd(&s_base[ce], before);
      if (all != 0) atomicAdd(&s_tot[ce], all);
    }
  }
  const unsigned peers = __match_any_sync(0xffffffffu, e);
  const unsigned before_me = peers & ((1u << lane) - 1u);
  if (e < E && before_me == 0u) s_w[wid * E + e] = static_cast<unsigned short>(__popc(peers));
  __syncthreads();
  if (offsets_out != nullptr) {  // exclusive scan of all counts, an expert per thread
    const int v = tid < E ? s_tot[tid] : 0;
    int wtot;
    int ex = warp_excl_scan(v, lane, &wtot);
    if (lane == 0) s_misc[wid] = wtot;
    __syncthreads();
    for (int i = 0; i < wid; ++i) ex += s_misc[i];
    if (tid < E) {
      s_base[tid] += ex;
      if (blk == nblk - 1) {
        offsets_out[tid] = ex;
        if (tid == E - 1) offsets_out[E] = ex + v;
      }
    }
  } else if (offsets != nullptr && tid < E) {
    s_base[tid] += offsets[tid];
  }
  if (tid < E) {
    unsigned run = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const unsigned c = s_w[w * E + tid];
      s_w[w * E + tid] = static_cast<unsigned short>(run);
      run += c;
    }
  }
  __syncthreads();
  if (e < E) {
    const int p = s_base[e] + s_w[wid * E + e] + __popc(before_me);
    perm[p] = s;
    inv_perm[s] = p;
  }
}

// Large S, pass 3: gather rows, one warp per sorted row.
// range: null, or two device words {first sorted row, row after the last} - only those rows are copied (a rank of an
// expert-parallel job needs the rows of its own experts only)
__global__ void __launch_bounds__(256) permute_gather_kernel(const __nv_bfloat16* __restrict__ x,
                                                             const int* __restrict__ perm, int S, int H, int k,
                                                             __nv_bfloat16* __restrict__ x_perm, const int* __restrict__ range_lo,
                                                             const int* __restrict__ range_hi) {
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  pdl_wait();
  pdl_launch_dependents();
  const int p_lo = range_lo != nullptr ? *range_lo : 0, p_hi = range_hi != nullptr ? *range_hi : S;
  for (int p = p_lo + blockIdx.x * wpb + (threadIdx.x >> 5); p < p_hi; p += gridDim.x * wpb) {
    const int s = perm[p];
    warp_copy_row(x + static_cast<size_t>(s / k) * H, x_perm + static_cast<size_t>(p) * H, H, lane);
  }
}

int launch_gather_rows(const __nv_bfloat16* x, const int* perm, const moe_shape_t& sh, __nv_bfloat16* x_perm, cudaStream_t st) {
  const int S = sh.T * sh.k, grid = min((S + 7) / 8, sm_count() * 16);
  if (launch_pdl(permute_gather_kernel, dim3(grid), dim3(256), 0, st, x, perm, S, sh.H, sh.k, x_perm, static_cast<const int*>(nullptr),
                 static_cast<const int*>(nullptr)) != cudaSuccess)
    return MOE_ERR_CUDA;
  note_kernel("permute_gather_rows", 1);
  return MOE_OK;
}

// count and scatter; offsets_out as permute_scatter_kernel has it
static int launch_chunked_sort(const int* ids, const int* offsets, int* offsets_out, int S, int E, int* perm, int* inv_perm, int* block_counts,
                               cudaStream_t st) {
  static PerDeviceFlag flag;
  if (!once_per_device(flag, [] {
        return cudaFuncSetAttribute(permute_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024) == cudaSuccess;
      }))
    return MOE_ERR_CUDA;
  const int nblk = (S + kPermuteChunk - 1) / kPermuteChunk;
  const size_t smem = static_cast<size_t>(2 * E + 32) * 4 + static_cast<size_t>(kPermuteChunk / 32) * E * 2;
  const bool scan = nblk > kSortChunks;  // (offsets is there in this case)
  if (launch_pdl(permute_count_kernel, dim3(nblk), dim3(256), E * 4, st, ids, S, E, block_counts) != cudaSuccess ||
      (scan && launch_pdl(permute_scan_kernel, dim3((E + 7) / 8), dim3(256), 0, st, offsets, E, nblk, block_counts) != cudaSuccess))
    return MOE_ERR_CUDA;
  if (scan) offsets = nullptr;
  if (launch_pdl(permute_scatter_kernel, dim3(nblk), dim3(kPermuteChunk), smem, st, ids, S, E, block_counts, offsets, offsets_out, perm, inv_perm) !=
          cudaSuccess)
    return MOE_ERR_CUDA;
  return MOE_OK;
}

int launch_permute(const __nv_bfloat16* x, const int* ids, const int* offsets, const moe_shape_t& sh,
                   __nv_bfloat16* x_perm, int* perm, int* inv_perm, int* block_counts, cudaStream_t st, const int* range_lo,
                   const int* range_hi) {
  const int S = sh.T * sh.k;
  if (S <= permute_direct(x_perm != nullptr, sh.H)) {
    if (launch_pdl(permute_small_kernel<false>, dim3((S + 7) / 8), dim3(256), 0, st, x, ids, const_cast<int*>(offsets), S, sh.H, sh.k, x_perm, perm,
                   inv_perm, range_lo, range_hi, sh.E) != cudaSuccess)
      return MOE_ERR_CUDA;
    note_kernel("permute_rank_by_count", 1);
  } else {
    const int rc = launch_chunked_sort(ids, offsets, nullptr, S, sh.E, perm, inv_perm, block_counts, st);
    if (rc != MOE_OK) return rc;
    if (x_perm != nullptr) {
      const int grid = min((S + 7) / 8, sm_count() * 16);
      if (launch_pdl(permute_gather_kernel, dim3(grid), dim3(256), 0, st, x, perm, S, sh.H, sh.k, x_perm, range_lo, range_hi) !=
          cudaSuccess)
        return MOE_ERR_CUDA;
    }
    note_kernel("permute_chunked_scan", x_perm != nullptr ? 3 : 2);
  }
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

bool route_permute_ok(const moe_shape_t& s) {
  return !route_sort_ok(s.T, s.E) && s.T > 32 && static_cast<long long>(s.T) * s.k <= static_cast<long long>(kSortChunks) * kPermuteChunk;
}
// Routing and sort of a call that makes both, for batches that no cluster routes: the router, then the sort with the offsets as its
// by-product.  The direct count doubles (it counts smaller experts too), so its line lies lower.  Whole layers in a graph, direct / chunked:
// two-term kernel, 256 experts of 256 x 256, top-8: 2072 slots 36.4 us and 39.6, 4096 39.6 and 41.2, 6144 44.7 and 43.5, 8192 59.9 and 54.5; with
// rows, 64 experts of 4096 x 256, top-2: 2072 slots 72.8 and 75.6, 4096 106.0 and 106.6, 6144 136.7 and 135.2.
int launch_route_permute(const float* logits, const __nv_bfloat16* x, const moe_shape_t& sh, int* ids, float* w, int* offsets,
                         __nv_bfloat16* x_perm, int* perm, int* inv_perm, int* block_counts, cudaStream_t st) {
  const int S = sh.T * sh.k;
  if (!route_attr_once()) return MOE_ERR_CUDA;
  int rc = launch_route_ids(logits, sh.T, sh.E, sh.k, ids, w, nullptr, 0, st);
  if (rc != MOE_OK) return rc;
  note_kernel("route_topk_multi_cta", 1);
  if (S <= 4096) {
    if (launch_pdl(permute_small_kernel<true>, dim3((S + 7) / 8 + 1), dim3(256), (static_cast<size_t>(sh.E) + 32) * 4, st, x, ids, offsets, S, sh.H,
                   sh.k, x_perm, perm, inv_perm, static_cast<const int*>(nullptr), static_cast<const int*>(nullptr), sh.E) != cudaSuccess)
      return MOE_ERR_CUDA;
    note_kernel("permute_rank_by_count", 1);
    return MOE_OK;
  }
  if ((rc = launch_chunked_sort(ids, nullptr, offsets, S, sh.E, perm, inv_perm, block_counts, st)) != MOE_OK) return rc;
  note_kernel("permute_chunked_scan", 2);
  return x_perm != nullptr ? launch_gather_rows(x, perm, sh, x_perm, st) : MOE_OK;
}

// =================================================================================================
// moe_combine
// =================================================================================================

// One thread per (token, 8 consecutive columns): k fused multiply-adds per column in slot order.
__global__ void __launch_bounds__(256) combine_kernel(const float* __restrict__ y, const int* __restrict__ inv_perm,
                                                      const float* __restrict__ w, int T, int H, int k,
                                                      __nv_bfloat16* __restrict__ out) {
  const int groups = H / 8;
  const size_t idx = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  pdl_wait();                // the per-slot rows of the expert FFN are complete
  pdl_launch_dependents();   // the next call on the stream (the next layer call's router) may start its set-up
  if (idx >= static_cast<size_t>(T) * groups) return;
  const int t = static_cast<int>(idx / groups);
  const int c = static_cast<int>(idx % groups) * 8;
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
  // slots in groups of four: the four row indices, then the eight row loads, are in flight together; the
  // multiply-adds stay in slot order
  for (int j0 = 0; j0 < k; j0 += 4) {
    int p[4];
    float wj[4];
    float4 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < k) {
        p[u] = __ldg(&inv_perm[static_cast<size_t>(t) * k + j0 + u]);
        wj[u] = __ldg(&w[static_cast<size_t>(t) * k + j0 + u]);
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < k) {
        const float4* src = reinterpret_cast<const float4*>(y + static_cast<size_t>(p[u]) * H + c);
        a[u] = __ldg(src);
        b[u] = __ldg(src + 1);
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < k) {
        acc[0] = __fmaf_rn(wj[u], a[u].x, acc[0]);
        acc[1] = __fmaf_rn(wj[u], a[u].y, acc[1]);
        acc[2] = __fmaf_rn(wj[u], a[u].z, acc[2]);
        acc[3] = __fmaf_rn(wj[u], a[u].w, acc[3]);
        acc[4] = __fmaf_rn(wj[u], b[u].x, acc[4]);
        acc[5] = __fmaf_rn(wj[u], b[u].y, acc[5]);
        acc[6] = __fmaf_rn(wj[u], b[u].z, acc[6]);
        acc[7] = __fmaf_rn(wj[u], b[u].w, acc[7]);
      }
  }
  __nv_bfloat162 o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = __floats2bfloat162_rn(acc[2 * i], acc[2 * i + 1]);
  *reinterpret_cast<uint4*>(out + static_cast<size_t>(t) * H + c) = *reinterpret_cast<uint4*>(o);
}

int launch_combine(const float* y_perm, const int* inv_perm, const float* w, const moe_shape_t& sh,
                   __nv_bfloat16* out, cudaStream_t st) {
  const size_t n = static_cast<size_t>(sh.T) * (sh.H / 8);
  if (launch_pdl(combine_kernel, dim3(static_cast<unsigned>((n + 255) / 256)), dim3(256), 0, st, y_perm, inv_perm, w, sh.T,
                 sh.H, sh.k, out) != cudaSuccess)
    return MOE_ERR_CUDA;
  note_kernel("combine_slot_order_fma", 1);
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

// =================================================================================================
// moe_validate_scales
// =================================================================================================

__global__ void __launch_bounds__(256) validate_scales_kernel(const uint8_t* __restrict__ s, size_t n, int* bad) {
  int c = 0;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x)
    c += (s[i] > 128);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(bad, c);
}

int launch_validate_scales(const uint8_t* scales, size_t n, int* bad, cudaStream_t st) {
  if (cudaMemsetAsync(bad, 0, 4, st) != cudaSuccess) return MOE_ERR_CUDA;
  const int grid = static_cast<int>(min(static_cast<size_t>(sm_count()) * 8, (n + 255) / 256));
  validate_scales_kernel<<<grid > 0 ? grid : 1, 256, 0, st>>>(scales, n, bad);
  note_kernel("validate_scales", 1);
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

}  // namespace moe
