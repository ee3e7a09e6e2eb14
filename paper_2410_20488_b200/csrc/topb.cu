// Top-B of logits rows by (value descending, id ascending), one launch (Section 4: greedy tokens and candidates).
//
// A row is shared by a cluster of up to 8 CTAs, 4096 logits each per pass.  A logit becomes a 64-bit key (value in an
// order-preserving integer form, complement of the id), so that the order of keys is the order wanted and keys are
// unique.  Selection is by threshold: the B-th best of a warp's 32 per-thread maxima has at least B logits at or
// above it, so the largest such value of a CTA bounds the row's B-th best from below; only the logits at or above it
// (a dozen of 4096 on ordinary rows, at most 64 per warp on any) go to a list in shared memory, and an entry's place is the
// number of entries above it.  The CTAs' B best meet in the first CTA of the cluster the same way.
//
// Bound: latency (35 x 32000 logits are 4.5 MB, 0.7 us of HBM).  Measured per call, back to back, against two launches
// with a sorted 8-entry list per thread and three block barriers per selected entry: 35 x 32000, b = 8: 22.5 -> 14.3 us;
// 1 x 50257, b = 5: 14.3 -> 10.2 us.
#include <cooperative_groups.h>

#include "firp_kernels.cuh"
#include "launch_util.cuh"

namespace cg = cooperative_groups;

namespace firp {

namespace {

typedef unsigned long long u64;

constexpr int kTopThreads = 512, kTopWarps = kTopThreads / 32;
constexpr int kTopEpt = 8;                                // logits of a thread per pass
constexpr int kTopChunk = kTopThreads * kTopEpt;          // logits of a CTA per pass
constexpr int kTopCluster = 8;                            // portable cluster size limit
// at most B of a warp's lanes have a maximum at or above the warp's own threshold, and each of those holds kTopEpt logits
constexpr int kTopList = kTopWarps * kMaxTopB * kTopEpt + kMaxTopB;

// order-preserving: greater float <=> greater integer, -0 = +0; 0 for NaN, which is never selected
__device__ __forceinline__ uint32_t order_key(float v) {
  if (v != v) return 0u;
  const uint32_t b = __float_as_uint(v + 0.f);
  return b ^ (((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float order_value(uint32_t k) {
  return __uint_as_float(k & 0x80000000u ? k ^ 0x80000000u : ~k);
}

// entries of list[0, n) into best[0, B) by rank (keys are unique; 0 marks an empty entry)
__device__ __forceinline__ void rank_list(const u64 *list, int n, int B, u64 *best) {
  for (int i = threadIdx.x; i < n; i += kTopThreads) {
    const u64 k = list[i];
    int rank = 0;
    for (int j = 0; j < n && rank < B; ++j) rank += list[j] > k;
    if (k != 0 && rank < B) best[rank] = k;
  }
}

__global__ void __launch_bounds__(kTopThreads)
topb_kernel(const float *__restrict__ vals, int V, int B, int32_t *out_ids, float *out_vals, int pdl) {
  __shared__ u64 s_list[kTopList];
  __shared__ u64 s_best[kMaxTopB], s_all[kTopCluster * kMaxTopB], s_thr;
  __shared__ int s_n;
  if (pdl) { griddep_launch(); griddep_wait(); }
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), nc = (int)cluster.num_blocks();
  if (nc > 1) cluster.barrier_arrive();
  const int tid = threadIdx.x, lane = tid & 31;
  const float *row = vals + (size_t)blockIdx.y * V;
  if (tid < kMaxTopB) s_best[tid] = 0;
  if (tid == 0) { s_thr = 0; s_n = 0; }
  const int per_pass = nc * kTopChunk, passes = (V + per_pass - 1) / per_pass;
  for (int p = 0; p < passes; ++p) {
    const int base = p * per_pass + rank * kTopChunk + tid;
    float f[kTopEpt];
#pragma unroll
    for (int e = 0; e < kTopEpt; ++e) {
      const int id = base + e * kTopThreads;
      f[e] = (id < V && id >= 0) ? __ldg(row + id) : __int_as_float(0x7fffffff);   // beyond the row: NaN
    }
    uint32_t k[kTopEpt], mh = 0, ml = 0;
#pragma unroll
    for (int e = 0; e < kTopEpt; ++e) {
      k[e] = order_key(f[e]);
      if (k[e] > mh) { mh = k[e]; ml = ~(uint32_t)(base + e * kTopThreads); }      // the first of equals has the lowest id
    }
    uint32_t th = 0, tl = 0;
    for (int b = 0; b < B; ++b) {          // the B-th best of the lanes' maxima
      th = __reduce_max_sync(0xffffffffu, mh);
      tl = __reduce_max_sync(0xffffffffu, mh == th ? ml : 0u);
      if (mh == th && ml == tl) { mh = 0; ml = 0; }
    }
    __syncthreads();                       // s_thr, s_n are set
    if (lane == 0) atomicMax(&s_thr, ((u64)th << 32) | tl);
    __syncthreads();
    const u64 thr = s_thr;
#pragma unroll
    for (int e = 0; e < kTopEpt; ++e) {
      const u64 key = ((u64)k[e] << 32) | ~(uint32_t)(base + e * kTopThreads);
      if (k[e] != 0 && key >= thr) s_list[atomicAdd(&s_n, 1)] = key;
    }
    __syncthreads();
    const int n = s_n;
    rank_list(s_list, n, B, s_best);
    __syncthreads();
    if (p + 1 < passes) {                  // carried into the next pass: the best so far, and the bound they give
      if (tid < min(n, B)) s_list[tid] = s_best[tid];
      if (tid == 0) { s_n = min(n, B); s_thr = n >= B ? s_best[B - 1] : 0; }
    }
  }
  const u64 *list = s_best;
  int n = B;
  if (nc > 1) {
    cluster.barrier_wait();                // every CTA of the cluster has started: its shared memory can be written
    if (tid < B) cluster.map_shared_rank(s_all, 0)[rank * B + tid] = s_best[tid];
    cluster.sync();
    if (rank != 0) return;
    if (tid < kMaxTopB) s_best[tid] = 0;
    __syncthreads();
    rank_list(s_all, nc * B, B, s_best);
    __syncthreads();
  }
  if (tid < n) {
    const u64 key = list[tid];
    const int id = key ? (int)~(uint32_t)key : 0x7fffffff;
    float v = key ? order_value((uint32_t)(key >> 32)) : -INFINITY;
    if (v == 0.f) v = row[id];             // the sign of a zero is not in the key
    out_ids[(size_t)blockIdx.y * B + tid] = id;
    out_vals[(size_t)blockIdx.y * B + tid] = v;
  }
}

}  // namespace

void launch_topb(const float *logits, int R, int V, int B, int32_t *ids, float *vals, bool pdl, cudaStream_t st) {
  // one pass for rows of up to 8 x 4096 logits
  const int nc = V >= kTopCluster * kTopChunk ? kTopCluster : (V + kTopChunk - 1) / kTopChunk;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nc, R);
  cfg.blockDim = dim3(kTopThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = nc; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  cudaLaunchKernelEx(&cfg, topb_kernel, logits, V, B, ids, vals, pdl ? 1 : 0);
}

}  // namespace firp
