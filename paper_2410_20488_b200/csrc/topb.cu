// Top-B of logits rows by (value descending, id ascending), one launch (Section 4: greedy tokens and candidates).
//
// A row of up to 32768 logits belongs to one CTA of 1024 threads, 32 logits in registers each; a longer one, or one of few rows, to
// a cluster of up to 8.  A logit becomes a 64-bit key (value in an order-preserving integer form, complement of the id), so that the order of keys
// is the order wanted and keys are unique.  Selection is by threshold: the B-th best of the 32 warps' maxima has at least B
// logits at or above it; only the logits at or above it (a dozen on ordinary rows) go to a list in shared memory, and an
// entry's place is the number of entries above it.  Rows on which the list overflows (sorted ones: neighbours in few warps)
// use the B-th best of the 1024 threads' maxima instead, with at most 32 B logits at or above it.  The CTAs' B best meet in the
// first CTA of the cluster the same way.
//
// Bound: latency (35 x 32000 logits are 4.5 MB, 0.7 us of HBM).  Measured per call, back to back, against a cluster of 8 CTAs
// per row with a threshold per warp, whose barriers and longer lists cost more than the eight times wider load saved:
// 35 x 32000, b = 8: 13.8 -> 9.6 us (22.5 with two launches and a sorted list per thread); on another box 7.2, of which the host needs 3.6 to issue it;
// 131 x 32000 in a step 29 -> 13 us.
#include <cooperative_groups.h>

#include "firp_kernels.cuh"
#include "launch_util.cuh"

namespace cg = cooperative_groups;

namespace firp {

namespace {

typedef unsigned long long u64;

constexpr int kTopWarps = 32;                             // of the largest CTA
constexpr int kTopCluster = 8;                            // portable cluster size limit
constexpr int kTopFill = 74;                              // CTAs: half of a B200's SMs
constexpr int kTopList = 1024;                            // entries, and kMaxTopB carried ones
static_assert(kTopList >= kMaxTopB * 32, "the list holds what the threads' threshold lets through");

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
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const u64 k = list[i];
    int rank = 0;
#pragma unroll 8
    for (int j = 0; j < n; ++j) rank += list[j] > k;
    if (k != 0 && rank < B) best[rank] = k;
  }
}

// the B-th best of a warp's 32 keys (hi, lo), 0 if there are fewer
__device__ __forceinline__ u64 warp_bth(uint32_t hi, uint32_t lo, int B) {
  uint32_t th = 0, tl = 0;
  for (int b = 0; b < B; ++b) {
    th = __reduce_max_sync(0xffffffffu, hi);
    tl = __reduce_max_sync(0xffffffffu, hi == th ? lo : 0u);
    if (hi == th && lo == tl) { hi = 0; lo = 0; }
  }
  return th ? ((u64)th << 32) | tl : 0;
}

// EPT: logits of a thread per pass.  VEC: four neighbouring logits per load (rows start on 16-byte boundaries).  The kernel is
// launched beside the one that writes the logits: they are read through L2, never through the read-only path, whose data must
// not change while a kernel lives.
template <int EPT, bool VEC>
__global__ void __launch_bounds__(32 * kTopWarps)
topb_kernel(const float *vals, int V, int B, int32_t *out_ids, float *out_vals, int pdl) {
  __shared__ u64 s_list[kTopList + kMaxTopB], s_max[kTopWarps];
  __shared__ u64 s_best[kMaxTopB], s_all[kTopCluster * kMaxTopB];
  __shared__ int s_n;
  if (pdl) { griddep_launch(); griddep_wait(); }
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), nc = (int)cluster.num_blocks();
  if (nc > 1) cluster.barrier_arrive();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float *row = vals + (size_t)blockIdx.y * V;
  if (tid < kMaxTopB) s_best[tid] = 0;
  if (tid == 0) s_n = 0;
  const int threads = blockDim.x, chunk = threads * EPT, per_pass = nc * chunk, passes = (V + per_pass - 1) / per_pass;
  u64 bound = 0;                           // of the passes so far
  for (int p = 0; p < passes; ++p) {
    const int base = p * per_pass + rank * chunk;
    // ids of a thread ascend with e
    auto id_of = [&](int e) { return base + (VEC ? (e >> 2) * 4 * threads + tid * 4 + (e & 3) : e * threads + tid); };
    uint32_t k[EPT], mh = 0, ml = 0;
#pragma unroll
    for (int e = 0; e < EPT; e += VEC ? 4 : 1) {
      const int id = id_of(e);
      const bool in = id < V && id >= 0;
      if (VEC) {
        const float4 f = in ? __ldcg(reinterpret_cast<const float4 *>(row + id)) : make_float4(0.f, 0.f, 0.f, 0.f);
        k[e] = in ? order_key(f.x) : 0u; k[e + (VEC ? 1 : 0)] = in ? order_key(f.y) : 0u;
        k[e + (VEC ? 2 : 0)] = in ? order_key(f.z) : 0u; k[e + (VEC ? 3 : 0)] = in ? order_key(f.w) : 0u;
      } else {
        k[e] = in ? order_key(__ldcg(row + id)) : 0u;
      }
    }
#pragma unroll
    for (int e = 0; e < EPT; ++e)
      if (k[e] > mh) { mh = k[e]; ml = ~(uint32_t)id_of(e); }      // the first of equals has the lowest id
    const uint32_t wh = __reduce_max_sync(0xffffffffu, mh), wl = __reduce_max_sync(0xffffffffu, mh == wh ? ml : 0u);
    if (lane == 0) s_max[warp] = ((u64)wh << 32) | wl;
    __syncthreads();                       // (s_n and the carried entries are set, too)
    u64 thr = lane < threads >> 5 ? s_max[lane] : 0;
    thr = warp_bth((uint32_t)(thr >> 32), (uint32_t)thr, B);
    if (thr < bound) thr = bound;
    const int carried = s_n;
    __syncthreads();
    auto push = [&]() {
#pragma unroll
      for (int e = 0; e < EPT; ++e) {
        const u64 key = ((u64)k[e] << 32) | ~(uint32_t)id_of(e);
        if (k[e] != 0 && key >= thr) {
          const int at = atomicAdd(&s_n, 1);
          if (at < kTopList) s_list[at] = key;
        }
      }
    };
    push();
    __syncthreads();
    if (s_n > kTopList) {                  // the same in every thread
      for (int b = 0; b < B; ++b) {
        const uint32_t h = __reduce_max_sync(0xffffffffu, mh), l = __reduce_max_sync(0xffffffffu, mh == h ? ml : 0u);
        if (lane == 0) s_max[warp] = ((u64)h << 32) | l;
        __syncthreads();
        const u64 m = lane < threads >> 5 ? s_max[lane] : 0;
        thr = warp_bth((uint32_t)(m >> 32), (uint32_t)m, 1);
        if (thr && mh == (uint32_t)(thr >> 32) && ml == (uint32_t)thr) { mh = 0; ml = 0; }
        __syncthreads();
      }
      if (thr < bound) thr = bound;
      if (tid == 0) s_n = carried;
      __syncthreads();
      push();
      __syncthreads();
    }
    const int n = s_n;
    rank_list(s_list, n, B, s_best);
    __syncthreads();
    if (p + 1 < passes) {                  // carried into the next pass: the best so far, and the bound they give
      if (tid < min(n, B)) s_list[tid] = s_best[tid];
      if (tid == 0) s_n = min(n, B);
      if (n >= B) bound = s_best[B - 1];
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
    if (v == 0.f) v = __ldcg(row + id);             // the sign of a zero is not in the key
    out_ids[(size_t)blockIdx.y * B + tid] = id;
    out_vals[(size_t)blockIdx.y * B + tid] = v;
  }
}

}  // namespace

void launch_topb(const float *logits, int R, int V, int B, int32_t *ids, float *vals, bool pdl, cudaStream_t st) {
  // 32 logits per thread keep a row in one CTA up to 32768 of them, which is best once the rows alone fill half the chip.  Few
  // rows are cut into shares of 8192, and rows below that use CTAs of 4 logits per thread: 1 x 50257 in
  // shares of 8192 / 32768 9.4 / 11.4 us, the round of the two-layer shape (11 x 1024) with 256 / 1024 threads 86.0 / 90.6 us,
  // 35 x 32000 alike either way, 9.6 us (one box; on another 1 x 50257 takes 6.0 us, 35 x 32000 7.2, and the host 3.6 for any call).
  const int nc8 = (V + 8191) / 8192;
  const bool wide = nc8 > 1 && (nc8 > kTopCluster || (long long)R * nc8 > kTopFill);
  const int chunk = wide ? 32768 : 8192;
  const int nc = V > (kTopCluster - 1) * chunk ? kTopCluster : (V + chunk - 1) / chunk;
  const int threads = V >= 4096 ? 1024 : V <= 1024 ? 256 : ((V + 3) / 4 + 31) / 32 * 32;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nc, R);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (pdl) { attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization; attr[na++].val.programmaticStreamSerializationAllowed = 1; }
  if (nc > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = nc; attr[na].val.clusterDim.y = 1; attr[na].val.clusterDim.z = 1; ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  const bool vec = (V & 3) == 0 && (reinterpret_cast<uintptr_t>(logits) & 15) == 0;
  cudaLaunchKernelEx(&cfg, wide ? (vec ? topb_kernel<32, true> : topb_kernel<32, false>) : vec ? topb_kernel<8, true> : topb_kernel<8, false>, logits, V, B, ids, vals, pdl ? 1 : 0);
}

}  // namespace firp
