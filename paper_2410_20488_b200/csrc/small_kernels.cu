// Small kernels of the FIRP step: tree bookkeeping and embedding, the acceptance walk / next tree, KV compaction.
#include "finish_device.cuh"
#include "firp_kernels.cuh"
#include "launch_util.cuh"


namespace firp {

// ---------------------------------------------------------------------------
// Everything a step needs before its first layer, one CTA per row:
//   bookkeeping (Section 3.4 "Tree attention"; Section 3.3 for the pseudo rows): depth, absolute position,
//   ancestor-or-self bitmask, rotary table
//   embedding: the fp32 residual row of a tree row from the bf16 table, and what the first layer reads of it
// Latency-bound; rows are independent once each CTA has the parents of its sequence in shared memory.
// ---------------------------------------------------------------------------
constexpr int kPrepThreads = 128;

__global__ void __launch_bounds__(kPrepThreads) prep_kernel(PrepArgs a, int pdl) {
  __shared__ int32_t ext[kMaxTreeRows];
  __shared__ int s_depth;
  if (pdl) { griddep_launch(); griddep_wait(); }
  const Rows &rw = a.rw;
  const int r = blockIdx.x, s = r / rw.Ms, v = r - s * rw.Ms, ar = act_row(rw, s, v), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (a.zero_word && r == 0 && tid == 0) *a.zero_word = 0u;
  if (rw.by_step && tid == 0) a.meta.row_of[ar] = seq_row(s, v);
  const int n = a.ctx_len[a.seq_ids[s]];
  if (v == 0 && tid == 0) a.meta.n0[s] = n;
  for (int u = tid; u <= v && !rw.prompt; u += kPrepThreads) {
    int p;
    if (u < rw.T) p = a.parents[s * a.parents_stride + u];
    else if (rw.chains) p = u - rw.T;   // step 1 of node w (row T + w) hangs off w, step i off step i-1 of the same node
    else p = (u == rw.T) ? rw.anchor : u - 1;
    ext[u] = p;
  }
  __syncthreads();
  if (rw.prompt) {                      // a chain: the row index is the depth, and says who sees whom
    if (tid == 0) { s_depth = v; a.meta.pos[r] = n + v; }
  } else if (tid == kPrepThreads - 1) { // the last warp: the rotary table below is the first ones'
    uint32_t bits[kMaskWords];
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) bits[w] = 0u;
    int dep = -1;
    int u = v;
    for (int it = 0; it < rw.Ms && u >= 0; ++it) {   // parents[u] < u, so at most Ms hops
      if (!(rw.masked && u >= rw.T && u != v)) {     // "Masked": other pseudo rows stay invisible, depth still counts them
#pragma unroll
        for (int w = 0; w < kMaskWords; ++w) if ((u >> 5) == w) bits[w] |= 1u << (u & 31);
      }
      ++dep;
      u = ext[u];
    }
    s_depth = dep;
    a.meta.depth[r] = dep;
    a.meta.pos[r] = n + dep;
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) a.meta.mask[(size_t)r * kMaskWords + w] = bits[w];
    if (a.out_depth) a.out_depth[r] = dep;
    if (a.out_mask)
      for (int w = 0; w < a.out_mask_words; ++w) a.out_mask[(size_t)r * a.out_mask_words + w] = bits[w];
  }
  if (v < rw.T) {                       // pseudo rows get their residual from Eq. 3
    const int tok = min(max(a.tokens[s * rw.T + v], 0), a.vocab - 1);
    const int xp_row = a.xp == nullptr ? -1 : rw.chains ? s * rw.T + v : v == rw.anchor ? s : -1;
    for (int c = warp * 128 + lane * 4; c < a.d; c += kPrepThreads * 4)
    {
      const float4 e = load_bf16x4(a.embed + (size_t)tok * a.d + c);
      store_residual(a, ar, xp_row, c, e, a.x ? load_bf16x4(a.g + c) : e, warp_sq(e), lane);
    }
  }
  __syncthreads();
  const int half = a.dh / 2;
  const double l2t = log2((double)a.theta);
  if (tid < half) {
    const double inv_freq = exp2(-2.0 * (double)tid / (double)a.dh * l2t);
    const double ang = (double)(n + s_depth) * inv_freq;
    double sn, cs;
    sincos(ang, &sn, &cs);
    a.meta.rope[(size_t)ar * half + tid] = make_float2((float)cs, (float)sn);
  }
}

void launch_prep(const PrepArgs &a, bool pdl, cudaStream_t st) {
  launch_k(prep_kernel, dim3(a.rw.R), dim3(kPrepThreads), 0, st, pdl, a, pdl ? 1 : 0);
}

// ---------------------------------------------------------------------------
// Greedy acceptance walk and next tree (Section 3.4).  One CTA per sequence.  Bound by its chains of dependent loads, so the
// trees are brought into shared memory first and a warp looks at 32 children at a time (one thread on global memory:
// 39 us after a step with 128 tree rows, now 9; the two-layer shape's round of 8 rows 92.2 -> 89.2 us).
// ---------------------------------------------------------------------------
__global__ void accept_kernel(Rows rw, AcceptArgs a, int pdl) {
  __shared__ int32_t s_best[kMaxTreeRows], tok[kMaxTreeRows], parents[kMaxTreeRows], next_parents[kMaxTreeRows];
  __shared__ int32_t s_bonus, s_end;
  if (pdl) { griddep_launch(); griddep_wait(); }
  const int s = blockIdx.x, tid = threadIdx.x;
  // own tree of the sequence (rows beyond its size are padding and can neither be accepted nor take a candidate)
  const int Ts = a.sizes ? min(a.sizes[s], rw.T) : rw.T, Tn = a.sizes ? min(a.sizes[s], a.T_next) : a.T_next;
  for (int v = tid; v < rw.T; v += blockDim.x) {
    const int32_t b = a.top_ids[(size_t)(s * rw.Ms + v) * a.B];
    s_best[v] = b;
    tok[v] = a.tokens[(size_t)s * rw.T + v];
    parents[v] = a.parents[(size_t)s * a.parents_stride + v];
    if (a.o_best) a.o_best[(size_t)s * rw.T + v] = b;
  }
  for (int v = tid; v < a.T_next; v += blockDim.x) next_parents[v] = a.next_parents[(size_t)s * a.parents_stride + v];
  __syncthreads();
  if (tid < 32) {
    int32_t *path = a.path + (size_t)s * a.S, *acc = a.accepted + (size_t)s * a.S;
    int cur = 0, na = 0;
    if (tid == 0) path[0] = 0;
    if (a.prefill_last_row >= 0) {
      cur = a.prefill_last_row;
    } else {
      while (na + 1 < a.S) {
        int next = -1;
        for (int c0 = cur + 1; c0 < Ts && next < 0; c0 += 32) {
          const int ch = c0 + tid;
          const uint32_t hit = __ballot_sync(0xffffffffu, ch < Ts && parents[ch] == cur && tok[ch] == s_best[cur]);
          if (hit) next = c0 + __ffs((int)hit) - 1;
        }
        if (next < 0) break;
        if (tid == 0) {
          acc[na] = tok[next];
          path[na + 1] = next;
          if (a.o_accepted) a.o_accepted[(size_t)s * a.S + na] = tok[next];
          if (a.o_path) a.o_path[(size_t)s * a.S + na + 1] = next;
        }
        ++na;
        cur = next;
      }
    }
    if (tid == 0) {
      acc[na] = s_best[cur];
      s_bonus = s_best[cur];
      s_end = cur;
      a.n_accepted[s] = na + 1;
      if (a.o_n_accepted) a.o_n_accepted[s] = na + 1;
      if (a.o_path) a.o_path[(size_t)s * a.S] = 0;
      if (a.o_accepted) a.o_accepted[(size_t)s * a.S + na] = s_best[cur];
    }
  }
  __syncthreads();
  // the pseudo row that holds the candidates of depth j (1-based): row j of the one chain, or of the chain
  // under the node the walk ended on
  const int steps = rw.chains ? rw.kc : rw.k;
  const size_t row0 = (size_t)s * rw.Ms + rw.T + (rw.chains ? s_end : 0);
  const int row_step = rw.chains ? rw.T : 1;
  if (a.o_topb_ids || a.o_topb_vals) {
    for (int i = tid; i < steps * a.B; i += blockDim.x) {
      const size_t src = (row0 + (size_t)(i / a.B) * row_step) * a.B + i % a.B;
      if (a.o_topb_ids) a.o_topb_ids[(size_t)s * steps * a.B + i] = a.top_ids[src];
      if (a.o_topb_vals) a.o_topb_vals[(size_t)s * steps * a.B + i] = a.top_vals[src];
    }
  }
  for (int v = tid; v < a.T_next; v += blockDim.x) {
    int32_t t;
    if (v == 0 || v >= Tn) {
      t = s_bonus;
    } else {
      int dep = 0;
      for (int u = v; u > 0 && dep <= a.T_next; u = next_parents[u]) ++dep;
      int rank = 0;
      for (int u = 1; u < v; ++u) rank += (next_parents[u] == next_parents[v]);
      dep = min(dep, max(steps, 1));
      rank = min(rank, a.B - 1);
      t = (steps > 0) ? a.top_ids[(row0 + (size_t)(dep - 1) * row_step) * a.B + rank] : s_bonus;
    }
    a.next_tokens[(size_t)s * a.T_next + v] = t;
    if (a.o_next_tokens) a.o_next_tokens[(size_t)s * a.T_next + v] = t;
  }
}

void launch_accept(const Rows &rw, const AcceptArgs &a, bool pdl, cudaStream_t st) {
  launch_k(accept_kernel, dim3(rw.n_seq), dim3(128), 0, st, pdl, rw, a, pdl ? 1 : 0);
}

// ---------------------------------------------------------------------------
// KV compaction of the accepted path.  Each thread owns one 16-byte column slice of a
// (layer, K|V) plane and moves it for every path entry: it loads all source rows before
// storing any, so a destination slot that is another entry's source is never clobbered.
// One block moves the context length on; all take it from the step's bookkeeping, at a place that does not hang on the step's sizes, so
// that a captured commit serves steps of any (a kernel of its own for the length: 3 us of the host and 2 of the two-layer shape's round,
// 78.2 -> 76.2 us).
// ---------------------------------------------------------------------------
constexpr int kMaxPath = 16;

__global__ void __launch_bounds__(128) commit_kernel(CommitArgs a, int pdl) {
  if (pdl) { griddep_launch(); griddep_wait(); }
  const int s = blockIdx.y, plane = blockIdx.x;     // plane = layer * 2 + (0 K, 1 V)
  const int slot = a.seq_ids[s];
  const int n = a.n0[s];                            // not from ctx_len, which one block writes below while others start
  const int len = min(a.path_len[s], kMaxPath);
  if (plane == 0 && threadIdx.x == 0) a.ctx_len[slot] = n + len;
  const int32_t *path = a.path + (size_t)s * a.S;
  bf16 *base = a.kv + (size_t)(plane >> 1) * a.layer_stride + (size_t)(plane & 1) * a.kv_stride;
  const int nvec = a.nkv >> 3;
  size_t src_row[kMaxPath], dst_row[kMaxPath];
#pragma unroll
  for (int j = 0; j < kMaxPath; ++j) {
    if (j < len) { src_row[j] = kv_row(a.pages, slot, n + path[j], a.max_ctx); dst_row[j] = kv_row(a.pages, slot, n + j, a.max_ctx); }
  }
  for (int c = threadIdx.x; c < nvec; c += blockDim.x) {
    uint4 tmp[kMaxPath];
#pragma unroll
    for (int j = 0; j < kMaxPath; ++j)
      if (j < len) tmp[j] = reinterpret_cast<const uint4 *>(base + src_row[j] * a.nkv)[c];
#pragma unroll
    for (int j = 0; j < kMaxPath; ++j)
      if (j < len && path[j] != j) reinterpret_cast<uint4 *>(base + dst_row[j] * a.nkv)[c] = tmp[j];
  }
}

__global__ void advance_ctx_kernel(int n_seq, const int32_t *seq_ids, int32_t *ctx_len, int amount, int pdl) {
  if (pdl) { griddep_launch(); griddep_wait(); }
  const int s = threadIdx.x;
  if (s < n_seq) ctx_len[seq_ids[s]] += amount;
}

void launch_commit(int n_seq, const CommitArgs &a, bool pdl, cudaStream_t st) {
  launch_k(commit_kernel, dim3(a.n_layers * 2, n_seq), dim3(128), 0, st, pdl, a, pdl ? 1 : 0);
}

void launch_advance_ctx(int n_seq, const int32_t *seq_ids, int32_t *ctx_len, int amount, bool pdl, cudaStream_t st) {
  launch_k(advance_ctx_kernel, dim3(1), dim3(32), 0, st, pdl, n_seq, seq_ids, ctx_len, amount, pdl ? 1 : 0);
}

}  // namespace firp
