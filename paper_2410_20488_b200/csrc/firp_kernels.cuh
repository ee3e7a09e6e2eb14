// Internal launcher interface between the step scheduler and the sm_100a kernels.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_plan.h"
#include "rows.h"

namespace firp {

typedef __nv_bfloat16 bf16;

constexpr int kMaskWords = 5;      // ceil(136 / 32)
constexpr int kMaxTopB = 8;
constexpr int kAttnTile = 64;      // kv positions per attention tile

// Rows of the KV cache.  A (layer, K|V) plane holds max_batch * max_ctx rows of Hkv * dh elements.  Without a
// page table position `pos` of slot `slot` is row slot * max_ctx + pos; with one (pages of kKvPage positions,
// table[slot * pages_per_seq + pos / kKvPage] = physical page) it is row page * kKvPage + pos % kKvPage.
constexpr int kKvPage = 64;               // = kAttnTile: an attention tile never straddles two pages
struct KvPages { const int32_t *table; int pages_per_seq; };
__device__ __forceinline__ size_t kv_row(const KvPages &pg, int slot, int pos, int max_ctx) {
  if (pg.table == nullptr) return (size_t)slot * max_ctx + pos;
  return (size_t)pg.table[slot * pg.pages_per_seq + pos / kKvPage] * kKvPage + (pos % kKvPage);
}

constexpr int kGemmMaxCtas = 192;         // scratch slots are provided for this many CTAs
constexpr int kGemmSlots = 3;             // partial tiles (segments) per CTA

// Stream-K schedule of one GEMM launch.  Unit u = supertile * KB + k block (supertile = 256 weight
// rows, k block = 64 elements); CTA c owns units [sk_begin(c), sk_begin(c + 1)) and its s-th segment
// is the part of supertile sk_begin(c) / KB + s inside that range.
struct StreamK {
  int U;        // units (supertiles x k blocks; U * G stays far below 2^31 for every supported shape)
  int KB;       // k blocks per supertile
  int G;        // CTAs (<= U, so no range is empty)
};
__host__ __device__ __forceinline__ int sk_begin(const StreamK &s, int c) { return (int)(((unsigned)s.U * (unsigned)c) / (unsigned)s.G); }
// CTA whose range holds unit u: the largest c with floor(U c / G) <= u, i.e. c < (u + 1) G / U
__host__ __device__ __forceinline__ int sk_owner(const StreamK &s, int u) {
  return (int)((((unsigned)u + 1u) * (unsigned)s.G + (unsigned)s.U - 1u) / (unsigned)s.U) - 1;
}
// The CTAs c_first..c_last that hold a piece of supertile st.  Every one but the first starts its range
// inside st, so its piece is its segment 0; the first one's piece is segment ord_first.
struct SkContrib { int c_first, c_last, ord_first; };
__host__ __device__ __forceinline__ SkContrib sk_contributors(const StreamK &s, int st) {
  SkContrib k;
  k.c_first = sk_owner(s, st * s.KB);
  k.c_last = sk_owner(s, (st + 1) * s.KB - 1);
  k.ord_first = st - sk_begin(s, k.c_first) / s.KB;
  return k;
}

// ---- tree bookkeeping (Section 3.4) ---------------------------------------
struct TreeMeta {
  int32_t *depth;      // [R]
  int32_t *pos;        // [R] absolute position = ctx_len + depth
  uint32_t *mask;      // [R][kMaskWords] bit u: row v attends to new row u of its sequence
  float2 *rope;        // [R][dh/2] (cos, sin) of pos * theta^(-2c/dh), by row of the activations
  uint16_t *row_of;    // [R] seq_row of each row of the activations
  int32_t *n0;         // [n_seq] committed length of each sequence when the step began
};
struct PrepArgs {
  Rows rw;
  const int32_t *parents; int parents_stride;     // [T] shared by the sequences (stride 0) or [n_seq][T] (stride T)
  const int32_t *seq_ids, *ctx_len;
  int dh; float theta;
  TreeMeta meta;
  int32_t *out_depth; uint32_t *out_mask; int out_mask_words;     // caller's copies or NULL
  unsigned *zero_word;                            // a device word to clear (the arrival counter of the persistent kernel)
  const int32_t *tokens; const bf16 *embed; int d, vocab;
  float *h;
  // operand of the first layer's QKV projection: x = h * g as bf16 planes and the sums of squares (x == NULL: not wanted),
  // and, if that layer inserts pseudo rows, the rows Eq. 3 reads (xp, as in LinArgs)
  const bf16 *g; bf16 *x; size_t x_plane; int x_planes; float *ss_out;
  bf16 *xp; size_t xp_plane; int xp_normed;
};
// The step's bookkeeping (Section 3.4 "Tree attention") and h[r] = embed[token] of the tree rows.
void launch_prep(const PrepArgs &a, bool pdl, cudaStream_t st);

// Activations that feed a GEMM or the attention are stored as two bf16 planes (hi, lo) with
// hi + lo = the fp32 value to ~16 mantissa bits; the lo plane starts *_lo_off elements after hi.

// Partial tiles a stream-K GEMM left in scratch: slot (c, s) = segment s of CTA c, laid out
// [2 tiles][ws_rows token rows][128 lanes] fp32; whoever consumes the GEMM sums them in CTA order.
struct Partials {
  StreamK sk;        // schedule of the GEMM that wrote the tiles (U = 0: nothing pending)
  const float *ws;   // its scratch slots
  int ws_rows;       // token rows per scratch tile
};
constexpr int kNormMaxWarps = 64;   // sums of squares per row, one for 128 columns (d <= 8192)

// top-B (B <= kMaxTopB) of every row of logits by (value desc, id asc) into ids, vals [R][B]; a row with fewer than B
// numbers is padded with (-inf, INT_MAX)
void launch_topb(const float *logits, int R, int V, int B, int32_t *ids, float *vals, bool pdl, cudaStream_t st);

struct AcceptArgs {
  const int32_t *tokens;        // [n_seq][T]
  const int32_t *parents;       // [T], or [n_seq][T] with parents_stride = T
  const int32_t *next_parents;  // [T_next], likewise
  int parents_stride;           // 0: one template for every sequence
  const int32_t *sizes;         // NULL, or [n_seq]: nodes of each sequence's own tree (the rest of its T rows is padding)
  const int32_t *top_ids;       // [R][B] (row r's candidates; [0] is the argmax)
  const float *top_vals;        // [R][B]
  int T_next, B, S;             // S = path stride
  int prefill_last_row;         // >= 0: prefill mode, the root is the argmax of this row; -1: verify walk
  int32_t *path, *n_accepted, *accepted;  // internal copies [n_seq][S], [n_seq], [n_seq][S]
  int32_t *next_tokens;                   // [n_seq][T_next]
  // optional caller buffers (may be NULL)
  int32_t *o_path, *o_n_accepted, *o_accepted, *o_next_tokens, *o_best, *o_topb_ids;
  float *o_topb_vals;
};
void launch_accept(const Rows &rw, const AcceptArgs &a, bool pdl, cudaStream_t st);

// KV compaction: rows path[j] -> slot n + j in every layer; ctx_len = n + len
struct CommitArgs {
  bf16 *kv;                 // cache base
  size_t seq_stride;        // elements per sequence
  size_t layer_stride;      // elements per layer (2 * max_ctx * nkv)
  size_t kv_stride;         // elements per K or V plane (max_ctx * nkv)
  int n_layers, nkv;        // nkv = Hkv * dh
  const int32_t *seq_ids;   // [n_seq] device
  const int32_t *path;      // [n_seq][S] device
  const int32_t *path_len;  // [n_seq] device
  int S;
  int32_t *ctx_len;         // [max_batch] device
  const int32_t *n0;        // [n_seq] device: n, the committed lengths of the step
  int max_ctx; KvPages pages;
};
void launch_commit(int n_seq, const CommitArgs &a, bool pdl, cudaStream_t st);
void launch_advance_ctx(int n_seq, const int32_t *seq_ids, int32_t *ctx_len, int amount, bool pdl, cudaStream_t st);   // after a stretch of a prompt

// ---- weight-streaming GEMM ---------------------------------------------------
// One GEMM of the kernel-per-operation mode: out[m][n] = sum_k X[m][k] W[n][k] and the elementwise step behind it.
struct LinArgs {
  const bf16 *X;    // [planes][plane_rows][K] activations as bf16 planes
  int plane_rows, planes;
  const bf16 *W;    // [N][K] weights
  int R, N, K;      // token rows (<= kMaxPromptRows): the first R of the activations
  int call_rows;    // rows of the call's last layers, where all pseudo rows are in: they set how long the sums may be (gemm_plan.h)
  Rows rw;
  const uint16_t *row_of;       // seq_row of every row of the activations; NULL: one sequence, row v is row v
  int *err;         // device status word (set to a non-zero code if a bounded wait gives up)
  unsigned long long wait_ns;   // bounded waits give up after this many nanoseconds (0: the default of 2 s)
  // X holds h * g, not yet divided by the RMS: row m of the result is scaled by 1 / sqrt(sum_w ss[m][w] / K + eps)
  // (ss == NULL: X is used as it is)
  const float *ss; float eps;
  // EPI_RESIDUAL, EPI_PSEUDO: rows of the residual stream h [R][d].  x (NULL: nothing reads it) gets h * g as x_planes
  // bf16 planes, ss_out[row][c / 128] the sums of squares; xp (NULL: the next layer inserts no pseudo rows) the rows
  // Eq. 3 reads there, raw or (xp_normed) as h * g: every sequence's anchor, or all its tree rows when every node
  // carries a chain.
  float *h; int d;
  const bf16 *g; bf16 *x; size_t x_plane; int x_planes; float *ss_out;
  bf16 *xp; size_t xp_plane; int xp_normed;
  // EPI_PSEUDO (Eq. 3): output n = i * d + o of map pseudo0 + i (+ pred_b[n]).  One chain: token row m = sequence m, result
  // to h row act_row(m, T + pseudo0 + i).  A chain per node: token row m = s * T + v, result to h row
  // act_row(s, T + (pseudo0 + i) * T + v).
  const bf16 *pred_b; int pseudo0;
  // EPI_QKV_ROPE
  int H, Hkv, dh;
  const float2 *rope; const int32_t *seq_ids, *pos;   // pos[R]: row positions
  bf16 *q; size_t q_plane;       // [R][H*dh] hi plane, lo plane
  bf16 *kcache; size_t kv_stride; int max_ctx;        // kcache points at this layer's K plane (row 0)
  KvPages pages;
  // EPI_SWIGLU: y[R][F], N = 2F
  bf16 *y; size_t y_plane; int F;
  // EPI_LOGITS: logits[n_seq * Ms][N], rows as the caller counts them
  float *logits;
};
// row of ss that belongs to token row m (Eq. 3 multiplies rows of the residual stream: all tree rows, or each sequence's anchor)
template <int EPI> __device__ __forceinline__ int lin_src_row(const LinArgs &a, int m) {
  return EPI == EPI_PSEUDO && !a.rw.chains ? act_row(a.rw, m, a.rw.anchor) : m;
}
// pdl: launch with programmatic stream serialization (the kernel waits on its predecessor itself).
cudaError_t launch_gemm(GemmEpilogue epi, const LinArgs &a, bool pdl, cudaStream_t st);
// additions in a row that an accumulator of that GEMM sees (its precision, for the tests)
int gemm_additions(GemmEpilogue epi, int N, int K, int F, int dh, int R, int planes);
bool gemm_tc_available();         // the driver entry point for tensor-map encoding was found

// What the finishers of the persistent kernel's GEMMs read (fused_step.cu).
struct GemmArgs {
  int R, N, K;      // token rows; output columns; contraction length
  Rows rw; int rows_active;      // rows with v < rows_active are written, the others skipped
  // X holds h * g, not yet divided by the RMS: row m of the result is scaled by
  // 1 / sqrt(sum_w ss[m][w] / K + eps) (ss == NULL: X is used as it is)
  const float *ss; float eps;
  // EPI_QKV_ROPE
  int H, Hkv, dh;
  const float2 *rope; const int32_t *seq_ids; const int32_t *ctx_len; const int32_t *pos;   // pos[R]: row positions
  bf16 *q; size_t q_lo_off;      // [R][H*dh] hi plane, lo plane
  bf16 *kcache; size_t seq_stride, kv_stride; int max_ctx;  // kcache points at this layer's K plane (row 0)
  KvPages pages;
  // EPI_SWIGLU: y[R][F], N = 2F
  bf16 *y; size_t y_lo_off; int F;
  // EPI_LOGITS: logits[R][N]
  float *logits;
  // EPI_PSEUDO: output n = i * K + o of map pseudo0 + i (+ pred_b[n]).  One chain: row m = sequence m, result to
  // h_rows[(m * Ms + T + pseudo0 + i) * K + o].  A chain per node: row m = s * T + v, result to
  // h_rows[(s * Ms + T + (pseudo0 + i) * T + v) * K + o].
  float *h_rows; const bf16 *pred_b; int pseudo0;
};

// ---- tree-masked split-KV attention ---------------------------------------
constexpr int kAttnMaxSplits = 8;   // kv splits = CTAs per cluster (portable cluster size limit)
// Blocks of query rows: `rows`: up to 128 as the MMA's M dimension, else up to 48 as its N; qblocks of qper each.
struct AttnTcPlan { bool rows; int qblocks, qper, splits; };
struct AttnArgs {
  AttnTcPlan tc;
  Rows rw; int rows_active;
  int H, Hkv, dh;
  const bf16 *q; size_t q_lo_off;   // [R][H*dh] rotated queries, hi and lo planes
  const bf16 *kcache;         // this layer's K plane of slot 0; V plane = kcache + kv_stride
  size_t seq_stride, kv_stride; int max_ctx;
  KvPages pages;
  const int32_t *seq_ids, *ctx_len;
  const int32_t *pos;         // [R] absolute position of every row (row 0 of a sequence: its committed length)
  const uint32_t *mask;       // [R][kMaskWords]
  int splits;                 // kv splits (grid.x = cluster size), 1 to kAttnMaxSplits
  int q_planes, p_planes;     // bf16 planes of the queries / of the probabilities that enter the tensor cores: 2 (hi, lo) or 1
  bf16 *o; size_t o_lo_off;   // [R][H*dh] hi plane, lo plane
  int *err; unsigned long long wait_ns;   // status word and bound of the device-side waits (tensor-core kernel; 0: default)
};
// kv splits for `groups` = sequences x kv heads x query blocks and `kv_tiles` 64-position tiles
int attention_splits(int groups, int kv_tiles);
cudaError_t launch_attention(const AttnArgs &a, bool pdl, cudaStream_t st);
bool attention_early(int dh, int rows, int kv_tiles);     // whether its early launch pays: rows of a sequence, 64-position tiles
// The tcgen05 kernels (head dimension 128): 128-position tiles, query rows x heads of the group in blocks of at most
// kAttnTcMaxCols or 128; a.tc and a.splits from attention_tc_plan.  seq_heads = sequences x kv heads.
constexpr int kAttnTcTile = 128, kAttnTcMaxCols = 48;
AttnTcPlan attention_tc_plan(int qrows, int seq_heads, int kv_tiles, bool prompt, int sm_count);
cudaError_t launch_attention_tc(const AttnArgs &a, bool pdl, cudaStream_t st);

// ---- the decoder layers of a step as one persistent kernel (fused_step.cu) ------------------------------
struct FusedShape { int L, d, H, Hkv, dh, F, V, max_ctx; float eps; };
struct FusedStep {
  FusedShape shape;
  Rows rw;
  int tl[8];                 // insertion layer of each prediction step (non-decreasing)
  bool want_head;            // final norm + lm-head
  bool prenorm;              // Eq. 3 reads the anchor through the insertion layer's input RMSNorm
  int Rp, ws_rows;           // rows per activation plane, per scratch tile
  int n_hi_max;              // upper bound of the longest committed context among the sequences
  int max_batch;             // of the configuration (sizes the attention scratch)
  uint64_t weights_gen;      // changes whenever the weight pointers change
  unsigned long long wait_ns;   // bound of every device-side wait (0: default)
  // weights (device pointers; the per-layer arrays are host arrays of L pointers)
  const void *const *wqkv, *const *wo, *const *wgu, *const *wd, *const *g_attn, *const *g_mlp;
  const void *g_final, *lm_head, *pred_w, *pred_b;
  // workspace
  float *h, *ws, *ss, *logits, *attn_ws;
  bf16 *x, *xp, *q, *o, *y, *kv;
  size_t kv_seq, kv_layer, kv_plane;
  KvPages pages;
  const float2 *rope; const int32_t *pos, *seq_ids, *ctx_len; const uint32_t *mask;
  int *err; unsigned *bar;   // status word; arrival counter of the grid barrier (zero before the launch)
  void *d_maps;              // device room for the tensor maps: fused_map_bytes(L) bytes, 128-byte aligned
};
struct FusedPlan;            // host-side cache of the phase list and the tensor maps of one step shape
FusedPlan *fused_plan_create();
void fused_plan_destroy(FusedPlan *p);
size_t fused_map_bytes(int n_layers);
size_t fused_attn_ws_floats(int max_batch, int H, int Hkv, int dh);   // scratch of the attention splits
// whether the fused kernel can run this step (at most 48 rows; every GEMM's stream-K schedule fits its scratch)
bool fused_eligible(const FusedShape &sh, const Rows &rw);
// Runs everything between the embedding and the top-B: all decoder layers, Eq. 3 at its layers, and (want_head)
// the final norm and the lm-head.  Cooperative launch, one CTA per SM.
cudaError_t launch_fused_layers(FusedPlan *plan, const FusedStep &fs, bool pdl, cudaStream_t st, int *launches);
// one CTA waits (bounded by wait_ns, 0 = default) on a barrier nobody arrives on, sets *err and returns
cudaError_t launch_wait_selftest(int *err, unsigned long long wait_ns, cudaStream_t st);

}  // namespace firp
