// The rows of a step, in plain C++: the CPU tests run it.
#pragma once
#include <stdint.h>

#ifndef FIRP_HD
#ifdef __CUDACC__
#define FIRP_HD __host__ __device__ __forceinline__
#else
#define FIRP_HD inline
#endif
#endif

namespace firp {

constexpr int kMaxSeq = 16;        // sequences per step
constexpr int kMaxTreeRows = 144;  // rows per sequence: T + k (128 + 8), or T (1 + k) with a chain under every node
constexpr int kMaxPromptRows = 2047;  // rows of a prompt that run at once, pseudo rows included

// Per-step row geometry shared by every kernel.  Row r = s * Ms + v in what the caller gives and gets and in TreeMeta.
struct Rows {
  int n_seq;   // sequences in this step
  int T;       // tree rows per sequence
  int k;       // pseudo rows per sequence
  int Ms;      // T + k
  int R;       // n_seq * Ms
  int anchor;  // tree row the pseudo chain hangs off (one chain)
  int chains;  // != 0: a chain under every tree node; chain row i (1-based) of node v is row T + (i-1) T + v
  int kc;      // prediction steps per chain (k = kc with one chain, k = T * kc with a chain per node)
  int masked;  // != 0: a pseudo row sees no other pseudo row (the "Masked" ablation of Section 4.3)
  int prompt;  // != 0: a stretch of a prompt: one sequence, rows 0 .. T-1 a chain, the pseudo rows behind it; more rows than a
               // tree may have, no masks in TreeMeta (row v sees the rows up to itself)
  int by_step; // != 0: the rows of the activations (act_row below) go by prediction step
};
// Row of the activations (residual stream, GEMM operands, queries, rotary table) that holds row v of sequence s.  By step: the tree
// rows of all sequences, then their rows of the first prediction step, of the second, ..., so that the rows that a layer has are
// the first ones and its GEMMs carry no others.
FIRP_HD int act_row(const Rows &rw, int s, int v) {
  if (!rw.by_step) return s * rw.Ms + v;
  if (v < rw.T) return s * rw.T + v;
  const int per = rw.chains ? rw.T : 1, i = (v - rw.T) / per;
  return rw.n_seq * (rw.T + i * per) + s * per + (v - rw.T - i * per);
}
// what a row of the activations is, in a word
FIRP_HD uint16_t seq_row(int s, int v) { return (uint16_t)(s << 11 | v); }
FIRP_HD int row_seq(int w) { return w >> 11; }
FIRP_HD int row_in_seq(int w) { return w & 2047; }

}  // namespace firp
