// The plan of a weight-streaming GEMM (gemm_tcgen05.cu): which tiles and k blocks a CTA multiplies, into which accumulators, and what
// its shared memory holds.  Plain C++, so that the CPU tests can ask for the plan of any shape.
#pragma once
#include <stdint.h>

#include <algorithm>

#include "rows.h"

namespace firp {

enum GemmEpilogue { EPI_RESIDUAL = 0, EPI_QKV_ROPE = 1, EPI_SWIGLU = 2, EPI_LOGITS = 3, EPI_PSEUDO = 4 };

constexpr int kGemmBK = 64;        // k elements per pipeline stage

namespace gemm {

constexpr int BM = 128;            // weight rows per MMA tile
constexpr int BK = kGemmBK;        // k elements of a pipeline stage: 64 bf16 = 128 bytes = one swizzle row
constexpr int kThreads = 384;      // 12 warps
constexpr int kEpiWarps = 8;
constexpr int W_TILE = BM * 128;   // bytes of one 128-row weight tile of a k block
constexpr int kSmemMax = 227 * 1024;
constexpr int kTailBytes = 2496;   // row scales, slots and lengths, row indices, barriers, TMEM address (behind the rings)
constexpr int kMaxRows = 256;      // token rows of a CTA (MMA N)
constexpr int kMaxW = 12, kMaxX = 6;  // ring depths: weight tiles, activation stages

// How the rows of the weight are dealt to tiles of 128, each one TMA box per k block.
//   ROWS_LINEAR   128 neighbouring rows
//   ROWS_GATE_UP  64 gate rows and the up rows that go with them, in turns of 8, so that such a pair is 8 lanes apart in one warp
//   ROWS_ROTARY   128 / dh heads; the rows of a head in groups of 32: 16 columns of its first half, then their partners in
//                 the second half, so that a rotary pair is 16 lanes apart in one warp
enum RowMode { ROWS_LINEAR = 0, ROWS_GATE_UP = 1, ROWS_ROTARY = 2 };
// Which tiles and k blocks a CTA multiplies.
struct TileSched {
  int mode, heads;   // heads: of a tile (ROWS_ROTARY)
  int n_tiles, KB;   // tiles; 64-wide k blocks
  int jobs, split;   // job j = tiles [n_tiles j / jobs, n_tiles (j + 1) / jobs), its k blocks cut over `split` CTAs
  int blocks;        // of token rows: the CTAs of a job's blocks are neighbours, so that its weights come from HBM once
};
// Shared memory and operand shape of a launch.
struct TileCfg {
  int planes, npad;     // activation planes; token rows of a block padded to the MMA's N
  int rpb;              // token rows of a block
  int acc;              // accumulator columns per tile
  int issuers, by_tile; // MMA issuing warps: they take the units in turn, each with accumulator sets of its own, or the tiles
  int sets, acc_set;    // accumulator sets (summed in the epilogue), columns per set
  int sw, sx;           // ring depths: weight tiles, activation stages
  int planes_side;      // planes that sit side by side in the accumulator's columns
  int tpo, inv_tpo;     // token rows finished per CTA of a cluster; ceil(65536 / tpo)
  int tp;               // tiles per epilogue pass (what the ring's memory holds)
  int tail;             // bytes from the rings' start to what lies behind them
  int red_off;          // where the sums over the k slices go: behind the rings, or 0: over them
  int rope_off, rope_bytes;      // the step's rotary table, if it is brought into shared memory
  int pdl;
  uint32_t idesc, tmem_cols;
};

constexpr int align_n(int v, int a) { return (v + a - 1) / a * a; }
constexpr uint32_t pow2_cols(int c) { return c <= 32 ? 32 : c <= 64 ? 64 : c <= 128 ? 128 : c <= 256 ? 256 : 512; }
constexpr bool few_rows(int r) { return r <= 48; }      // of a block: the epilogue takes 8 at a time

struct Plan { TileSched sc; TileCfg cf; int tm, merged, smem, adds; };

// cycles of one M = 128, K = 16 MMA of n columns: reading the operands from shared memory (128 + n rows of 32 bytes at 128
// bytes a cycle), computing, or issuing it, whichever takes longest (measured: 50 at 16 columns, 55 at 80, 72 at 144)
inline float mma_clk(int n) { return std::max(50.f, std::max(n / 2.f, 34.f + n / 4.f)); }

// Additions in a row that an accumulator would see if every SM of a B200 had an equal share of the matrix, in pairs of tiles, with two
// planes into the same columns from 49 rows on.  The tensor core truncates where it adds to an accumulator, so the error of a sum
// grows with their number: against 64-bit sums of the same planes, in the 2-norm, 0.24e-6 after 16, 0.48e-6 after 32, 1.1e-6 after
// 76, 2.1e-6 after 128, 4.5e-6 after 256, 9.2e-6 after 512; what the two planes leave out of an activation is 2.4e-6.
inline int longest_sum(int n_tiles, int KB, int rows, int planes) {
  const int units = (n_tiles + 1) / 2 * KB, share = std::min(KB, (units + 147) / 148);
  return std::max(16, 4 * share * (planes == 1 || rows <= (planes == 3 ? 80 : 48) ? 1 : planes));
}

// What a plan costs, in microseconds: the weights at the rate HBM gives that many CTAs (6.8 TB/s from 84 on), a CTA's MMAs, its bytes
// from L2 (which gives a CTA 150 GB/s and all of them 15 TB/s), or a ring's turnaround, whichever is longest; a share of the others; and
// for each wave its start and its epilogue: from registers, or a push to the CTAs of the cluster and the sums there.
struct Rates {
  float mma_mhz;                          // cycles above to microseconds
  float deep_row;                         // per tile and token row: reading a third and fourth accumulator set
  float direct, direct_row;               // epilogue from registers: start, per tile and token row
  float push_row, own_row;                // push, sums: per tile and token row
  float lone, beside, over;               // barriers: one CTA, sums beside the rings, sums over them
  float ring_x, ring_w;                   // a ring slot goes round in that time: activations, weights
  float share, wave;                      // of what is not the longest; a wave's start
  float wide_split; int wide_split_rows;  // seven or eight k slices, at more rows than that
  int tail_bytes;                         // of shared memory behind the rings
  bool pairs;                             // gate/up jobs have two tiles, whose sums are made together
};
// Two sets of them, because what is fastest must not decide how long the sums are.  How long: kBySums, set by hand; the plan that it finds
// for the rows of the whole call is the measure of precision, and stays as it is.  Which of the plans whose sums are no longer: kByTime, a
// fit to every plan of the 7B, 13B and 34B shapes' projections at 20-140 token rows and at prompts of 150-2002 (9216 times of launches
// back to back), within 7 % of the times of the plans near the best.  Under the same limit, us per step with the first set's constants alone / with
// pairs of gate/up tiles only / so: a chain under each of 32 nodes 3766 / 3777 / 3737, 6 x 18 rows 4754 / 4733 / 4718, 131 rows 5771 / 5766 / 5754,
// 67 rows of the 13B shape 6351 / 6325 / 6327, 4 x 35 of the 34B shape 5833 / 5798 / 5842 (spread 0.3 %, the last 0.8).  (Without that limit jobs of three gate/up tiles with sums twice as
// long would be chosen: 45 instead of 51 us at 131 rows of the 7B shape, 137 instead of 160 at 140 of the 34B shape.)
constexpr Rates kBySums{1850.f, 0.004f, 0.5f, 0.025f, 0.025f, 0.05f, 0.5f, 1.f, 2.f, 0.9f, 1.4f, 0.1f, 2.f, 3.f, 128, 1984, true};
constexpr Rates kByTime{1570.f, 0.008f, 0.f, 0.028f, 0.017f, 0.0017f, 1.2f, 1.7f, 3.8f, 0.72f, 1.12f, 0.035f, 1.5f, 1.f, 0, kTailBytes, false};

struct GemmShape { GemmEpilogue epi; int N, K, F, dh, planes; };
inline int gemm_tiles(const GemmShape &g) { return g.epi == EPI_SWIGLU ? (g.F + BM / 2 - 1) / (BM / 2) : (g.N + BM - 1) / BM; }

// The cheapest plan whose accumulators see at most `limit` additions (twice as many, and so on, where there is none).
// step: of a step or of a prompt.  cluster_ctas[n]: CTAs that can run at once in clusters of n.
inline Plan cheapest_plan(const GemmShape &g, int rows, bool step, int limit, const Rates &rt, const int *cluster_ctas) {
  const GemmEpilogue epi = g.epi;
  const int planes = g.planes;
  Plan best{};
  float best_cost = 1e30f;
  TileSched s{};
  s.mode = epi == EPI_SWIGLU ? ROWS_GATE_UP : epi == EPI_QKV_ROPE ? ROWS_ROTARY : ROWS_LINEAR;
  s.heads = s.mode == ROWS_ROTARY ? BM / g.dh : 0;
  s.n_tiles = gemm_tiles(g);
  s.KB = (g.K + BK - 1) / BK;
  const int share = longest_sum(s.n_tiles, s.KB, rows, planes);
  for (int max_adds = limit; best.tm == 0 && max_adds < (1 << 20); max_adds *= 2)
  for (int most : {256, 192, 128}) {         // token rows of a block: blocks of equal size
  s.blocks = (rows + most - 1) / most;
  const int R = align_n((rows + s.blocks - 1) / s.blocks, s.blocks > 1 ? 16 : 1);
  s.blocks = (rows + R - 1) / R;
  if (most < 256 && step) break;
  for (int merged = 1; merged >= 0; --merged) {
    if (!merged && planes == 1) continue;
    const int npad = merged ? align_n(R, planes == 2 ? 8 : 16) : align_n(R, 16);
    const int n_mma = merged ? planes * npad : npad;
    if (n_mma > 256) continue;
    const int x_stage = planes * npad * 128;
    for (int tm = 1; tm <= 3; ++tm) {
      // the epilogue of many rows reads 16 columns at a time, 8 of them beyond the last plane's when npad is an odd multiple of 8
      const int over = few_rows(R) ? 0 : npad & 8;
      if (tm * n_mma + over > 512) continue;
      for (int split = 1; split <= 8 && split <= s.KB; ++split) {
        const int cap = cluster_ctas[split] / split * split;
        int jobs = (s.n_tiles + tm - 1) / tm;
        const int waves = (jobs * s.blocks * split + cap - 1) / cap, kb = (s.KB + split - 1) / split;
        // single gate/up tiles in several waves bring the activations to every one of them again, which the costs below do not see: a step
        // of the 34B shape (12 layers) at 45 / 48 rows 3450 / 3671 us with them, 3400 / 3639 without
        if (s.mode == ROWS_GATE_UP && (rt.pairs ? tm != 2 : tm == 1 && waves > 1 && step)) continue;
        const int per = std::min(tm, s.n_tiles);
        // rings: four activation stages (two or three of the wide ones), the rest for weight tiles
        // and, when it is not much, room for the sums over the k slices (saves a cluster barrier) or the rotary table (an L2
        // round trip every 16 token rows)
        const int tpo = align_n((R + split - 1) / split, 4), per_tile = split * tpo * 512;         // bytes of a tile's sums
        int red = split > 1 ? per * per_tile : 0, rope = epi == EPI_QKV_ROPE ? align_n(std::min(tpo, R) * g.dh * 4, 128) : 0;
        if (red > 40 * 1024) red = 0;
        if (rope > 24 * 1024) rope = 0;
        const int side = red + rope;
        const int avail = kSmemMax - 1024 - rt.tail_bytes - side;
        int sx = std::min(x_stage <= 12 * 1024 ? 4 : x_stage <= 24 * 1024 ? 3 : 2, std::max(kb, 1));
        const bool by_unit = tm == 1 && 2 * n_mma + over <= 512 && s.KB / split >= 2;
        if (by_unit) sx = std::max(2, sx & ~1);
        int sw = std::min(std::min(kMaxW, (avail - sx * x_stage) / W_TILE), kb * per);
        if (by_unit) sw &= ~1; else sw = sw / per * per;
        if (sw < per || sw * W_TILE + sx * x_stage > avail) continue;
        if (x_stage <= 24 * 1024) sx = std::min(std::min(kMaxX, kb), (avail - sw * W_TILE) / x_stage);      // what is left
        if (by_unit) sx &= ~1;
        if (sw < 2 * per && kb > 1) continue;
        // As many accumulator sets as fit, up to four, share the k blocks; what is still longer than the limit is left to a
        // split.
        int sets = by_unit ? 2 : 1;
        const int per_kb = (BK / 16) * (merged ? 1 : planes);
        auto adds_of = [&](int n) { return (kb + n - 1) / n * per_kb; };
        while (sets < 4 && (adds_of(sets) > std::min(share, max_adds) || (adds_of(sets) > 96 && (sets < 2 || !step))) &&
               2 * sets * tm * n_mma + over <= 512 && s.KB / split >= 2 * sets) sets *= 2;
        // Three are not dealt to two issuers, and one is too slow for a whole contraction (13B shape, 131 rows: the QKV projection
        // 49.6 us so, 44.2 in three slices of three tiles; down in three slices 41.5, in eight of three tiles 46.6).
        const bool lone = by_unit && sets == 2 && adds_of(2) > std::min(share, max_adds) && split > 1 && 3 * n_mma + over <= 512 && s.KB / split >= 3;
        if (lone) sets = 3;
        const int adds = adds_of(sets);
        if (adds > max_adds) continue;
        const int ctas = std::min(jobs * s.blocks * split, cap), own = std::min(tpo, R);
        const float hbm = (float)s.n_tiles * s.KB * W_TILE / 6.8e6f * std::max(1.f, 84.f / ctas);
        const float mma = (float)waves * per * kb * 4.f * (merged ? 1 : planes) * mma_clk(n_mma) / rt.mma_mhz;
        const float ingest = (float)waves * kb * (per * W_TILE + x_stage) / std::min(150e3f, 15e6f / ctas);
        const bool direct = split == 1 && (epi == EPI_QKV_ROPE || epi == EPI_SWIGLU || epi == EPI_LOGITS);
        const float out = (sets > 2 ? rt.deep_row * R * per : 0.f) + (direct ? rt.direct + rt.direct_row * R * per : rt.push_row * R * per + rt.own_row * own * per + (split == 1 ? rt.lone : red ? rt.beside : rt.over));
        const float rings_us = (float)waves * kb * std::max(rt.ring_x / sx, rt.ring_w * per / sw);
        const float cost = std::max(std::max(hbm, rings_us), std::max(mma, ingest)) + rt.share * (hbm + mma + ingest) + waves * (rt.wave + out) + (split >= 7 && rows > rt.wide_split_rows ? rt.wide_split : 0.f);
        TileCfg c{};
        c.planes = planes; c.rpb = R; c.npad = npad; c.acc = n_mma; c.sw = sw; c.sx = sx;
        c.tpo = tpo; c.inv_tpo = (65536 + c.tpo - 1) / c.tpo;
        c.planes_side = merged ? planes : 1; c.acc_set = tm * n_mma; c.sets = sets; c.issuers = (by_unit && !lone) || tm >= 2 ? 2 : 1; c.by_tile = tm >= 2;
        c.tmem_cols = pow2_cols(c.sets * tm * n_mma + over);
        const int rings = align_n(sw * W_TILE + sx * x_stage, 128);
        if (red) {
          c.red_off = rings; c.tp = per; c.tail = rings + red;
        } else {
          c.tail = align_n(std::max(rings, direct ? 0 : rt.pairs && s.mode == ROWS_GATE_UP ? 2 * per_tile : per_tile), 128);      // over the rings
          c.tp = direct ? per : std::min(per, c.tail / per_tile);
        }
        if (rope) { c.rope_off = c.tail; c.rope_bytes = rope; c.tail += rope; }
        const int smem = c.tail + 1024 + rt.tail_bytes;
        if (smem > kSmemMax || cost >= best_cost) continue;
        best_cost = cost;
        best = Plan{s, c, tm, merged, smem, adds};
        best.sc.jobs = jobs; best.sc.split = split;
      }
    }
  }
  }
  return best;
}

// The plan of a layer's GEMM on `rows` token rows, of a call that has `call_rows` of them once all pseudo rows are inserted.
//
// A prompt's sums may be longer than a step's: its results are as far from a 64-bit run as with the equal shares' (cache rows of 1999
// tokens of the 7B shape 2.24e-3 / 2.32e-3, of 500 2.76e-3 / 2.88e-3: the rounding of the cache to bf16 hides them), and the equal shares'
// limit costs it 5 %.  A step's keep it, or 96 where that is more (an error below the planes' own).
inline Plan make_plan(const GemmShape &g, int rows, int call_rows, const int *cluster_ctas) {
  const int KB = (g.K + BK - 1) / BK;
  const bool step = call_rows <= kMaxTreeRows;
  int limit = g.epi == EPI_RESIDUAL ? std::max(176, (step ? 2 : 1) * KB) : (g.epi == EPI_SWIGLU ? 260 : g.epi == EPI_LOGITS ? 512 : 176) * std::max(64, KB) / 64;
  if (step) limit = std::min(limit, std::max(96, longest_sum(gemm_tiles(g), KB, call_rows, g.planes)));
  const Plan sums = cheapest_plan(g, call_rows, step, limit, kBySums, cluster_ctas);
  return cheapest_plan(g, rows, step, sums.adds, kByTime, cluster_ctas);
}

}  // namespace gemm
}  // namespace firp
