// Weight-streaming GEMM of the step on the 5th-generation tensor cores (tcgen05 + TMEM), operands staged by TMA, with
// the elementwise step that follows the contraction in its epilogue.
//   out[m][n] = sum_k X[m][k] * W[n][k], m = the T + k token rows of a step (at most 144) or the rows of a prompt.
//
// Roles are swapped: weight rows are the MMA M dimension (one TMEM lane each), token rows the MMA N dimension (one
// TMEM column each).  A tile is 128 weight rows (64 gate rows and the up rows that go with them); a job is up to TM tiles
// that one thread block, or a cluster, finishes by itself for up to 256 token rows: the k blocks of a job are cut over
// the `split` CTAs of the cluster.  Grid = jobs x blocks of token rows x split, one wave wherever the matrix allows it.
//
// Why whole tiles and not one equal share of the matrix per SM: HBM does not need every SM.  A TMA ring of 6 x 32 KB per
// CTA streams 6.7 TB/s from 86 CTAs, 6.8 from 108, 6.9 from 128 (measured), so a schedule that leaves some SMs without
// weights costs 1-3 % of the stream, while shares that end in mid-tile cost a pass over fp32 partial tiles in global
// memory, a kernel of its own to sum them and a hand-over: 7 us after the QKV, gate/up and down projections and 14 us after
// the O projection at 35 rows of the 7B shape, 37 of 102 us per layer.  Step at the 7B shape, 35 rows, 512 cached tokens:
// 3534 -> 3121 us; one row 3062 -> 2696; 13B shape, 67 rows 8958 -> 6734; 34B shape, 140 rows 6631 -> 6230.  (With the limit on a
// step's sums, in turn on one box: 3133 -> 3163, 2706 -> 2728, 6532 -> 6518, 6045 -> 6118.)
//
// A prompt comes as one stretch of up to 2047 rows, in blocks of up to 256: the weights, 13.5 GB at the 7B shape, are read
// once instead of once per 141 rows.  It is bound by the MMA issue of two passes over the bf16 planes: 1999 tokens of the 7B
// shape 92.2 -> 65.9 ms (61.3 with attn_tc.cu's blocks of 128 rows); per layer QKV 0.44, attention 0.16, O 0.19, gate/up 0.60,
// down 0.45 ms.
//
// Bound now, per layer of 93 us at 35 rows (device timestamps): the weight stream (QKV 15 us, O 5, gate/up 27, down 13.5, 6.1-6.9 TB/s),
// the epilogues (2-2.5 each), four hand-overs of 2 (1.3 until the wait for the kernel before returns, 0.7 until its output is in
// shared memory; O's first weights, behind the attention's late blocks, take 4.5) and the attention's 11-13.
//
// Per CTA (one per SM at the large shapes):
//   warp 0     : weight producer (one thread, TMA, 128-byte swizzle, deep ring).  Weights never depend on the previous
//                kernel, so under programmatic dependent launch this stream starts while the predecessor drains.
//   warp 2     : activation producer: the bf16 planes of the k block, after waiting for the previous kernel.
//   warps 1, 3 : MMA issuers: tcgen05.mma kind::f16, M = 128, K = 16.  The planes of the activations (hi, lo) either sit
//                side by side as ONE operand of N = planes x npad columns (added in the epilogue) or are accumulated
//                one after the other into npad columns.  The whole warp runs the loop and an elected lane issues, which
//                keeps the descriptors in uniform registers (M = 128, N = 80: 59 cycles per MMA; one lane alone: 86).  One of them
//                issues alone where a job has one tile of one accumulator set, or of three.
//   warps 4-11 : epilogue.  TMEM -> shared memory of the CTA of the cluster that finishes the token row (the ring's
//                memory, no longer needed), cluster barrier, sum over the k slices in rank order, then the fused step:
//                residual + RMSNorm operand, rotary + cache, SwiGLU, logits, or Eq. 3.
// Every mbarrier wait is bounded (2 s, or what the caller set, counted from the previous kernel's completion: an early launch
// does not count against it).  On expiry the status word is set and the kernel runs to its end; the producers stop
// loading, and the block ends when what it has started has landed and the last MMA has completed.  (Only then: producers that
// always waited for their last loads cost a step of up to 32 rows 1-5 %.)
#include <cooperative_groups.h>
#include <cuda.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "finish_device.cuh"
#include "firp_kernels.cuh"
#include "gemm_plan.h"
#include "launch_util.cuh"
#include "pipeline.h"
#include "tc_device.cuh"

namespace cg = cooperative_groups;

namespace firp {

using namespace gemm;

namespace {

constexpr int kNoRow = -1, kNoKv = -2;      // of s_kv below

// A CTA starts its k range at a place of its own and wraps around: CTAs that march through k together would ask the same
// L2 slices for the same activation rows, and HBM for weight rows whose addresses differ only above bit 12.
struct CtaWork { int t0, nt, kb0, kb1, off, block; };
__device__ __forceinline__ CtaWork cta_work(const TileSched &s, int cta) {
  const int jb = cta / s.split, r = cta - jb * s.split, j = s.blocks == 1 ? jb : jb / s.blocks;
  CtaWork w;
  w.block = jb - j * s.blocks;
  w.t0 = s.n_tiles * j / s.jobs;
  w.nt = s.n_tiles * (j + 1) / s.jobs - w.t0;
  w.kb0 = s.KB * r / s.split;
  w.kb1 = s.KB * (r + 1) / s.split;
  w.off = (cta * 10) % (w.kb1 - w.kb0) & ~1;      // even: pairs of k blocks share 256-byte lines
  return w;
}
// k block of unit u
__device__ __forceinline__ int unit_kb(const CtaWork &w, int u) { const int k = w.kb0 + w.off + u; return k < w.kb1 ? k : k - (w.kb1 - w.kb0); }

// one k block of one tile: 16 KB
__device__ __forceinline__ void load_tile(uint32_t dst, const CUtensorMap *tm, const TileSched &s, int tile, int kb, uint32_t bar, uint64_t pol) {
  if (s.mode == ROWS_ROTARY) tma_load_5d(dst, tm, kb * BK, tile * s.heads, bar, pol);
  else if (s.mode == ROWS_GATE_UP) tma_load_4d(dst, tm, kb * BK, 0, 0, tile * 8, bar, pol);
  else tma_load_2d(dst, tm, kb * BK, tile * BM, bar, pol);
}

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// every thread of the cluster has got as far as cluster_arrive
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 mul4(float4 a, float s) { return make_float4(a.x * s, a.y * s, a.z * s, a.w * s); }
// The rings as their producers see them (pipeline.h).
struct RingBase {
  uint32_t full, empty;          // barriers of slot 0
  int *err; unsigned long long wait_ns; bool dead;
  __device__ __forceinline__ bool free(int, int slot, uint32_t parity) { return mbar_wait(empty + 8 * slot, parity, err, dead, wait_ns); }
};
struct Landing {
  uint32_t full; int *err;
  __device__ __forceinline__ void landed(int slot, uint32_t parity) { mbar_drain(full + 8 * slot, parity, err); }
};
struct WeightRing : RingBase {   // one tile per slot
  const CUtensorMap *tm; const TileSched &sc; const CtaWork &wk;
  uint32_t ring; uint64_t pol;
  int it, t;                     // of the next load: unit, tile
  __device__ __forceinline__ void load(int, int slot) {
    mbar_expect_tx(full + 8 * slot, W_TILE);
    load_tile(ring + slot * W_TILE, tm, sc, wk.t0 + t, unit_kb(wk, it), full + 8 * slot, pol);
    if (++t == wk.nt) { t = 0; ++it; }
  }
};
struct ActRing : RingBase {      // all planes of a k block per slot
  const CUtensorMap *tm; const CtaWork &wk;
  uint32_t ring, stage; uint64_t pol;
  int row0;
  __device__ __forceinline__ void load(int u, int slot) {
    mbar_expect_tx(full + 8 * slot, stage);
    tma_load_3d(ring + slot * stage, tm, unit_kb(wk, u) * BK, row0, 0, full + 8 * slot, pol);
  }
};
// MERGED: the activation planes sit side by side in one operand (or there is only one); else one after the other.  DEEP: more than two
// accumulator sets, or planes side by side (in one kernel with the others the code they skip cost them 1-2 % of a two-layer step).
// The epilogue's code runs once per launch from a cold instruction cache, in the shadow of nothing: one kernel per epilogue
// and rolled loops keep it short (all five in one kernel, four items unrolled: 5-7 us instead of 1-2).
// C: token rows (TMEM columns) that the epilogue takes at a time.  Eight for up to 48 rows: its passes are then so short that they run
// about as long as their code takes to come from a cold instruction cache (us per step with 16 / with 8, nothing else changed: two-layer
// shape 80.7 / 76.4, one row of the 7B shape 2643 / 2603, 35 rows 3047 / 3038); with more rows sixteen hide more of the TMEM loads (128 and 131 rows 5987 / 6033).
template <int TM, bool MERGED, bool DEEP, int C, int EPI>
__global__ void __launch_bounds__(kThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ LinArgs a,
            const __grid_constant__ TileSched sc, const __grid_constant__ TileCfg cf) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;      // swizzled tiles need 1024-byte alignment
  uint8_t *data = smem_raw + (base - smem_u32(smem_raw));
  const int sx_n = cf.sx;
  const uint32_t x_plane = (uint32_t)cf.npad * 128u, x_stage = x_plane * cf.planes;
  const uint32_t w_ring = base, x_ring = base + cf.sw * W_TILE;
  float *s_rs = reinterpret_cast<float *>(data + cf.tail);          // 1 / RMS of every token row
  int *s_slot = reinterpret_cast<int *>(s_rs + kMaxRows), *s_pos = s_slot + kMaxSeq;      // of every sequence
  uint16_t *s_row = reinterpret_cast<uint16_t *>(s_pos + kMaxSeq);                        // seq_row of every token row, 0xffff: none
  int *s_kv = reinterpret_cast<int *>(s_pos + kMaxSeq);      // QKV: instead, every token row's row of a cache plane; kNoKv: none, kNoRow: no token row
  const uint32_t bars = base + cf.tail + kMaxRows * 8 + 2 * kMaxSeq * 4;
  const uint32_t full_w = bars, empty_w = full_w + 8 * kMaxW, full_x = empty_w + 8 * kMaxW, empty_x = full_x + 8 * kMaxX,
                 acc_full = empty_x + 8 * kMaxX, rope_full = acc_full + 8, tmem_slot = rope_full + 8;
  volatile int *gave_up = reinterpret_cast<volatile int *>(data + (tmem_slot + 4 - base));   // a thread's wait has run out
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const CtaWork wk = cta_work(sc, blockIdx.x);
  const int row0 = wk.block * cf.rpb, R = min(cf.rpb, a.R - row0);      // this CTA's token rows
  const int n_units = wk.kb1 - wk.kb0;
  // The weight ring holds single tiles (16 KB slots: a slot is free again after four MMAs).  Its depth is a multiple of the
  // job's tiles, so that a slot always holds the same tile and is read by the same issuer: one that skipped a phase of a
  // slot's barrier would take the phase before it for its own (parity tells neighbouring phases apart, no more).
  const int sw_n = cf.by_tile ? cf.sw / wk.nt * wk.nt : cf.sw;

  if (threadIdx.x == 0) {
    const int readers = cf.by_tile ? cf.issuers : 1;
    for (int i = 0; i < sw_n; ++i) { mbar_init(full_w + 8 * i, 1); mbar_init(empty_w + 8 * i, 1); }
    for (int i = 0; i < sx_n; ++i) { mbar_init(full_x + 8 * i, 1); mbar_init(empty_x + 8 * i, readers); }
    *gave_up = 0;
    mbar_init(acc_full, cf.issuers);
    mbar_init(rope_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(cf.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(data + (tmem_slot - base));
  // Dependents may start as SMs free up.  Not before TMEM is allocated: a dependent on the same SM then only ever waits
  // for columns of a kernel that does not wait for it.
  // The attention reads what was complete before the QKV projection started (context lengths, committed cache rows) before its own
  // wait, so that projection lets it start only after waiting itself.
  if (cf.pdl && EPI != EPI_QKV_ROPE) griddep_launch();
  if (sc.split > 1 && cf.red_off) cluster_arrive();

  bool dead = false;
  const unsigned long long wait_ns = a.wait_ns ? a.wait_ns : kDefaultWaitNs;
  // For what only the issuers' commits end: they start waiting when the previous kernel has completed, bound each of their waits
  // and commit in any case.  (The weight producer does not wait for the previous kernel itself: griddepcontrol.wait between its
  // loads cost a step of up to 32 rows 2-6 %.)
  const unsigned long long all_ns = kDefaultWaitNs + min(wait_ns, 1ull << 48) * (unsigned)(2 * n_units * TM + 2);
  int started = 0;               // loads of a producer
  if (warp == 0) {
    if (lane == 0) {             // ---- weight producer: does not wait for the previous kernel
      uint64_t pol;
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
      WeightRing ring{{full_w, empty_w, a.err, all_ns, false}, &tmW, sc, wk, w_ring, pol, 0, 0};
      started = produce(ring, n_units * wk.nt, sw_n);
      dead = ring.dead;
    }
  } else if (warp == 2) {
    if (lane == 0) {             // ---- activation producer
      uint64_t pol;
      asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
      if (cf.pdl) griddep_wait();
      if (cf.pdl && EPI == EPI_QKV_ROPE) griddep_launch();
      if (EPI == EPI_QKV_ROPE && cf.rope_bytes) {
        const int r0 = (int)(blockIdx.x % sc.split) * cf.tpo, bytes = max(0, min(cf.tpo, R - r0)) * (a.dh >> 1) * 8;   // of the rows finished here
        mbar_expect_tx(rope_full, bytes);
        if (bytes) bulk_load(base + cf.rope_off, a.rope + (size_t)(row0 + r0) * (a.dh >> 1), bytes, rope_full);
      }
      ActRing ring{{full_x, empty_x, a.err, wait_ns, false}, &tmX, wk, x_ring, x_stage, pol, row0};
      started = produce(ring, n_units, sx_n);
      dead = ring.dead;
    }
  } else if (warp == 1 || warp == 3) {        // ---- MMA issuers
    const int iw = warp >> 1;
    if (iw < cf.issuers) {
      if (cf.pdl) griddep_wait();        // the limit of the waits below starts here
      // by units: unit iw, iw + issuers, ... into accumulator sets of its own; by tiles: every unit, tiles iw, iw + issuers, ...
      const int u0 = cf.by_tile ? 0 : iw, du = cf.by_tile ? 1 : cf.issuers;
      const uint32_t tm0 = __shfl_sync(0xffffffffu, tmem, 0);
      uint32_t acc = tm0 + (uint32_t)(u0 * cf.acc_set);      // unit it goes to accumulator set it % sets
      const uint32_t acc_end = tm0 + (uint32_t)(cf.sets * cf.acc_set), acc_step = (uint32_t)(du * cf.acc_set);
      int sw = cf.by_tile ? iw : u0, sx = u0;            // slot of the unit's first tile of this issuer; X slot
      uint32_t parw = 0, parx = 0;
      if (sw >= sw_n) { sw -= sw_n; parw ^= 1; }
      if (sx >= sx_n) { sx -= sx_n; parx ^= 1; }
      for (int it = u0; it < n_units; it += du) {
        const uint64_t dx = smem_desc(x_ring + sx * x_stage);
        bool first = true;
#pragma unroll
        for (int t = 0; t < TM; ++t) {
          if (t < wk.nt && (!cf.by_tile || (t & 1) == iw)) {
            const int sl = cf.by_tile ? sw + t - iw : sw;
            mbar_wait(full_w + 8 * sl, parw, a.err, dead, wait_ns);
            if (first) mbar_wait(full_x + 8 * sx, parx, a.err, dead, wait_ns);
            first = false;
            __syncwarp();                // lanes may leave a wait one by one; what follows is for a converged warp
            tc_fence_after();
            const uint64_t dw = smem_desc(w_ring + sl * W_TILE);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
              if (elect_one()) tc_mma(acc + t * cf.acc, dw + 2 * kk, dx + 2 * kk, cf.idesc, (it >= cf.sets || kk > 0) ? 1u : 0u);
#pragma unroll
              for (int pl = 1; pl < 3; ++pl)
                if (!MERGED && pl < cf.planes && elect_one()) tc_mma(acc + t * cf.acc, dw + 2 * kk, dx + (uint64_t)(pl * (x_plane >> 4)) + 2 * kk, cf.idesc, 1u);
            }
            if (elect_one()) tc_commit(empty_w + 8 * sl);      // the slot is free once these MMAs have read it
          }
        }
        if (first) mbar_wait(full_x + 8 * sx, parx, a.err, dead, wait_ns);      // an issuer without tiles only keeps count
        __syncwarp();
        if (elect_one()) tc_commit(empty_x + 8 * sx);
        sw += cf.by_tile ? wk.nt : du;
        if (sw >= sw_n) { sw -= sw_n; parw ^= 1; }
        acc += acc_step;
        if (acc >= acc_end) acc -= acc_end - tm0;
        sx += du;
        if (sx >= sx_n) { sx -= sx_n; parx ^= 1; }
      }
      if (elect_one()) tc_commit(acc_full);
    }
  }
  __syncwarp();

  // ---- epilogue: warps 4..11 work, the others only take part in the cluster's barriers
  const bool epi = warp >= 4;
  const int ew = warp - 4, quarter = warp & 3, half_w = ew >> 2;
  const int split = sc.split;
  const uint32_t rank = (uint32_t)(blockIdx.x % split);
  const int own0 = (int)rank * cf.tpo, n_own = max(0, min(cf.tpo, R - own0));     // token rows (of the block) this CTA finishes
  const float *red = reinterpret_cast<const float *>(data + cf.red_off);         // [k slice][own row][tile of the pass][128]
  constexpr bool kDirect = EPI == EPI_QKV_ROPE || EPI == EPI_SWIGLU || EPI == EPI_LOGITS;   // may leave from registers
  const int half = EPI == EPI_QKV_ROPE ? a.dh >> 1 : 1;
  if (epi) {
    if (cf.pdl) griddep_wait();
    // one load per CTA (thousands of warps asking L2 for the same word at once take microseconds)
    if (EPI == EPI_QKV_ROPE && warp == 4 && lane < a.rw.n_seq) {
      s_slot[lane] = __ldcg(a.seq_ids + lane);
      s_pos[lane] = __ldcg(a.pos + lane * a.rw.Ms);      // committed length (position of the root row)
    }
    // of every row this CTA finishes: its sequence and row (0xffff: none), and
    // 1 / sqrt(mean(h^2) + eps) from the per-128-column sums of squares, added in a fixed order
    const int nw = a.K >> 7;
    const int m_end = min(kMaxRows, own0 + ((n_own + 15) & ~15));
    for (int m0 = own0 + ew; m0 < m_end; m0 += 4 * kEpiWarps) {
      float v[4];
      uint16_t w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = row0 + min(m0 + u * kEpiWarps, R - 1);
        w[u] = EPI == EPI_PSEUDO && !a.rw.chains ? seq_row(r, 0) : a.row_of ? __ldcg(a.row_of + r) : seq_row(0, r);
        v[u] = 0.f;
        if (a.ss == nullptr) continue;
        const float *p = a.ss + (size_t)lin_src_row<EPI>(a, r) * kNormMaxWarps;
        v[u] = (lane < nw ? __ldcg(p + lane) : 0.f) + (lane + 32 < nw ? __ldcg(p + lane + 32) : 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
        const int m = m0 + u * kEpiWarps;
        if (lane == 0 && m < m_end) {
          s_rs[m] = a.ss ? rsqrtf(v[u] / (float)a.K + a.eps) : 1.f;
          if (EPI == EPI_QKV_ROPE) s_kv[m] = m < own0 + n_own ? w[u] : kNoRow;
          else s_row[m] = m < own0 + n_own ? w[u] : 0xffff;
        }
      }
    }
    if (EPI == EPI_QKV_ROPE) {       // once per row here, and not by every thread that writes to it
      epi_sync();
      const int m = own0 + (int)threadIdx.x - 128;
      if (m < m_end && s_kv[m] != kNoRow) {
        const int s = row_seq(s_kv[m]), pos = s_pos[s] + row_in_seq(s_kv[m]);
        s_kv[m] = pos < a.max_ctx ? (int)kv_row(a.pages, s_slot[s], pos, a.max_ctx) : kNoKv;
      }
    }
  }
  // columns [c0, c0 + C) of tile t: the sums over the planes' columns and the accumulator sets
  auto ld = [](uint32_t ta, float *r) { if (C == 16) tc_ld16(ta, r); else tc_ld8(ta, r); };
  const uint32_t tquarter = tmem + ((uint32_t)(quarter * 32) << 16);
  auto load_acc = [&](int t, int c0, float *r) {
    const uint32_t ta = tquarter + (uint32_t)(t * cf.acc + c0);
    float l[DEEP ? 4 : 3][C];
    auto add = [&](const float *x) {
#pragma unroll
      for (int j = 0; j < C; ++j) r[j] += x[j];
    };
    ld(ta, r);
    if (cf.planes_side > 1) ld(ta + cf.npad, l[0]);
    if (cf.sets > 1) {
      ld(ta + cf.acc_set, l[1]);
      if (cf.planes_side > 1) ld(ta + cf.acc_set + cf.npad, l[2]);
    }
    tc_ld_wait();
    if (cf.planes_side > 1) add(l[0]);
    if (cf.sets > 1) {
      add(l[1]);
      if (cf.planes_side > 1) add(l[2]);
    }
    if (DEEP) {       // the third and fourth set's columns, the third plane's
      if (cf.sets > 2) {
        ld(ta + 2 * cf.acc_set, l[0]);
        if (cf.planes_side > 1) ld(ta + 2 * cf.acc_set + cf.npad, l[1]);
        if (cf.sets > 3) {
          ld(ta + 3 * cf.acc_set, l[2]);
          if (cf.planes_side > 1) ld(ta + 3 * cf.acc_set + cf.npad, l[3]);
        }
        tc_ld_wait();
        add(l[0]);
        if (cf.planes_side > 1) add(l[1]);
        if (cf.sets > 3) {
          add(l[2]);
          if (cf.planes_side > 1) add(l[3]);
        }
      }
      if (cf.planes_side > 2) {
#pragma unroll 1
        for (int i = 0; i < cf.sets; ++i) {
          ld(ta + i * cf.acc_set + 2 * cf.npad, l[0]);
          tc_ld_wait();
          add(l[0]);
        }
      }
    }
  };
  auto wait_acc = [&]() {
    // one warp polls, the others sleep at a block barrier: eight polling warps halve the rate of the producer's and the
    // issuers' shared-memory operations
    if (warp == 4) mbar_wait(acc_full, 0, a.err, dead, all_ns);
    if (EPI == EPI_QKV_ROPE && cf.rope_bytes) mbar_wait(rope_full, 0, a.err, dead, wait_ns);      // long complete
    epi_sync();
    tc_fence_after();
  };
  if (kDirect && split == 1) {
    // ---- no other CTA contributes: a thread has one weight row of its tile in C token rows at a time, and what it is
    // combined with in the same thread (gate and up) or 16 lanes away (rotary pair)
    if (epi) {
      const int rowi = quarter * 32 + lane;                     // row of the tile
      const int c = EPI == EPI_QKV_ROPE ? (quarter * 16 + (lane & 15)) & (half - 1) : 0, hi_half = (lane >> 4) & 1;
      // the rotary table of the step lies in shared memory, or, when it does not fit beside the rings, in L2
      const float2 *rope = cf.rope_bytes ? reinterpret_cast<const float2 *>(data + cf.rope_off) : a.rope + (size_t)row0 * half;
      wait_acc();
#pragma unroll 1
      for (int t = 0; t < wk.nt; ++t) {
        const int tile = wk.t0 + t;
        const int unit = EPI == EPI_QKV_ROPE ? tile * sc.heads + (sc.heads == 2 ? quarter >> 1 : 0) : 0;    // query, key or value head
#pragma unroll 1
        for (int c0 = half_w * C; c0 < R; c0 += 2 * C) {
          float r[C], rs[C];
          uint32_t row[EPI == EPI_QKV_ROPE ? C : C / 2];            // two rows each, or one row's place in the cache
          load_acc(t, c0, r);
#pragma unroll
          for (int q = 0; q < C / 4; ++q) *reinterpret_cast<float4 *>(rs + 4 * q) = *reinterpret_cast<const float4 *>(s_rs + c0 + 4 * q);
          if (EPI == EPI_QKV_ROPE) {
#pragma unroll
            for (int q = 0; q < C / 4; ++q) *reinterpret_cast<uint4 *>(row + 4 * q) = *reinterpret_cast<const uint4 *>(s_kv + c0 + 4 * q);
          } else {
#pragma unroll
            for (int q = 0; q < C / 8; ++q) *reinterpret_cast<uint4 *>(row + 4 * q) = *reinterpret_cast<const uint4 *>(s_row + c0 + 8 * q);
          }
          auto row_of = [&](int j) { return (int)((row[j >> 1] >> (16 * (j & 1))) & 0xffffu); };       // 0xffff: none
          if (EPI == EPI_LOGITS) {
            const int n = tile * BM + rowi;
            if (n < a.N) {
#pragma unroll
              for (int j = 0; j < C; ++j) {
                const int w = row_of(j);
                if (w != 0xffff) a.logits[(size_t)(row_seq(w) * a.rw.Ms + row_in_seq(w)) * a.N + n] = r[j] * rs[j];
              }
            }
          } else if (EPI == EPI_SWIGLU) {
            // lanes 8 apart hold the gate and the up value of a column of y; each takes half of the token rows
            const bool up = (lane & 8) != 0;
            const int n = tile * (BM / 2) + (rowi >> 4) * 8 + (rowi & 7), m0 = c0 + (up ? C / 2 : 0);
#pragma unroll
            for (int j = 0; j < C; ++j) r[j] *= rs[j];
#pragma unroll
            for (int j = 0; j < C / 2; ++j) {
              const float got = __shfl_xor_sync(0xffffffffu, up ? r[j] : r[j + C / 2], 8);
              const float g = up ? got : r[j], u = up ? r[j + C / 2] : got;
              r[j] = g / (1.f + __expf(-g)) * u;
            }
            bf16 *dst = a.y + (size_t)(row0 + m0) * a.F + n;
            if (n < a.F) {
#pragma unroll
              for (int j = 0; j < C / 2; ++j) {
                const bf16 h = __float2bfloat16_rn(r[j]);
                if (m0 + j < R) {
                  dst[(size_t)j * a.F] = h;
                  dst[(size_t)j * a.F + a.y_plane] = __float2bfloat16_rn(r[j] - __bfloat162float(h));
                }
              }
            }
          } else {
            // queries and keys are rotated at the row's tree position (Section 3.4): y = x cos -+ (other half) sin
#pragma unroll
            for (int j = 0; j < C; ++j) r[j] *= rs[j];
            if (unit < a.H + a.Hkv) {
#pragma unroll
              for (int j = 0; j < C; ++j) {
                const float2 cs = rope[min(c0 + j, R - 1) * half + c];
                const float o = __shfl_xor_sync(0xffffffffu, r[j], 16);
                r[j] = r[j] * cs.x + (hi_half ? o : -o) * cs.y;
              }
            }
            const int col = c + hi_half * half;
            if (unit < a.H) {
              bf16 *dst = a.q + (size_t)(row0 + c0) * a.H * a.dh + unit * a.dh + col;
              const int stride = a.H * a.dh;
#pragma unroll
              for (int j = 0; j < C; ++j) {
                const bf16 h = __float2bfloat16_rn(r[j]);
                if ((int)row[j] != kNoRow) {
                  dst[(size_t)j * stride] = h;
                  dst[(size_t)j * stride + a.q_plane] = __float2bfloat16_rn(r[j] - __bfloat162float(h));
                }
              }
            } else if (unit < a.H + 2 * a.Hkv) {                // the cache stores bf16: one rounding, on store
              const int is_v = unit >= a.H + a.Hkv, kvh = unit - a.H - (is_v ? a.Hkv : 0);
              bf16 *dst = a.kcache + (is_v ? a.kv_stride : 0) + kvh * a.dh + col;
              const size_t stride = (size_t)a.Hkv * a.dh;
#pragma unroll
              for (int j = 0; j < C; ++j) {
                if ((int)row[j] >= 0) dst[(size_t)row[j] * stride] = __float2bfloat16_rn(r[j]);
              }
            }
          }
        }
      }
    }
  } else {
  for (int p0 = 0; p0 < wk.nt; p0 += cf.tp) {
    const int tp = min(cf.tp, wk.nt - p0);
    // the residual rows a warp adds to first, and their gain, are on their way before the contraction is complete
    float4 h0, h1, gain = make_float4(0.f, 0.f, 0.f, 0.f);
    auto residual = [&](int loc, int tl) {
      return __ldcg(reinterpret_cast<const float4 *>(a.h + (size_t)(row0 + min(own0 + loc, R - 1)) * a.d + (wk.t0 + p0 + tl) * BM + lane * 4));
    };
    auto gain_of = [&](int tl) { return load_bf16x4(a.g + (wk.t0 + p0 + tl) * BM + lane * 4); };
    if (epi) {
      if (EPI == EPI_RESIDUAL && n_own > 0) {
        h0 = residual(ew, 0);
        h1 = ew + kEpiWarps < n_own ? residual(ew + kEpiWarps, 0) : residual(ew, min(1, tp - 1));
        if (a.x) gain = gain_of(0);
      }
      if (p0 == 0) wait_acc();
    }
    if (split > 1) {
      // No CTA of the cluster reads its ring, or the previous pass's sums, any more.  With room of their own for the sums
      // the first pass only needs every CTA to have started.
      if (p0 == 0 && cf.red_off) cluster_wait(); else cg::this_cluster().sync();
    } else if (epi && p0 > 0) {
      epi_sync();
    }
    if (epi) {
      const uint32_t mine = base + cf.red_off + (uint32_t)((quarter * 32 + lane) * 4), step = (uint32_t)tp * 512u;
#pragma unroll 1
      for (int tl = 0; tl < tp; ++tl) {
#pragma unroll 1
        for (int c0 = half_w * C; c0 < R; c0 += 2 * C) {
          float r[C];
          load_acc(p0 + tl, c0, r);
#pragma unroll
          for (int g = 0; g < C / 4; ++g) {            // four token rows go to one CTA (tpo is a multiple of four)
            const int m = c0 + 4 * g;
            if (m < R) {
              const int o = (m * cf.inv_tpo) >> 16;
              const uint32_t dst = map_rank(mine + (uint32_t)(((int)rank * cf.tpo + m - o * cf.tpo) * tp + tl) * 512u, (uint32_t)o);
#pragma unroll
              for (int j = 0; j < 4; ++j) st_cluster(dst + j * step, r[4 * g + j]);
            }
          }
        }
      }
      tc_fence_before();
    }
    if (split > 1) cg::this_cluster().sync();
    else if (epi) epi_sync();
    if (!epi) continue;
    const int slice = cf.tpo * tp * BM;            // floats of one k slice's part
    auto sums = [&](int idx) {                     // sum over the k slices, in rank order
      float4 v = *reinterpret_cast<const float4 *>(red + idx);
#pragma unroll 1
      for (int s = 1; s < split; ++s) v = add4(v, *reinterpret_cast<const float4 *>(red + s * slice + idx));
      return v;
    };
    if (EPI == EPI_RESIDUAL) {
      // a warp per (token row, tile), 4 neighbouring columns per lane
      auto finish = [&](int loc, int n0, float4 v, float sq) {
        const int row = s_row[own0 + loc], s = row_seq(row), w = row_in_seq(row);
        if (row == 0xffff) return;
        int xp_row = -1;
        if (a.xp != nullptr) {
          if (a.rw.chains) xp_row = w < a.rw.T ? s * a.rw.T + w : -1;
          else xp_row = w == a.rw.anchor ? s : -1;
        }
        store_residual(a, row0 + own0 + loc, xp_row, n0, v, gain, sq, lane);
      };
      if (n_own <= 4 * kEpiWarps) {                // few rows: one after the other, two residual rows ahead
        int loc = ew, tl = ew < n_own ? 0 : tp;
#pragma unroll 1
        while (tl < tp) {
          int nloc = loc + kEpiWarps, ntl = tl;
          if (nloc >= n_own) { nloc = ew; ++ntl; }
          const float4 v = add4(h0, sums((loc * tp + tl) * BM + lane * 4));
          h0 = h1;
          int l2 = nloc + kEpiWarps, t2 = ntl;
          if (l2 >= n_own) { l2 = ew; ++t2; }
          if (t2 < tp) h1 = residual(l2, t2);
          finish(loc, (wk.t0 + p0 + tl) * BM + lane * 4, v, warp_sq(v));
          if (a.x && ntl != tl && ntl < tp) gain = gain_of(ntl);
          loc = nloc; tl = ntl;
        }
      } else {                                     // a prompt's: four at a time, so that their chains overlap
#pragma unroll 1
        for (int tl = 0; tl < tp; ++tl) {
          const int n0 = (wk.t0 + p0 + tl) * BM + lane * 4;
          if (a.x && tl) gain = gain_of(tl);
#pragma unroll 1
          for (int l0 = ew; l0 < n_own; l0 += 4 * kEpiWarps) {
            float4 v[4];
            float sq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = residual(l0 + u * kEpiWarps, tl);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              v[u] = add4(v[u], sums((min(l0 + u * kEpiWarps, n_own - 1) * tp + tl) * BM + lane * 4));
              sq[u] = v[u].x * v[u].x + v[u].y * v[u].y + v[u].z * v[u].z + v[u].w * v[u].w;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
              for (int u = 0; u < 4; ++u) sq[u] += __shfl_xor_sync(0xffffffffu, sq[u], o);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (l0 + u * kEpiWarps < n_own) finish(l0 + u * kEpiWarps, n0, v[u], sq[u]);
          }
        }
      }
      continue;
    }
    // a warp per (token row, tile), 4 neighbouring columns per lane, or half a warp, 4 rotary or gate and up pairs per lane
    constexpr bool kPairs = EPI == EPI_QKV_ROPE || EPI == EPI_SWIGLU;
    const int loc0 = kPairs ? 2 * ew + (lane >> 4) : ew, dloc = kPairs ? 2 * kEpiWarps : kEpiWarps;
    int loc = loc0, tl = loc0 >= n_own ? tp : 0;
#pragma unroll 1
    while (tl < tp) {
      const int lm = own0 + loc, m = row0 + lm, tile = wk.t0 + p0 + tl, row = EPI == EPI_QKV_ROPE ? s_kv[lm] : s_row[lm], s = row_seq(row), v = row_in_seq(row);
      const float rs = s_rs[lm];
      const int idx = (loc * tp + tl) * BM, rope_row = (cf.rope_bytes ? loc : m) * half;
      loc += dloc;
      if (loc >= n_own) { loc = loc0; ++tl; }
      if (row == (EPI == EPI_QKV_ROPE ? kNoRow : 0xffff)) continue;
      if (EPI == EPI_PSEUDO || EPI == EPI_LOGITS) {
        const int n0 = tile * BM + lane * 4;
        const float4 sum = mul4(sums(idx + lane * 4), rs);
        if (EPI == EPI_PSEUDO) {                   // output column = (map, column); d is a multiple of 128: one map per tile
          const int i = n0 / a.d, o = n0 - i * a.d;
          const float4 r = a.pred_b ? add4(sum, load_bf16x4(a.pred_b + n0)) : sum;
          store_residual(a, act_row(a.rw, s, a.rw.T + (a.rw.chains ? (a.pseudo0 + i) * a.rw.T + v : a.pseudo0 + i)), -1, o, r, load_bf16x4(a.g + o), warp_sq(r), lane);
        } else if (n0 < a.N) {                     // EPI_LOGITS
          float *dst = a.logits + (size_t)(s * a.rw.Ms + v) * a.N + n0;
          if ((a.N & 3) == 0) {
            *reinterpret_cast<float4 *>(dst) = sum;
          } else {
            const float t[4] = {sum.x, sum.y, sum.z, sum.w};
            for (int j = 0; j < 4 && n0 + j < a.N; ++j) dst[j] = t[j];
          }
        }
      } else if (EPI == EPI_SWIGLU) {
        const int e = (lane & 15) * 4, i1 = (e >> 3) * 16 + (e & 7), j0 = tile * (BM / 2) + e;
        if (j0 >= a.F) continue;
        const float4 va = mul4(sums(idx + i1), rs), vb = mul4(sums(idx + i1 + 8), rs);
        const float gg[4] = {va.x, va.y, va.z, va.w}, uu[4] = {vb.x, vb.y, vb.z, vb.w};
        float y[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = gg[j] / (1.f + __expf(-gg[j])) * uu[j];
        uint2 hi, lo;
        split4(y, hi, lo);
        bf16 *dst = a.y + (size_t)m * a.F + j0;
        *reinterpret_cast<uint2 *>(dst) = hi;
        *reinterpret_cast<uint2 *>(dst + a.y_plane) = lo;
      } else {
        const int e = (lane & 15) * 4, hd = e / half, c = e - hd * half;
        const int i1 = hd * a.dh + (c >> 4) * 32 + (c & 15);
        const int unit = tile * sc.heads + hd;     // query, key or value head
        if (unit >= a.H + 2 * a.Hkv) continue;
        const float4 va = mul4(sums(idx + i1), rs), vb = mul4(sums(idx + i1 + 16), rs);
        const float2 *rope = (cf.rope_bytes ? reinterpret_cast<const float2 *>(data + cf.rope_off) : a.rope) + rope_row + c;
        const float4 c0 = *reinterpret_cast<const float4 *>(rope), c1 = *reinterpret_cast<const float4 *>(rope + 2);
        float x1[4] = {va.x, va.y, va.z, va.w}, x2[4] = {vb.x, vb.y, vb.z, vb.w};
        if (unit < a.H + a.Hkv) {        // queries and keys are rotated at the row's tree position (Section 3.4)
          const float co[4] = {c0.x, c0.z, c1.x, c1.z}, si[4] = {c0.y, c0.w, c1.y, c1.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float y1 = x1[j] * co[j] - x2[j] * si[j], y2 = x2[j] * co[j] + x1[j] * si[j];
            x1[j] = y1; x2[j] = y2;
          }
        }
        if (unit < a.H) {
          uint2 h1, l1, h2, l2;
          split4(x1, h1, l1); split4(x2, h2, l2);
          bf16 *dst = a.q + (size_t)m * a.H * a.dh + unit * a.dh + c;
          *reinterpret_cast<uint2 *>(dst) = h1;
          *reinterpret_cast<uint2 *>(dst + half) = h2;
          *reinterpret_cast<uint2 *>(dst + a.q_plane) = l1;
          *reinterpret_cast<uint2 *>(dst + a.q_plane + half) = l2;
        } else {                         // the cache stores bf16: one rounding, on store
          const int is_v = unit >= a.H + a.Hkv, kvh = unit - a.H - (is_v ? a.Hkv : 0);
          if (row >= 0) {
            bf16 *dst = a.kcache + (is_v ? a.kv_stride : 0) + ((size_t)row * a.Hkv + kvh) * a.dh + c;
            *reinterpret_cast<uint2 *>(dst) = round4(x1);
            *reinterpret_cast<uint2 *>(dst + half) = round4(x2);
          }
        }
      }
    }
  }
  }
  tc_fence_before();
  if (dead) *gave_up = 1;
  __syncthreads();
  if (*gave_up) {                // some loads or MMAs may still be under way (otherwise the accumulators were waited for, and they for all)
    if (lane == 0 && warp == 0) { Landing r{full_w, a.err}; drain(r, started, sw_n); }
    if (lane == 0 && warp == 2) {
      Landing r{full_x, a.err};
      drain(r, started, sx_n);
      if (EPI == EPI_QKV_ROPE && cf.rope_bytes) mbar_drain(rope_full, 0, a.err);
    }
    if (lane == 0 && warp == 4) mbar_drain(acc_full, 0, a.err);
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cf.tmem_cols) : "memory");
  }
}

// ---- host side ---------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Tensor maps of bf16 matrices with 64-element (128-byte) inner boxes, 128-byte swizzle, zero fill out of bounds; `rank`
// dimensions from the second on in dims / strides (bytes) / box.  Encoded maps are cached: the same few (pointer, shape)
// pairs recur every step.
struct MapDims { int rank; cuuint64_t dim[5], stride[4]; cuuint32_t box[5]; };
bool make_map(CUtensorMap *m, const void *ptr, const MapDims &d) {
  typedef std::tuple<const void *, cuuint64_t, cuuint64_t, cuuint64_t, cuuint64_t, cuuint64_t, cuuint64_t, cuuint32_t, cuuint32_t> Key;
  static std::map<Key, CUtensorMap> cache;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  const Key key(ptr, d.dim[0], d.dim[1], d.dim[2], d.dim[3], d.dim[4], d.stride[1], d.box[1], d.box[2] * 8u + (cuuint32_t)d.rank);
  auto it = cache.find(key);
  if (it != cache.end()) { *m = it->second; return true; }
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  if (encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)d.rank, const_cast<void *>(ptr), d.dim, d.stride, d.box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  if (cache.size() > 4096) cache.clear();
  cache[key] = *m;
  return true;
}
// weights [N][K] in the tile order of the epilogue
bool weight_map(CUtensorMap *m, int epi, const void *W, uint64_t N, uint64_t K, uint64_t F, uint64_t dh) {
  MapDims d{};
  d.dim[0] = K; d.box[0] = BK;
  if (epi == EPI_SWIGLU) {
    d.rank = 4; d.dim[1] = 8; d.dim[2] = 2; d.dim[3] = F / 8;
    d.stride[0] = K * 2; d.stride[1] = F * K * 2; d.stride[2] = 8 * K * 2;
    d.box[1] = 8; d.box[2] = 2; d.box[3] = 8;
  } else if (epi == EPI_QKV_ROPE) {
    const uint64_t half = dh / 2;
    d.rank = 5; d.dim[1] = 16; d.dim[2] = 2; d.dim[3] = half / 16; d.dim[4] = N / dh;
    d.stride[0] = K * 2; d.stride[1] = half * K * 2; d.stride[2] = 16 * K * 2; d.stride[3] = dh * K * 2;
    d.box[1] = 16; d.box[2] = 2; d.box[3] = (cuuint32_t)(half / 16); d.box[4] = (cuuint32_t)(BM / dh);
  } else {
    d.rank = 2; d.dim[1] = N; d.stride[0] = K * 2; d.box[1] = BM;
  }
  return make_map(m, W, d);
}
// activation planes [planes][plane_rows][K], the first npad rows of all planes per box
bool plane_map(CUtensorMap *m, const void *X, uint64_t planes, uint64_t plane_rows, uint64_t K, uint32_t npad) {
  MapDims d{};
  d.rank = 3; d.dim[0] = K; d.dim[1] = plane_rows; d.dim[2] = planes; d.stride[0] = K * 2; d.stride[1] = plane_rows * K * 2;
  d.box[0] = BK; d.box[1] = npad; d.box[2] = (cuuint32_t)planes;
  return make_map(m, X, d);
}

typedef void (*KernelFn)(const CUtensorMap, const CUtensorMap, const LinArgs, const TileSched, const TileCfg);
template <bool MERGED, bool DEEP, int C, int EPI> KernelFn kernel_tm(int tm) {
  return tm == 1 ? gemm_kernel<1, MERGED, DEEP, C, EPI> : tm == 2 ? gemm_kernel<2, MERGED, DEEP, C, EPI> : gemm_kernel<3, MERGED, DEEP, C, EPI>;
}
template <int EPI> KernelFn kernel_epi(int tm, bool merged, bool deep, bool few) {
  if (!merged) return deep ? kernel_tm<false, true, 16, EPI>(tm) : kernel_tm<false, false, 16, EPI>(tm);
  if (few) return deep ? kernel_tm<true, true, 8, EPI>(tm) : kernel_tm<true, false, 8, EPI>(tm);
  return deep ? kernel_tm<true, true, 16, EPI>(tm) : kernel_tm<true, false, 16, EPI>(tm);
}
KernelFn kernel_of(int epi, int tm, bool merged, bool deep, bool few) {
  switch (epi) {
    case EPI_RESIDUAL: return kernel_epi<EPI_RESIDUAL>(tm, merged, deep, few);
    case EPI_QKV_ROPE: return kernel_epi<EPI_QKV_ROPE>(tm, merged, deep, few);
    case EPI_SWIGLU: return kernel_epi<EPI_SWIGLU>(tm, merged, deep, few);
    case EPI_LOGITS: return kernel_epi<EPI_LOGITS>(tm, merged, deep, few);
    default: return kernel_epi<EPI_PSEUDO>(tm, merged, deep, few);
  }
}

// CTAs that can run at once in clusters of n with one CTA per SM (GPCs hold whole clusters only: 148, 148, 135, 132,
// 130, 132, 105, 120 for n = 1 .. 8 on a B200)
int cluster_ctas(int n) {
  static int cap[9] = {0};
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  if (cap[n] == 0) {
    int dev = 0, sms = 0, k = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
    if (n == 1) { cap[n] = sms; return sms; }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n * 64); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kSmemMax;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    KernelFn fn = kernel_of(EPI_RESIDUAL, 1, true, false, true);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&k, fn, &cfg) != cudaSuccess || k < 1) { cudaGetLastError(); k = std::max(1, sms / n * 3 / 4); }
    cap[n] = k * n;
  }
  return cap[n];
}

Plan cached_plan(const GemmShape &g, int rows, int call_rows) {
  typedef std::tuple<int, int, int, int, int, int, int> Key;
  static std::map<Key, Plan> cache;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  const Key key((int)g.epi * 256 + g.dh, g.N, g.K, g.F, rows, call_rows, g.planes);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  int ctas[9] = {0};
  for (int n = 1; n <= 8; ++n) ctas[n] = cluster_ctas(n);
  const Plan p = make_plan(g, rows, call_rows, ctas);
  if (cache.size() > 4096) cache.clear();
  return cache[key] = p;
}

}  // namespace

int gemm_additions(GemmEpilogue epi, int N, int K, int F, int dh, int R, int planes) { return cached_plan({epi, N, K, F, dh, planes}, R, R).adds; }

bool gemm_tc_available() { return encode_fn() != nullptr; }

cudaError_t launch_gemm(GemmEpilogue epi, const LinArgs &a, bool pdl, cudaStream_t st) {
  if (!encode_fn()) return cudaErrorNotSupported;
  Plan p = cached_plan({epi, a.N, a.K, a.F, a.dh, a.planes}, a.R, a.call_rows);
  if (p.tm == 0 || p.smem > kSmemMax || p.cf.tp < 1 || p.cf.sw < 1 || p.cf.sx < 1 || (!p.cf.by_tile && p.cf.issuers == 2 && ((p.cf.sw | p.cf.sx | p.cf.sets) & 1)))
    return cudaErrorInvalidConfiguration;
  p.cf.pdl = pdl ? 1 : 0;
  p.cf.idesc = instr_desc_m128(p.cf.acc);
  KernelFn fn = kernel_of(epi, p.tm, p.merged != 0, p.cf.sets > 2 || p.cf.planes_side > 2, few_rows(p.cf.rpb));
  static std::map<KernelFn, int> configured;
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!configured[fn]) {
      cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
      if (e != cudaSuccess) return e;
      configured[fn] = 1;
    }
  }
  CUtensorMap tmW, tmX;
  if (!weight_map(&tmW, epi, a.W, (uint64_t)a.N, (uint64_t)a.K, (uint64_t)a.F, (uint64_t)a.dh)) return cudaErrorInvalidValue;
  if (!plane_map(&tmX, a.X, (uint64_t)a.planes, (uint64_t)a.plane_rows, (uint64_t)a.K, (uint32_t)p.cf.npad)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(p.sc.jobs * p.sc.blocks * p.sc.split));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (pdl) { attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization; attr[na++].val.programmaticStreamSerializationAllowed = 1; }
  if (p.sc.split > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = p.sc.split; attr[na].val.clusterDim.y = 1; attr[na].val.clusterDim.z = 1; ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, fn, tmW, tmX, a, p.sc, p.cf);
}

}  // namespace firp
