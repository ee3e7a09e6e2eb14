// The order in which the warps of a pipeline wait for one another, apart from the device code that waits: plain C++, so that
// it can be run on the host with any timing.
#pragma once

#ifndef FIRP_HD
#ifdef __CUDACC__
#define FIRP_HD __host__ __device__ __forceinline__
#else
#define FIRP_HD inline
#endif
#endif

namespace firp {

// "Of tile i": the barrier of a ring and the parity of its phase that completes with that tile.  A wait by parity tells a
// phase only from its neighbours, so a ring must be deep enough that the phase after the awaited one cannot complete
// before the waiter has looked: whatever completes it has to depend on something the waiter does afterwards.
struct TilePhase { int bar; unsigned parity; };

// tree_attn_rows_kernel (attn_tc.cu).  K and V tiles: the next phase is tile i + 2, loaded into the buffer that tile i's MMAs
// have given back.
constexpr int kRowsKvRing = 2;
FIRP_HD TilePhase rows_kv(int i) { return TilePhase{i % kRowsKvRing, (unsigned)(i / kRowsKvRing) & 1u}; }
// S, P and O of tile i, three barriers each, as there are three score buffers: the next phase is tile i + 3, whose S is issued
// only after O of tile i is complete and seen by the issuer of S.  (With two barriers for O the issuer of S, which waits for K
// of tile i + 3 before it looks for O of tile i, could find O of tile i + 2 there, which depends on nothing it has yet to issue.)
constexpr int kRowsSpoRing = 3;
FIRP_HD TilePhase rows_spo(int i) { return TilePhase{i % kRowsSpoRing, (unsigned)(i / kRowsSpoRing) & 1u}; }

// A producer: loads 0 .. n - 1 go, in order, into a ring of `depth` slots.  It gives up with the first slot that does not come
// free in time: a load into it would be counted on a barrier whose phase is still open.  Returns the number of loads started.
//   bool ring.free(u, slot, parity)    bounded wait for the slot's phase of that parity; false: it ran out
//   void ring.load(u, slot)            starts load u
template <class Ring> FIRP_HD int produce(Ring &ring, int n, int depth) {
  int u = 0, slot = 0;
  unsigned parity = 1;
  for (; u < n && ring.free(u, slot, parity); ++u) {
    ring.load(u, slot);
    if (++slot == depth) { slot = 0; parity ^= 1u; }
  }
  return u;
}
// The last of n loads started have landed, oldest first.  After a wait that ran out nobody else may have looked, and a copy must
// not outlive the memory it writes to, which the next block on the SM may own.
//   void ring.landed(slot, parity)     bounded wait, under a limit of its own, for the slot's phase of that parity
template <class Ring> FIRP_HD void drain(Ring &ring, int n, int depth) {
  for (int v = n > depth ? n - depth : 0; v < n; ++v) ring.landed(v % depth, (unsigned)(v / depth) & 1u);
}

}  // namespace firp
