// The order in which the warps of a pipeline wait for one another, apart from the device code that waits: plain C++, so that
// it can be run on the host with any timing.
#pragma once

#ifdef __CUDACC__
#define FIRP_HD __host__ __device__ __forceinline__
#else
#define FIRP_HD inline
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

}  // namespace firp
