// The turns of the prefill attention's two softmax groups (head_dim 128), for the kernel and for the
// host-side model of its barriers.
//
// The groups of Q tile 0 and of Q tile 1 take turns in the tiles of an item that both read, over all
// items of a CTA in a row: group 0's first such tile, group 1's, group 0's second, group 1's, ...
// Each turn is a phase of an mbarrier: turn[1] is given by group 0 as it leaves a tile, turn[0] by
// group 1.  A barrier that is waited on by parity holds one phase that was not yet waited for, not two.
// That holds here because every shared tile takes one turn and gives one, whichever item it belongs
// to: group 0 gives the next phase of turn[1] only after it took turn[0], which group 1 gave after
// it took the phase before.  (Q tile 0's first tile of the CTA finds nothing given: it counts as
// taken, `turns_before`.  Group 1's last turn is never taken.)  Nothing waits in a circle: what a group
// waits for was given in a tile that comes earlier in the ring of K/V tiles.
#pragma once

#ifdef __CUDACC__
#define HAM_TURNS_FN __host__ __device__ inline
#else
#define HAM_TURNS_FN inline
#endif

namespace ham {

// Tiles of an item, from its first one, in which the groups take turns; nt0 and nt1 are the tiles that
// Q tile 0 and 1 read (nt1 = 0: no rows; else nt1 >= nt0).
HAM_TURNS_FN int turn_tiles(int nt0, int nt1) { return nt1 > 0 ? nt0 : 0; }

// Turns that the group of Q tile q has behind it when its CTA starts.
HAM_TURNS_FN unsigned turns_before(int q) { return q == 0 ? 1u : 0u; }

}  // namespace ham
