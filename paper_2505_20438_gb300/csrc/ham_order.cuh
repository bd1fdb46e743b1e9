// The order of a prefill call's query blocks, for the plan kernel and for its host test.
//
// The attention's CTAs take blocks from a counter, so the blocks that attend over the most slots come
// first: block j of a sequence with L cached slots and n new rows reaches slot L + min(n, (j + 1) rows a
// block) at the most.  Blocks that reach equally far follow their sequences' order; of one sequence no
// two do.  Each block's place is the number of blocks before it, which every other sequence gives in
// closed form.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define HAM_ORDER_FN __host__ __device__ inline
#else
#define HAM_ORDER_FN inline
#endif

namespace ham {

// Blocks of 2^shift rows that n rows fill.
HAM_ORDER_FN uint32_t query_blocks(uint32_t n, int shift) {
  return (n >> shift) + ((n & ((1u << shift) - 1)) != 0 ? 1u : 0u);
}

// How far block j of a sequence reaches (1 past the last slot).
HAM_ORDER_FN uint32_t block_reach(uint32_t L, uint32_t n, uint32_t j, int shift) {
  const uint32_t rows = (j + 1) << shift;
  return L + (rows < n ? rows : n);
}

// Blocks of a sequence (L, n) that come before a block of another one that reaches `reach`; `first`:
// the sequence comes before the other, so that an equal reach counts too.
HAM_ORDER_FN uint32_t blocks_before(uint32_t L, uint32_t n, uint32_t reach, bool first, int shift) {
  const uint32_t least = reach + (first ? 0u : 1u);  // blocks that reach at least this far
  if (n == 0 || L + n < least) return 0;
  const uint32_t m = query_blocks(n, shift);
  if (least <= L) return m;
  const uint32_t j = (least - L - 1) >> shift;  // the first of them (the last block reaches L + n)
  return m - (j < m ? j : m - 1);
}

}  // namespace ham
