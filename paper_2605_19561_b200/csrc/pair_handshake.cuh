// Rules of the CTA-pair kernels that need no device: plain functions, so that a host compiler can check them.
#pragma once
#if defined(__CUDACC__)
#define TORQ_HD __host__ __device__ __forceinline__
#else
#define TORQ_HD inline
#endif

namespace torq {

// Whether the epilogue tells the issuer that it has read the accumulator of `tile`.  A pair walks the tiles tile, tile + npairs,
// ... and gives them its `accs` accumulators in turn, so the issuer waits for that arrival `accs` tiles later, and only if it has
// such a tile.  An arrival that nobody waits for would cross to the leader's shared memory with nothing to keep that CTA
// there: the kernels' last cluster barrier is relaxed and orders no arrivals.
TORQ_HD bool accumulator_is_waited_for(int tile, int npairs, int accs, int total_tiles) {
  return tile + accs * npairs < total_tiles;
}

// Sleeps until `cycles` have passed since `since`, by a counter that wraps around.  Whatever the counter does, the wait ends: it
// goes on only while the counter shows a time within `cycles` after `since`, so a counter that jumps (a CTA that is moved to
// another SM reads another one), back or ahead, ends it.
template <typename Clock, typename Sleep>
TORQ_HD void paced_wait(unsigned since, unsigned cycles, Clock clock, Sleep sleep) {
  while (clock() - since < cycles) sleep();
}

}  // namespace torq
