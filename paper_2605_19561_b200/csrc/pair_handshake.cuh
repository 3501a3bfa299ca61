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
  return tile < total_tiles - accs * npairs;
}

// Sleeps until `clock` has reached `until`, at most `tries` times: a wait for a time has a limit of its own, like one for a
// barrier, so that it ends whatever the counter does (a CTA that is moved to another SM reads another one).
template <typename Clock, typename Sleep>
TORQ_HD void paced_wait(long long until, int tries, Clock clock, Sleep sleep) {
  for (; tries > 0 && clock() < until; --tries) sleep();
}

}  // namespace torq
