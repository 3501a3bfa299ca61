// What kernels ask the L2 for while the kernel before still runs: rules that need no device, as plain functions that a host compiler can
// check.  A request moves nothing to an SM; it can only ask for too little, for something twice, or for what is not there.
#pragma once
#if defined(__CUDACC__)
#define TORQ_ASK_HD __host__ __device__ __forceinline__
#else
#define TORQ_ASK_HD inline
#endif

namespace torq {

// `bytes` of contiguous memory dealt over the 32 lanes of a warp in whole 128-byte lines: the first byte of a lane's share, and how
// many it has (0: none).
TORQ_ASK_HD int lane_share_first(int lane, int bytes) { return lane * (((bytes + 31) / 32 + 127) / 128 * 128); }
TORQ_ASK_HD int lane_share_bytes(int lane, int bytes) {
  const int first = lane_share_first(lane, bytes), next = lane_share_first(lane + 1, bytes);
  return first >= bytes ? 0 : (next < bytes ? next : bytes) - first;
}

// K step of X that the pair of CTAs with this first tile asks for.  The pairs of one row tile have its columns from the first on, so
// each asks for another step and together for the first ones; a narrow tile lies behind the row's wide ones.
TORQ_ASK_HD int x_step_of_tile(int first_column, bool narrow) { return first_column / (narrow ? 192 : 256); }

}  // namespace torq
