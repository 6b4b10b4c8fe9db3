// How a consumer warp goes through the stages of a shared-memory ring.  Plain C++,
// so that the rule also compiles on the host.
#pragma once

#ifdef __CUDACC__
#define KVQ_RING_FN __device__ __forceinline__
#else
#define KVQ_RING_FN inline
#endif

namespace kvq {
namespace stream {

// Passes the stages from `next` up to but not including `stage`: waits for each
// one's copies and leaves it.  A barrier is waited for by parity, which tells a phase
// only from its neighbours, so a warp goes through every stage, whether or not it
// has a block in it: a stage is refilled once all warps have left it, and no warp is
// ever more than one phase away from a barrier.  (A warp that skipped a stage could
// take the phase before the skipped one for the one it waits for.)  False when a
// wait gives up.
template <class Wait, class Leave>
KVQ_RING_FN bool ring_pass(int& next, int stage, Wait wait, Leave leave) {
  for (; next < stage; ++next) {
    if (!wait(next)) return false;
    leave(next);
  }
  return true;
}

}  // namespace stream
}  // namespace kvq
