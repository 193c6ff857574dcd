// Hardware barriers between the control warp of attention_short_kernel and its Shiftmax threads (plain C++, so that the
// protocol can be compiled and run on the host too).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define IVIT_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define IVIT_HOST_DEVICE inline
#endif

namespace ivit {

constexpr int kBarScores = 6;   // scores and work item are there
constexpr int kBarOutput = 7;   // the output is there

// The control warp after a wait that ran out.  `done` items have been released twice; of the item at which the wait ran out
// the scores may have been released (scores_out).  The Shiftmax threads, told by a flag, walk on through both barriers of
// every item without work, and the control warp walks with them: it takes part in each barrier as one that waits.  (Arriving
// without waiting it would run ahead, and its second arrival would count for the phase that is still open: that phase
// ends a warp short, and the last one never ends.)
template <class Barriers>
IVIT_HOST_DEVICE void walk_out(Barriers bars, uint32_t done, uint32_t n_items, bool scores_out) {
  for (uint32_t n = done; n < n_items; ++n) {
    if (n > done || !scores_out) bars.sync(kBarScores);
    bars.sync(kBarOutput);
  }
}

}  // namespace ivit
