// The ring of load stages of a tensor-core kernel, as its producer sees it (plain C++, so that it can be run on the host too).
#pragma once

#ifdef __CUDACC__
#define IVIT_RING_FN __host__ __device__ __forceinline__
#else
#define IVIT_RING_FN inline
#endif

namespace ivit {

// Waits for the loads that the producer has requested and nobody may have waited for: the last one of every stage.  (Those
// before it on the same stage have landed, or the stage would not have been free.)  wait(stage, parity) waits for the
// phase of the stage's barrier that the load completes.
template <class Wait>
IVIT_RING_FN void drain_ring(int requested, int stages, Wait wait) {
  for (int kb = requested > stages ? requested - stages : 0; kb < requested; ++kb) wait(kb % stages, (unsigned)(kb / stages) & 1u);
}

}  // namespace ivit
