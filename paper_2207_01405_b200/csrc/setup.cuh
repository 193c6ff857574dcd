// The end of a tensor-core kernel's set-up where one warp goes ahead of the others (plain C++, so that it can be run on the
// host too).
#pragma once

#ifdef __CUDACC__
#define IVIT_SETUP_FN __host__ __device__ __forceinline__
#else
#define IVIT_SETUP_FN inline
#endif

namespace ivit {

// The next kernel of the stream may be scheduled once one thread of every CTA has triggered it.  A CTA of it that shares the SM
// then takes tensor memory and holds it until this grid has ended, and tcgen05.alloc waits without a limit: a CTA that
// triggered before its own allocation could wait for columns that the next kernel keeps while it waits for this one.
// So the warp that goes ahead to its loads only arrives at the set-up barrier and leaves the trigger to those behind it.
template <class Cta>
IVIT_SETUP_FN void end_of_setup(const Cta& cta, bool ahead) {
  if (ahead) {
    cta.arrive();
  } else {
    cta.sync();
    cta.trigger();
  }
}

}  // namespace ivit
