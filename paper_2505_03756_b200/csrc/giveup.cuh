// What is left to do when a bounded wait has given up, apart from the kernels so that it can be run on the host against a model of
// the barriers.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define GIVEUP_FN __host__ __device__ __forceinline__
#else
#define GIVEUP_FN inline
#endif

namespace giveup {

// A result that is a sum over the CTAs of a cluster holds only if every one of them has its part.  A CTA that has none tells the
// others, before the barrier behind which they add the parts up; one that has been told stores nothing.
template <typename Tell>
GIVEUP_FN void tell_cluster(bool ok, int rank, int n_ctas, Tell tell) {
  for (int p = 0; !ok && p < n_ctas; ++p)
    if (p != rank) tell(p);
}
GIVEUP_FN bool may_store(bool ok, int told) { return ok && told == 0; }

}  // namespace giveup
