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

constexpr uint32_t DRAIN_POLLS = 1u << 16;       // per barrier

// Parity of the last phase that was armed on slot s of a ring of ns barriers whose slots were armed `fills` times in ring order; -1
// for none.  (A test of the other parity is true at once, on a barrier whose copies are still on their way too.)
GIVEUP_FN int last_parity(long long fills, int ns, int s) { return s < fills ? (int)(((fills - 1 - s) / ns) & 1) : -1; }

// Waits until the copies behind every armed barrier of a ring have landed: they write into this CTA's shared memory, which must not
// be given up before.  A slot is armed again only after the phase before it was over, so the last phase is the one to wait for.
// landed(slot, parity) polls once.  False if a bound ran out.
template <typename Landed>
GIVEUP_FN bool drain(long long fills, int ns, Landed landed) {
  bool all = true;
  for (int s = 0; s < ns; ++s) {
    const int parity = last_parity(fills, ns, s);
    if (parity < 0) continue;
    uint32_t i = 0;
    while (i < DRAIN_POLLS && !landed(s, (uint32_t)parity)) ++i;
    all = all && i < DRAIN_POLLS;
  }
  return all;
}

// A ring whose barriers, in the first CTA of a pair, count the bytes that both CTAs bring, each into its own memory.  When the two
// have stopped at different stages, the phases behind the shorter one's are made to end with the other's half: armed(f) has armed
// stage f for both halves, and only the first CTA's is coming: counts the missing half as arrived; arm(f) arms it for the second
// CTA's half alone.  Returns the stages armed.
template <typename Arm, typename Complete>
GIVEUP_FN long long settle_pair(long long mine, long long other, int ns, Arm arm, Complete complete) {
  for (long long f = other; f < mine; ++f) complete((int)(f % ns));
  for (long long f = mine; f < other; ++f) arm((int)(f % ns));
  return mine > other ? mine : other;
}

}  // namespace giveup
