// The order in which the roles of the tcgen05 prefill attention kernel wait for K and V tiles, issue MMAs on them and give their
// slots back, apart from the kernel so that it can be run on the host against a model of the barriers.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ROLE_FN __host__ __device__ __forceinline__
#else
#define ROLE_FN inline
#endif

namespace attn {

// K and V have rings of their own: a barrier's test is true for the phase before last too, so whoever tests a slot must have seen every
// phase of it.  In one ring of five slots, where K and V take turns in every slot, the issuer of the scores saw every other phase, and
// with one query tile in the unit nothing but the order in which the copies landed kept it from a slot that still waited for its K.
// K is read a step ahead of V and given back a step earlier, so V has the third slot: attention of 64 prompts of U{128..1024} tokens, half
// of them cached, 7B 270.4 us with the one ring, 269.6 with 2 and 3 slots, 274.6 with 3 and 2; 4 x 1024 new tokens behind 3072, 34B 371.5,
// 371 and 371.
constexpr int K_SLOTS = 2, V_SLOTS = 3;

template <int N>
struct RingPos {          // a slot and the parity of its current use
  int s = 0;
  uint32_t ph = 0;
  ROLE_FN RingPos next() const {
    RingPos r;
    r.s = s + 1 == N ? 0 : s + 1;
    r.ph = s + 1 == N ? ph ^ 1u : ph;
    return r;
  }
};

// Producer: K_0, V_0, K_1, V_1, ... of a unit.  pages(j) looks the tile's pages up; fill_k and fill_v wait until the slot is free (its
// phase of the use before: parity ph ^ 1, over at once for the first) and load.
template <typename K, typename V, typename Pages, typename FillK, typename FillV>
ROLE_FN bool load_tiles(int n_kt, K& k, V& v, Pages pages, FillK fill_k, FillV fill_v) {
  for (int j = 0; j < n_kt; ++j) {
    pages(j);
    if (!fill_k(k)) return false;
    k = k.next();
    if (!fill_v(v)) return false;
    v = v.next();
  }
  return true;
}

// An issuer whose wait gave up leaves at once and gives nothing back: the copies into its slots may still be on their way, and the producer
// would arm a barrier whose phase is open, which the draining behind a wait that gave up (giveup.cuh) could not make out.

// Issuer of the scores S = Q_X K_j^T of both tiles, nA and nB steps of n_kt: ph_free is the parity of the score tile before, which its
// softmax warps have to have taken.
template <typename K, typename Full, typename Free, typename Issue, typename Release, typename ReleaseQ>
ROLE_FN bool issue_scores(int n_kt, int nA, int nB, K& k, uint32_t& ph_free, Full full, Free free, Issue issue, Release release, ReleaseQ release_q) {
  for (int j = 0; j < n_kt; ++j, k = k.next()) {
    if (!full(k)) return false;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      if (j >= (x == 0 ? nA : nB)) continue;
      if (!free(ph_free)) return false;
      ph_free ^= 1u;
      issue(x, k);
    }
    release(k);
  }
  release_q();
  return true;
}

// Issuer of O_X += P_X V_j of one tile, n steps of n_kt.  P of a step comes in two halves of 64 keys, and the product of the first runs
// while the softmax is at the last quarter of its exponentials.  A tile that has no part in a step waits for its V all the same: its share
// in the slot's release would be ahead by a phase otherwise.
template <typename V, typename Full, typename Part, typename Issue, typename Done, typename Release>
ROLE_FN bool issue_pv(int n_kt, int n, V& v, uint32_t& ph_p, Full full, Part part, Issue issue, Done done, Release release) {
  for (int j = 0; j < n_kt; ++j, v = v.next()) {
    if (!full(v)) return false;
    if (j < n) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!part(h, ph_p)) return false;
        issue(h, v, j == 0);
      }
      ph_p ^= 1u;
      done();
    }
    release(v);
  }
  return true;
}

// A look at a barrier, a test or a bounded wait, by all lanes of a warp that go on to tensor-memory instructions: those are aligned, so the
// lanes have to agree (each looks for itself, and the phase may end in between), and what the phase's MMAs touched is only theirs behind a
// tcgen05 fence.
template <typename Look, typename Vote, typename Fence>
ROLE_FN bool seen_by_all(Look look, Vote vote, Fence fence) {
  if (!vote(look())) return false;
  fence();
  return true;
}

}  // namespace attn
