// The base projection with the LoRA branch folded in, for batches of few tokens (see lora_skinny.cu).
#pragma once
#include "pool.cuh"
#include "sgmv.cuh"

namespace skinny {

constexpr int MAX_TOKENS = 256;      // two row tiles of 128
constexpr int MAX_LIN = 3;

struct Args {
  PoolView pv;
  const __nv_bfloat16* v;            // shrink result, scaled: [projection][token][rmax]
  int rmax;
  const int32_t* seg_indptr;
  const int32_t* lora_ids;
  int n_seg, n_tokens, d_in, n_mats;
  __nv_bfloat16* y[MAX_LIN];
  int d_out[MAX_LIN], mat_index[MAX_LIN];
  int kv_side[MAX_LIN];              // -1 = rows go to y, 0 = K, 1 = V rows of the requests' pool blocks
  const int32_t* req_indptr;
  const int32_t* tbl_indptr;
  const uint32_t* tbl;
  const int32_t* prefix_lens;
  int n_req, n_kv, bt;
};

// Whether `launch` is the faster way for a call (n_seg = 0: no adapters).
bool serves(const fl_pool* p, const int* d_out, int n_mats, int d_in, int n_tokens, int n_seg, int rank_max);

// What `launch` will take for these arguments.
sgmv::Follower footprint(const fl_pool* p, const Args& a);

// y = x W + (scaled x A) B for n_tokens <= MAX_TOKENS.  With n_seg > 0 the shrink that writes v must be the launch right
// before this one on the stream.
int launch(fl_pool* p, const Args& a, const void* x, const void* const* w, cudaStream_t st);

}  // namespace skinny
