// The V slots behind a request's last token in its last block, which the KV store of a call sets to zero (attention reads whole blocks).
#pragma once
#include "pool.cuh"

// Share `part` of `parts` of a call's (request, KV head) pairs, for warp `warp` of `n_warps`; all lanes take part.  A lane finds the
// place of one pair, then the warp clears the pairs' slots one after the other, up to 15 x 256 contiguous bytes each.  What it clears is
// known before anything has been computed, so every CTA of a projection takes its share while its product runs.  Left to
// the CTAs that own V's columns, behind the product, it took a decode step's q, k, v of 256 tokens from 45 to 80 us on 7B and from 72 to
// 104 on 34B, whose V has 8 heads and as many CTAs.
template <typename Args>
__device__ __forceinline__ void clear_v_tails(const Args& a, int part, int parts, int warp, int n_warps) {
  const int lane = threadIdx.x & 31, n_items = a.n_req * a.n_kv;
  for (int i0 = part + parts * 32 * warp; i0 < n_items; i0 += parts * 32 * n_warps) {
    const int i = i0 + parts * lane;
    unsigned char* at = nullptr;
    int n = 0;
    if (i < n_items) {
      const int r = i / a.n_kv, h = i - r * a.n_kv;
      const int beg = a.req_indptr[r], end = a.req_indptr[r + 1], pos = a.prefix_lens[r] + (end - beg) - 1;
      if (end > beg && end <= a.n_tokens && pos >= 0) {       // (the rows' own look-up raises the flags for what is out of range)
        const int entry = pos / a.bt, slot = pos - entry * a.bt, tab = a.tbl_indptr[r];
        const uint32_t blk = entry < a.tbl_indptr[r + 1] - tab ? a.tbl[tab + entry] : a.pv.n_blocks;
        if (blk < a.pv.n_blocks) {
          at = a.pv.slab + (size_t)blk * a.pv.block_bytes + ((size_t)(a.n_kv + h) * a.bt + slot + 1) * (FL_HEAD_DIM * 2);
          n = (a.bt - 1 - slot) * (FL_HEAD_DIM * 2 / 16);
        }
      }
    }
    for (uint32_t left = __ballot_sync(0xffffffffu, n > 0); left; left &= left - 1) {
      const int src = __ffs(left) - 1;
      uint4* const p = reinterpret_cast<uint4*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(at), src));
      const int m = __shfl_sync(0xffffffffu, n, src);
      for (int k = lane; k < m; k += 32) p[k] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
}
