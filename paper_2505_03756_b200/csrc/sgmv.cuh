// The shrink half of the segmented LoRA projection, for kernels that consume its partial sums themselves.
#pragma once
#include "pool.cuh"

namespace sgmv {

struct ShrinkInfo {
  int ksplit;   // slices of d_in whose partial sums have to be added
  int rmax;     // row pitch of the partial sums (16, 32 or 64: the pool's highest rank rounded up)
  bool final;   // slices added, scaled, rounded to bf16 as the expand product takes them, [projection][token][rmax]
};

struct Follower {      // the kernel that waits for v with all its CTAs: how many, in clusters of how many, and the shared memory of one
  int ctas, cluster;
  uint32_t smem;
};

// v = x A_i per segment for the listed projections (which share x): unscaled fp32 partial sums written to
// workspace as [projection][slice][token][rmax], or the final form; workspace sized by fl_lora_sgmv_workspace(n_tokens, n_mats).
// Rows of segments without an adapter are left untouched.
int shrink(fl_pool* p, const fl_bf16* x, const int* mat_indices, int n_mats, const int32_t* seg_indptr,
           const int32_t* lora_ids, int n_seg, int n_tokens, float scale, void* workspace, size_t workspace_bytes, fl_stream stream,
           ShrinkInfo* info);
// The same, always in its final form.
// Tiles of 16 tokens whatever the segments' lengths, each of which reads its adapter's rows again: for batches of up to a few hundred
// tokens, and beyond for short segments.  `next` is the kernel behind, null where that one has CTAs on all SMs anyway.
int shrink_scaled(fl_pool* p, const fl_bf16* x, const int* mat_indices, int n_mats, const int32_t* seg_indptr,
                  const int32_t* lora_ids, int n_seg, int n_tokens, float scale, void* workspace, size_t workspace_bytes,
                  fl_stream stream, ShrinkInfo* info, const Follower* next);

#ifdef __CUDACC__
// Token tile `tile` (tiles of tm tokens, counted over segments that carry an adapter, or over all segments) -> segment and
// token range.  Every warp evaluates it redundantly with a warp scan over 32 segments at a time.
__device__ __forceinline__ bool find_tile(const int tm, const int32_t* __restrict__ seg_indptr, const int32_t* __restrict__ lora_ids,
                                          int n_seg, int tile, int& seg, int& tok0, int& tok1, bool all_segments = false) {
  const int lane = threadIdx.x & 31;
  int base = 0;
  for (int s0 = 0; s0 < n_seg; s0 += 32) {
    const int s = s0 + lane;
    int lo = 0, hi = 0, nt = 0;
    if (s < n_seg) {
      lo = seg_indptr[s];
      hi = seg_indptr[s + 1];
      if ((all_segments || lora_ids[s] >= 0) && hi > lo) nt = (hi - lo + tm - 1) / tm;
    }
    int incl = nt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (tile < base + total) {
      const int first = base + incl - nt;
      const bool mine = nt > 0 && tile >= first && tile < first + nt;
      const int src = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
      const int k = tile - __shfl_sync(0xffffffffu, first, src);
      seg = s0 + src;
      tok0 = __shfl_sync(0xffffffffu, lo, src) + k * tm;
      tok1 = min(tok0 + tm, __shfl_sync(0xffffffffu, hi, src));
      return true;
    }
    base += total;
  }
  return false;
}

template <int TM>
__device__ __forceinline__ bool find_tile(const int32_t* __restrict__ seg_indptr, const int32_t* __restrict__ lora_ids,
                                          int n_seg, int tile, int& seg, int& tok0, int& tok1, bool all_segments = false) {
  return find_tile(TM, seg_indptr, lora_ids, n_seg, tile, seg, tok0, tok1, all_segments);
}

// Start of rank-row `row` of a stream (class table entry tab, first row row0, rows per block rpb, row width).
__device__ __forceinline__ const unsigned char* lora_row(const PoolView& pv, uint32_t table_off, uint32_t tab,
                                                         uint32_t row0, uint32_t rpb, int width, int row, bool& ok) {
  const uint32_t g = row0 + (uint32_t)row;
  const uint32_t blk = pv.tables[table_off + tab + g / rpb];
  if (blk >= pv.n_blocks) {
    atomicOr(pv.flags, (uint32_t)FLAG_BAD_BLOCK);
    ok = false;
    return pv.slab;
  }
  ok = true;
  return pv.slab + (size_t)blk * pv.block_bytes + (size_t)(g % rpb) * 2 * (size_t)width;
}

// The starts of a thread's COUNT rank-rows, of one or several streams: find(i, entry, offset) gives row i's table entry and its offset in
// the block, or false where there is no row.  All entries are asked for before any is looked at (one after the other, twelve of them took
// 3.5 us).  ok[i] = false where there is no row, or none to be read; its start is the slab's.
template <int COUNT, typename Find>
__device__ __forceinline__ void lora_rows(const PoolView& pv, Find find, const unsigned char* (&start)[COUNT], bool (&ok)[COUNT]) {
  uint32_t blk[COUNT], off[COUNT];
#pragma unroll
  for (int i = 0; i < COUNT; ++i) {
    uint32_t entry = 0;
    off[i] = 0;
    ok[i] = find(i, entry, off[i]);
    blk[i] = ok[i] ? pv.tables[entry] : 0u;
  }
  bool bad = false;
#pragma unroll
  for (int i = 0; i < COUNT; ++i) {
    if (blk[i] >= pv.n_blocks) {
      bad = true;
      ok[i] = false;
    }
    start[i] = ok[i] ? pv.slab + (size_t)blk[i] * pv.block_bytes + off[i] : pv.slab;
  }
  if (bad) atomicOr(pv.flags, (uint32_t)FLAG_BAD_BLOCK);
}
// Table entry and byte offset inside the block of rank-row `row` of a stream (arguments as for lora_row).
__device__ __forceinline__ void lora_row_at(uint32_t table_off, uint32_t tab, uint32_t row0, uint32_t rpb, int width, int row, uint32_t& entry, uint32_t& off) {
  const uint32_t g = row0 + (uint32_t)row, q = g / rpb;
  entry = table_off + tab + q;
  off = (g - q * rpb) * 2u * (uint32_t)width;
}

#endif

// The same shrink on the 5th-generation tensor cores for long segments (tiles of 128 tokens, x by TMA, adapter rows
// by cp.async, accumulator in TMEM), always in its final form.  The slices of d_in are the CTAs of a cluster.
constexpr int TC_MAX_SLICES = 8;
struct TcShrinkArgs {
  PoolView pv;
  __nv_bfloat16* v16;      // [projection][token][rmax]
  float scale;
  int ksplit, n_mats;
  int mat_index[3];
  const int32_t* seg_indptr;
  const int32_t* lora_ids;
  int n_seg, n_tokens, d_in;
};
int tc_slices(const fl_pool* p, int n_seg, int n_tokens, int d_in, int rmax, int n_mats);      // slices of d_in to take
int shrink_tc(fl_pool* p, const TcShrinkArgs& a, const void* x, int rmax, cudaStream_t st);

}  // namespace sgmv
