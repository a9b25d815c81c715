// Segmented LoRA projection y += scale * (x A_i) B_i over adapter rank-rows stored in pool blocks
// (Eq. 1, Eq. 2; the segmented batching of Section 2.1).
//
// Two kernels.  shrink: v = x A_i for a tile of tokens of one segment and a slice of d_in, adapter
// rows fetched through the adapter's block table with 16-byte cp.async, bf16 mma.sync with fp32
// accumulation, partial sums written to scratch [mat][k-slice][token][RMAX].  expand: sums the
// partials, scales, rounds v to bf16, multiplies by the B rows of a column range (fp32 accumulation),
// rounds that LoRA term to bf16 into a tile of its own and adds it to the staged y rows with packed
// bf16 adds while the rows go out as coalesced 16-byte stores: y_out = rn(y + rn(term)).  The term is a
// small correction of y, so its own 2^-9 roundings stay far below y's final rounding.  Both kernels are
// bound by memory traffic (x and y rows for long segments, adapter rows for decode-sized segments) and by
// the instructions spent per byte, not by the contraction.
#include <algorithm>
#include "mma_utils.cuh"
#include "pool.cuh"
#include "sgmv.cuh"

namespace {

using sgmv::find_tile;
using sgmv::lora_row;

constexpr int SG_THREADS = 128;
constexpr int KS = 64;            // d_in elements per shrink pipeline stage (128-byte rows)
constexpr int SH_STAGES = 4;
// Tiles of 16 tokens behind which the final form is wanted: a CTA's slice is 8 to 27 stages, each 0.5 us after the one before with four in
// flight.  With 8 or 12 in flight (rank 64) it takes half as long, but its CTAs take twice the shared memory, and the projection's CTAs, which
// are on their way to W meanwhile, wait for the SMs: `deeper` decides.
constexpr int deep_stages(int rmax) { return rmax == 64 ? 12 : 8; }
constexpr int NSUB = 128;         // y columns per expand sub-tile (256-byte rows)
constexpr int EXPAND_COLS_MIN = 512, EXPAND_COLS_MAX = 2048;   // y columns per expand CTA: picked per call
constexpr int KSPLIT_MAX = 8;

struct SgmvArgs {
  PoolView pv;
  const __nv_bfloat16* x;
  __nv_bfloat16* y[FL_MAX_MATS];
  int mat_index[FL_MAX_MATS];
  int n_mats;
  const int32_t* seg_indptr;
  const int32_t* lora_ids;
  int n_seg, n_tokens;
  float scale;
  float* v;        // [n_mats][ksplit][n_tokens][RMAX]
  __nv_bfloat16* v16;   // the scaled sum in bf16, [n_mats][n_tokens][RMAX], instead of v: tiles of 16 tokens, or the tcgen05 shrink; or null
  int ksplit;
  int tc_ksplit;     // slices of d_in for the tcgen05 shrink of long segments (0 = not applicable)
  int expand_cols;   // y columns one expand CTA covers
  int d_out[FL_MAX_MATS];
  // K / V projections whose result goes straight into the requests' pool blocks instead of back into y
  // (kv_side[j] = 0: K, 1: V, -1: y updated in place); then segments without an adapter are tiled too
  int kv_side[FL_MAX_MATS];
  int all_segments;
  const int32_t* req_indptr;
  const int32_t* tbl_indptr;
  const uint32_t* tbl;
  const int32_t* prefix_lens;
  int n_req, n_kv, bt;
  uint32_t bt_inv;     // 2^32 / bt, rounded up
};

// Eight bf16 sums (round to nearest even each) of two 16-byte chunks.
__device__ __forceinline__ uint4 add_bf16x8(uint4 a, uint4 b) {
  uint4 r;
  const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
  const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
  __nv_bfloat162* pr = reinterpret_cast<__nv_bfloat162*>(&r);
#pragma unroll
  for (int i = 0; i < 4; ++i) pr[i] = __hadd2(pa[i], pb[i]);
  return r;
}

// the pipeline's stages, and for short tiles (which reuse it) the sums of the four warps
__host__ __device__ constexpr int shrink_pipe_bytes(int tm, int rmax, int stages) { return stages * (tm + rmax) * 128; }

template <int TM, int RMAX, int STAGES>
__global__ void __launch_bounds__(SG_THREADS) sgmv_shrink_kernel(const SgmvArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_wait();                 // x may come from the kernel right before this one
  pdl_launch_dependents();    // the expand may start its look-ups and first loads while this grid drains
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int j = blockIdx.x % a.n_mats;
  const int tile = blockIdx.x / a.n_mats;
  const int split = blockIdx.y;
  int seg, tok0, tok1;
  if (!find_tile<TM>(a.seg_indptr, a.lora_ids, a.n_seg, tile, seg, tok0, tok1, a.all_segments != 0)) return;
  const int lid = a.lora_ids[seg];
  if (lid < 0) return;
  if ((uint32_t)lid >= a.pv.dir_cap || a.pv.dir[lid].rank <= 0 || a.mat_index[j] >= a.pv.dir[lid].n_mats) {
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
    return;
  }
  const LoraEntry* e = a.pv.dir + lid;
  const LoraMat lm = e->mats[a.mat_index[j]];
  const int rank = min(e->rank, RMAX);
  // an adapter of a higher rank than this instantiation covers (registered after the launch was recorded
  // into a graph): its extra rank-rows are left out, and the status word says so
  if (e->rank > RMAX && tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
  const uint32_t table_off = e->table_off;
  const bool clustered = TM == 16 && a.v16 && a.ksplit > 1;
  if (clustered) cluster_arrive();       // "this CTA is running"; the others wait for it before they store into its memory
  const int d_in = lm.d_in;
  const int kchunk = ((d_in + a.ksplit * KS - 1) / (a.ksplit * KS)) * KS;
  const int kb = split * kchunk, ke = min(d_in, kb + kchunk);
  const int n_it = ke > kb ? (ke - kb + KS - 1) / KS : 0;

  constexpr int XR = TM / 16;      // x rows per thread per stage
  constexpr int AR = RMAX / 16;    // adapter rows per thread per stage
  constexpr int STAGE_BYTES = (TM + RMAX) * 128;
  const int crow = tid >> 3, cchunk = tid & 7;
  const __nv_bfloat16* xrow[XR];
  bool xok[XR];
#pragma unroll
  for (int i = 0; i < XR; ++i) {
    const int t = tok0 + crow + 16 * i;
    xok[i] = t < tok1;
    xrow[i] = a.x + (size_t)(xok[i] ? t : tok0) * d_in;
  }
  const unsigned char* arow[AR];
  bool aok[AR];
  sgmv::lora_rows<AR>(a.pv, [&](int i, uint32_t& entry, uint32_t& off) {
    const int r = crow + 16 * i;
    if (r >= rank) return false;
    sgmv::lora_row_at(table_off, lm.a_tab, lm.a_row0, lm.a_rpb, d_in, r, entry, off);
    return true;
  }, arow, aok);
  const uint32_t sbase = smem_u32(smem);
  auto load_stage = [&](int it, int st) {
    const int kk = kb + it * KS + cchunk * 8;
    const bool kok = kk < ke;
    const uint32_t xs = sbase + st * STAGE_BYTES, as = xs + TM * 128;
#pragma unroll
    for (int i = 0; i < XR; ++i) cp_async16(xs + swz(crow + 16 * i, cchunk, 8), xrow[i] + kk, xok[i] && kok);
#pragma unroll
    for (int i = 0; i < AR; ++i) cp_async16(as + swz(crow + 16 * i, cchunk, 8), arow[i] + (size_t)kk * 2, aok[i] && kok);
  };

  float acc[RMAX / 8][4];
#pragma unroll
  for (int n = 0; n < RMAX / 8; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;

#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < n_it) load_stage(s, s);
    cp_async_commit();
  }
  const int mrow = (TM == 64 ? warp * 16 : 0) + (lane & 7) + 8 * ((lane >> 3) & 1);
  for (int it = 0; it < n_it; ++it) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();
    if (it + STAGES - 1 < n_it) load_stage(it + STAGES - 1, (it + STAGES - 1) % STAGES);
    cp_async_commit();
    const uint32_t xs = sbase + (it % STAGES) * STAGE_BYTES, as = xs + TM * 128;
#pragma unroll
    for (int ks = 0; ks < KS / 16; ++ks) {
      if (TM == 16 && ks != warp) continue;   // short tiles: the four warps split each stage along k
      uint32_t af[4];
      ldmatrix_x4(af, xs + swz(mrow, 2 * ks + (lane >> 4), 8));
#pragma unroll
      for (int p = 0; p < RMAX / 16; ++p) {
        if (16 * p < rank) {
          uint32_t bf[4];
          ldmatrix_x4(bf, as + swz(16 * p + (lane & 7) + 8 * (lane >> 4), 2 * ks + ((lane >> 3) & 1), 8));
          mma_bf16(acc[2 * p], af, bf[0], bf[1]);
          mma_bf16(acc[2 * p + 1], af, bf[2], bf[3]);
        }
      }
    }
  }
  const int g = lane >> 2, t4 = lane & 3;
  if (TM == 64) {
    float* vout = a.v + ((size_t)(j * a.ksplit + split) * a.n_tokens) * RMAX;
#pragma unroll
    for (int n = 0; n < RMAX / 8; ++n) {
      const int r0 = tok0 + warp * 16 + g;
      if (r0 < tok1) *reinterpret_cast<float2*>(vout + (size_t)r0 * RMAX + 8 * n + 2 * t4) = make_float2(acc[n][0], acc[n][1]);
      if (r0 + 8 < tok1) *reinterpret_cast<float2*>(vout + (size_t)(r0 + 8) * RMAX + 8 * n + 2 * t4) = make_float2(acc[n][2], acc[n][3]);
    }
  } else {
    cp_async_wait<0>();
    __syncthreads();
    float* red = reinterpret_cast<float*>(smem);   // [4 warps][16 rows][RMAX]
#pragma unroll
    for (int n = 0; n < RMAX / 8; ++n) {
      float* r = red + (warp * 16 + g) * RMAX + 8 * n + 2 * t4;
      r[0] = acc[n][0]; r[1] = acc[n][1];
      r[8 * RMAX] = acc[n][2]; r[8 * RMAX + 1] = acc[n][3];
    }
    if (!a.v16) {
      __syncthreads();
      float* vout = a.v + ((size_t)(j * a.ksplit + split) * a.n_tokens) * RMAX;
      for (int i = tid; i < 16 * RMAX; i += SG_THREADS) {
        const int row = i / RMAX;
        if (tok0 + row < tok1)
          vout[(size_t)(tok0 + row) * RMAX + (i % RMAX)] =
              red[i] + red[16 * RMAX + i] + red[32 * RMAX + i] + red[48 * RMAX + i];
      }
      return;
    }
    // The final form is wanted: the slices of d_in are the CTAs of one cluster, and each hands its sums to the first one
    // through distributed shared memory.  The slices are added in order: the result does not depend on timing.  (Where an
    // expand of the same few microseconds follows, it adds the slices itself: the cluster's barrier costs 1 to 2 us more than
    // it saves there.)
    float* all = reinterpret_cast<float*>(smem + shrink_pipe_bytes(TM, RMAX, STAGES));      // first CTA: [slice][16 rows][RMAX]
    __syncthreads();
    if (clustered) cluster_wait();
    const uint32_t dst = clustered ? map_cluster_rank(smem_u32(all + split * 16 * RMAX), 0) : 0;
    for (int i = tid; i < 16 * RMAX; i += SG_THREADS) {
      const float sum = red[i] + red[16 * RMAX + i] + red[32 * RMAX + i] + red[48 * RMAX + i];
      if (clustered) st_cluster_f32(dst + 4u * i, sum);
      else all[i] = sum;
    }
    if (clustered) cluster_sync(); else __syncthreads();
    if (split == 0) {
      const size_t vout = (size_t)j * a.n_tokens * RMAX;
      for (int i = tid; i < 16 * RMAX; i += SG_THREADS) {
        const int row = i / RMAX;
        if (tok0 + row < tok1) {
          float sum = 0.f;
          for (int sp = 0; sp < a.ksplit; ++sp) sum += all[sp * 16 * RMAX + i];
          a.v16[vout + (size_t)(tok0 + row) * RMAX + (i % RMAX)] = __float2bfloat16_rn(sum * a.scale);
        }
      }
    }
  }
}

// The shrink of three projections that share x (q, k, v) for long segments and ranks up to 16: one CTA stages each x tile once and
// multiplies it by the three adapters' rank-rows, instead of three CTAs reading the same x rows.  With long
// segments the shrink is bound by the traffic from L2 into shared memory, and x is most of it.
template <int RMAX, int STAGES>
__global__ void __launch_bounds__(SG_THREADS) sgmv_shrink3_kernel(const SgmvArgs a) {
  constexpr int TM = 64, NM = 3;
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_wait();                 // x may come from the kernel right before this one
  pdl_launch_dependents();    // the expand may start its look-ups and first loads while this grid drains
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = blockIdx.x, split = blockIdx.y;
  int seg, tok0, tok1;
  if (!find_tile<TM>(a.seg_indptr, a.lora_ids, a.n_seg, tile, seg, tok0, tok1, a.all_segments != 0)) return;
  const int lid = a.lora_ids[seg];
  if (lid < 0) return;
  if ((uint32_t)lid >= a.pv.dir_cap || a.pv.dir[lid].rank <= 0) {
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
    return;
  }
  const LoraEntry* e = a.pv.dir + lid;
  for (int m = 0; m < NM; ++m) {
    if (a.mat_index[m] >= e->n_mats) {
      if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
      return;
    }
  }
  const int rank = min(e->rank, RMAX);
  // an adapter of a higher rank than this instantiation covers (registered after the launch was recorded
  // into a graph): its extra rank-rows are left out, and the status word says so
  if (e->rank > RMAX && tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
  const uint32_t table_off = e->table_off;
  const int d_in = e->mats[a.mat_index[0]].d_in;
  const int kchunk = ((d_in + a.ksplit * KS - 1) / (a.ksplit * KS)) * KS;
  const int kb = split * kchunk, ke = min(d_in, kb + kchunk);
  const int n_it = ke > kb ? (ke - kb + KS - 1) / KS : 0;

  constexpr int XR = TM / 16, AR = RMAX / 16;
  constexpr int STAGE_BYTES = (TM + NM * RMAX) * 128;
  const int crow = tid >> 3, cchunk = tid & 7;
  const __nv_bfloat16* xrow[XR];
  bool xok[XR];
#pragma unroll
  for (int i = 0; i < XR; ++i) {
    const int t = tok0 + crow + 16 * i;
    xok[i] = t < tok1;
    xrow[i] = a.x + (size_t)(xok[i] ? t : tok0) * d_in;
  }
  const __nv_bfloat16* arow[NM][AR];
  bool aok[NM][AR];
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    const LoraMat lm = e->mats[a.mat_index[m]];
#pragma unroll
    for (int i = 0; i < AR; ++i) {
      const int r = crow + 16 * i;
      aok[m][i] = false;
      arow[m][i] = reinterpret_cast<const __nv_bfloat16*>(a.pv.slab);
      if (r < rank)
        arow[m][i] = reinterpret_cast<const __nv_bfloat16*>(
            lora_row(a.pv, table_off, lm.a_tab, lm.a_row0, lm.a_rpb, d_in, r, aok[m][i]));
    }
  }
  const uint32_t sbase = smem_u32(smem);
  auto load_stage = [&](int it, int st) {
    const int kk = kb + it * KS + cchunk * 8;
    const bool kok = kk < ke;
    const uint32_t xs = sbase + st * STAGE_BYTES;
#pragma unroll
    for (int i = 0; i < XR; ++i) cp_async16(xs + swz(crow + 16 * i, cchunk, 8), xrow[i] + kk, xok[i] && kok);
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      const uint32_t as = xs + (TM + m * RMAX) * 128;
#pragma unroll
      for (int i = 0; i < AR; ++i) cp_async16(as + swz(crow + 16 * i, cchunk, 8), arow[m][i] + kk, aok[m][i] && kok);
    }
  };

  float acc[NM][RMAX / 8][4];
#pragma unroll
  for (int m = 0; m < NM; ++m)
#pragma unroll
    for (int n = 0; n < RMAX / 8; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;

#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < n_it) load_stage(s, s);
    cp_async_commit();
  }
  const int mrow = warp * 16 + (lane & 7) + 8 * ((lane >> 3) & 1);
  for (int it = 0; it < n_it; ++it) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();
    if (it + STAGES - 1 < n_it) load_stage(it + STAGES - 1, (it + STAGES - 1) % STAGES);
    cp_async_commit();
    const uint32_t xs = sbase + (it % STAGES) * STAGE_BYTES;
#pragma unroll
    for (int ks = 0; ks < KS / 16; ++ks) {
      uint32_t af[4];
      ldmatrix_x4(af, xs + swz(mrow, 2 * ks + (lane >> 4), 8));
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        const uint32_t as = xs + (TM + m * RMAX) * 128;
#pragma unroll
        for (int p = 0; p < RMAX / 16; ++p) {
          if (16 * p < rank) {
            uint32_t bf[4];
            ldmatrix_x4(bf, as + swz(16 * p + (lane & 7) + 8 * (lane >> 4), 2 * ks + ((lane >> 3) & 1), 8));
            mma_bf16(acc[m][2 * p], af, bf[0], bf[1]);
            mma_bf16(acc[m][2 * p + 1], af, bf[2], bf[3]);
          }
        }
      }
    }
  }
  const int g = lane >> 2, t4 = lane & 3;
  const int r0 = tok0 + warp * 16 + g;
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    float* vout = a.v + ((size_t)(m * a.ksplit + split) * a.n_tokens) * RMAX;
#pragma unroll
    for (int n = 0; n < RMAX / 8; ++n) {
      if (r0 < tok1) *reinterpret_cast<float2*>(vout + (size_t)r0 * RMAX + 8 * n + 2 * t4) = make_float2(acc[m][n][0], acc[m][n][1]);
      if (r0 + 8 < tok1) *reinterpret_cast<float2*>(vout + (size_t)(r0 + 8) * RMAX + 8 * n + 2 * t4) = make_float2(acc[m][n][2], acc[m][n][3]);
    }
  }
}

// The expand of short segments (a decode step): tiles of 16 tokens.
// KV: some projections of the call write their result rows into pool blocks (SgmvArgs::kv_side).
// whether the LoRA-term tile reuses the adapter-row buffer of the stage
__host__ __device__ constexpr bool expand_alias(int rmax) { return rmax >= 64; }
constexpr int expand_smem_bytes(int rmax) { return 2 * (16 + rmax) * 256 + (expand_alias(rmax) ? 0 : 16 * 256); }

// Five CTAs per SM: the kernel is bound by memory latency, occupancy matters more than a few spilled values.
template <int RMAX, bool KV>
__global__ void __launch_bounds__(SG_THREADS, 5) sgmv_expand_kernel(const SgmvArgs a) {
  constexpr int TM = 16;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int j = blockIdx.x % a.n_mats;
  const int tile = blockIdx.x / a.n_mats;
  int seg, tok0, tok1;
  if (!find_tile<TM>(a.seg_indptr, a.lora_ids, a.n_seg, tile, seg, tok0, tok1, a.all_segments != 0)) return;
  const int lid = a.lora_ids[seg];
  const int side = KV ? a.kv_side[j] : -1;   // >= 0: the result rows go into the requests' pool blocks
  int rank = 0;
  uint32_t table_off = 0;
  LoraMat lm = {};
  if (lid >= 0) {
    if ((uint32_t)lid >= a.pv.dir_cap || a.pv.dir[lid].rank <= 0 || a.mat_index[j] >= a.pv.dir[lid].n_mats) return;
    const LoraEntry* e = a.pv.dir + lid;
    lm = e->mats[a.mat_index[j]];
    rank = min(e->rank, RMAX);
    table_off = e->table_off;
  } else if (side < 0) {
    return;                                // no adapter and y stays where it is: nothing to do
  }
  const int d_out = a.d_out[j];
  const int c0 = blockIdx.y * a.expand_cols;
  if (c0 >= d_out) return;
  const int c1 = min(d_out, c0 + a.expand_cols);
  const int n_sub = (c1 - c0 + NSUB - 1) / NSUB;

  constexpr int WM = TM / 16, WN = 4 / WM;     // warps along tokens / along columns
  constexpr int NTW = 16 / WN;                 // 8-column tiles per warp inside a sub-tile
  const int warp_m = warp % WM, warp_n = warp / WM;
  const int g = lane >> 2, t4 = lane & 3;

  constexpr int YR = TM / 8;       // y rows per thread per sub-tile
  constexpr int BR = RMAX / 8;     // adapter rows per thread per sub-tile
  constexpr int STAGE_BYTES = (TM + RMAX) * 256;
  const int crow = tid >> 4, cchunk = tid & 15;
  __nv_bfloat16* yrow[YR];
  bool yok[YR];
#pragma unroll
  for (int i = 0; i < YR; ++i) {
    const int t = tok0 + crow + 8 * i;
    yok[i] = t < tok1;
    yrow[i] = a.y[j] + (size_t)(yok[i] ? t : tok0) * d_out;
  }
  // K / V rows: where each of this thread's token rows lives in the pool (block and slot of its position),
  // and how many slots behind it have to be cleared (V of a request's last token)
  uint32_t kvloc[KV ? YR : 1];      // block << 8 | slot << 1 | "last token of its request" (slot < 128, block < 2^24)
  if (KV && side >= 0) {
    int r = 0;
    {
      int lo = 0, hi = a.n_req;
      const int t0 = tok0 + crow;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (a.req_indptr[mid] <= t0) lo = mid; else hi = mid;
      }
      r = lo;
    }
#pragma unroll
    for (int i = 0; i < YR; ++i) {
      kvloc[i] = 0;
      const int t = tok0 + crow + 8 * i;
      if (!yok[i]) continue;
      while (r + 1 < a.n_req && t >= a.req_indptr[r + 1]) ++r;
      const int pos = a.prefix_lens[r] + (t - a.req_indptr[r]);
      const int entry = pos / a.bt, slot = pos - entry * a.bt;
      if (pos < 0 || t < a.req_indptr[r] || t >= a.req_indptr[r + 1] || entry >= a.tbl_indptr[r + 1] - a.tbl_indptr[r]) {
        atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
        yok[i] = false;
        continue;
      }
      const uint32_t blk = a.tbl[a.tbl_indptr[r] + entry];
      if (blk >= a.pv.n_blocks || blk >= (1u << 24)) {
        atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_BLOCK);
        yok[i] = false;
        continue;
      }
      kvloc[i] = blk << 8 | (uint32_t)slot << 1 | (t == a.req_indptr[r + 1] - 1 ? 1u : 0u);
    }
  }
  const __nv_bfloat16* brow[BR];
  bool bok[BR];
#pragma unroll
  for (int i = 0; i < BR; ++i) {
    const int r = crow + 8 * i;
    bok[i] = false;
    brow[i] = reinterpret_cast<const __nv_bfloat16*>(a.pv.slab);
    if (r < rank)
      brow[i] = reinterpret_cast<const __nv_bfloat16*>(
          lora_row(a.pv, table_off, lm.b_tab, lm.b_row0, lm.b_rpb, d_out, r, bok[i]));
  }
  const uint32_t sbase = smem_u32(smem);
  auto load_sub = [&](int sub, int st) {
    const int col = c0 + sub * NSUB + cchunk * 8;
    const bool cok = col < c1;
    const uint32_t ys = sbase + st * STAGE_BYTES, bs = ys + TM * 256;
#pragma unroll
    for (int i = 0; i < YR; ++i) cp_async16(ys + swz(crow + 8 * i, cchunk, 16), yrow[i] + col, yok[i] && cok);
#pragma unroll
    for (int i = 0; i < BR; ++i) cp_async16(bs + swz(crow + 8 * i, cchunk, 16), brow[i] + col, bok[i] && cok);
  };

  load_sub(0, 0);
  cp_async_commit();
  // v fragments: sum of the k-slices, scaled, rounded to bf16.  Everything above reads only what was in memory
  // before the shrink started; v is the shrink's output, so this is where a programmatic dependent launch waits.
  pdl_wait();
  uint32_t av[RMAX / 16][4];
  {
    const int r0 = tok0 + warp_m * 16 + g, r1 = r0 + 8;
#pragma unroll
    for (int ks = 0; ks < RMAX / 16; ++ks) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int row = (q & 1) ? r1 : r0;
        const int col = 16 * ks + 2 * t4 + ((q & 2) ? 8 : 0);
        float2 s = make_float2(0.f, 0.f);
        if (row < tok1 && col < rank) {
          for (int sp = 0; sp < a.ksplit; ++sp) {
            const float2 p = *reinterpret_cast<const float2*>(
                a.v + ((size_t)(j * a.ksplit + sp) * a.n_tokens + row) * RMAX + col);
            s.x += p.x; s.y += p.y;
          }
        }
        s.x *= a.scale; s.y *= a.scale;
        av[ks][q] = pack_bf16(s.x, s.y);
      }
    }
  }

  for (int sub = 0; sub < n_sub; ++sub) {
    const int st = sub & 1;
    if (sub + 1 < n_sub) load_sub(sub + 1, st ^ 1);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    unsigned char* ysm = smem + st * STAGE_BYTES;
    const uint32_t bs = sbase + st * STAGE_BYTES + TM * 256;
    float acc[NTW][4];
#pragma unroll
    for (int n = 0; n < NTW; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < RMAX / 16; ++ks) {
      if (16 * ks < rank) {
#pragma unroll
        for (int p = 0; p < NTW / 2; ++p) {
          uint32_t bf[4];
          ldmatrix_x4_trans(bf, bs + swz(16 * ks + (lane & 7) + 8 * ((lane >> 3) & 1),
                                         warp_n * NTW + 2 * p + (lane >> 4), 16));
          mma_bf16(acc[2 * p], av[ks], bf[0], bf[1]);
          mma_bf16(acc[2 * p + 1], av[ks], bf[2], bf[3]);
        }
      }
    }
    // the LoRA term of this sub-tile as bf16 pairs into a tile of its own (each element is owned by exactly one
    // thread); at rank 64 that tile takes the place of the adapter rows the MMAs have just consumed, which brings
    // the CTA to 64 KB and a third CTA onto the SM
    constexpr bool ALIAS = expand_alias(RMAX);
    unsigned char* dsm = ALIAS ? smem + st * STAGE_BYTES + TM * 256 : smem + 2 * STAGE_BYTES;
    if (ALIAS) __syncthreads();
#pragma unroll
    for (int n = 0; n < NTW; ++n) {
      const int chunk = warp_n * NTW + n;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = warp_m * 16 + g + 8 * h;
        *reinterpret_cast<uint32_t*>(dsm + swz(row, chunk, 16) + 4 * t4) = pack_bf16(acc[n][2 * h], acc[n][2 * h + 1]);
      }
    }
    __syncthreads();
    {
      const int col = c0 + sub * NSUB + cchunk * 8;
      if (col < c1) {
        if (!KV || side < 0) {
#pragma unroll
          for (int i = 0; i < YR; ++i)
            if (yok[i])
              *reinterpret_cast<uint4*>(yrow[i] + col) = add_bf16x8(*reinterpret_cast<const uint4*>(ysm + swz(crow + 8 * i, cchunk, 16)),
                                                                    *reinterpret_cast<const uint4*>(dsm + swz(crow + 8 * i, cchunk, 16)));
        } else if (KV) {
          // a sub-tile is one KV head: [K|V][head][slot][128] inside the block
          static_assert(NSUB == FL_HEAD_DIM, "a sub-tile must be one head");
          const size_t head_off = ((size_t)side * a.n_kv + (c0 + sub * NSUB) / FL_HEAD_DIM) * a.bt * (FL_HEAD_DIM * 2) + cchunk * 16;
#pragma unroll
          for (int i = 0; i < YR; ++i) {
            if (yok[i]) {
              const uint32_t loc = kvloc[KV ? i : 0];
              const int slot = (loc >> 1) & 127;
              unsigned char* dst = a.pv.slab + (size_t)(loc >> 8) * a.pv.block_bytes + head_off + slot * (FL_HEAD_DIM * 2);
              const uint4 base = *reinterpret_cast<const uint4*>(ysm + swz(crow + 8 * i, cchunk, 16));
              *reinterpret_cast<uint4*>(dst) =
                  lid < 0 ? base : add_bf16x8(base, *reinterpret_cast<const uint4*>(dsm + swz(crow + 8 * i, cchunk, 16)));
              if (side == 1 && (loc & 1u))     // V of a request's last token: clear the slots behind it
                for (int z = slot + 1; z < a.bt; ++z)
                  *reinterpret_cast<uint4*>(dst + (z - slot) * (FL_HEAD_DIM * 2)) = make_uint4(0u, 0u, 0u, 0u);
            }
          }
        }
      }
    }
    __syncthreads();
  }
}

// The expand of long segments: a stream over y in which no warp waits for another.
// A CTA takes up to `tm` tokens of one segment and 256 columns, a warp 64 of them.  The adapter's B rows of those columns go
// through shared memory once and stay in registers as MMA fragments (64 at rank 64); then each warp walks the tokens 16 at a
// time.  A thread copies ahead (cp.async, EX_DEPTH tiles) exactly the 16-byte pieces of y that it will add to itself, and
// the LoRA term gets into that layout through 2 KB of shared memory of the warp's own (stmatrix), so the loop has no CTA
// barrier but one per 96 to 128 tokens, when their shrink results are brought in.
// What bounds it: reading and writing y; on the way there the instructions per piece of y and the latency of the prologue's
// look-ups, which is why all 64 row addresses are found at once (a lane each), and so are the places of all the CTA's K / V
// rows (a thread each; looked up tile by tile in the loop they cost 24 of 223 us for the q, k, v call of 64 prompts on 7B).
// Shrink and expand of 16384 tokens on 34B (rank 64): o 217 -> 179 us, q, k, v with the KV store 271 -> 240 us (171 and 226 with the
// shrink of today); of 19770
// tokens on 7B (rank 16): 98 -> 93 us and 232 -> 205 us; before, tiles of 64 tokens and 128 columns with three barriers
// each had one tile of y per CTA in flight and read the B rows again for every 64 tokens.
constexpr int EX_COLS = 256, EX_DEPTH = 4;
constexpr int EX_TILE = 16 * 128;                  // bytes of a tile of 16 tokens x 64 columns
constexpr int EX_RING = EX_TILE * EX_DEPTH;
constexpr int EX_TM = 256;                         // tokens per CTA, at most
// tokens whose v is in shared memory at a time: at rank 64 what leaves room for four CTAs per SM, at rank 16 for five
__host__ __device__ constexpr int ex_vt(int rmax) { return rmax == 64 ? 112 : rmax == 32 ? 128 : 96; }
__host__ __device__ constexpr int ex_smem(int rmax) { return ex_vt(rmax) * rmax * 2 + 4 * (EX_RING + EX_TILE) + EX_TM * 4; }
static_assert(FL_MAX_RANK * EX_COLS * 2 <= 4 * EX_RING, "the B rows are staged where the y tiles go later");
// 16-byte piece `chunk` of row `row` of the v tile; rows of 32, 64 or 128 bytes, conflict-free for ldmatrix
template <int RMAX>
__device__ __forceinline__ uint32_t ex_vswz(int row, int chunk) {
  constexpr int CH = RMAX / 8, SH = RMAX == 64 ? 0 : RMAX == 32 ? 1 : 2;
  return (uint32_t)((row * CH + (chunk ^ ((row >> SH) & (CH - 1)))) * 16);
}

// Request of a token, for tokens taken in ascending order, and where its K / V row lives in the pool.
struct KvCursor {
  int r, beg, end, pos0, tab, n_tab;
  __device__ __forceinline__ void load(const SgmvArgs& a) {
    beg = a.req_indptr[r];
    end = a.req_indptr[r + 1];
    pos0 = a.prefix_lens[r] - beg;
    tab = a.tbl_indptr[r];
    n_tab = a.tbl_indptr[r + 1] - tab;
  }
  // request of token t (the whole warp takes part with the same t): the first that ends behind it, 32 at a time
  __device__ __forceinline__ void init(const SgmvArgs& a, int t) {
    const int lane = threadIdx.x & 31;
    r = a.n_req - 1;
    for (int r0 = 0; r0 < a.n_req; r0 += 32) {
      const bool behind = r0 + lane < a.n_req && a.req_indptr[r0 + lane + 1] > t;
      const uint32_t m = __ballot_sync(0xffffffffu, behind);
      if (m) {
        r = r0 + __ffs(m) - 1;
        break;
      }
    }
    load(a);
  }
  // block << 8 | slot << 1 | "last token of its request", or ~0 when the token has no place (flag raised)
  __device__ __forceinline__ uint32_t find(const SgmvArgs& a, int t) {
    while (t >= end && r + 1 < a.n_req) {
      ++r;
      load(a);
    }
    const int pos = pos0 + t;
    // pos / bt by the rounded-up reciprocal 2^32 / bt: exact below 2^25 for bt <= 128
    const int entry = pos >= 0 && pos < (1 << 25) ? (a.bt == 1 ? pos : (int)__umulhi((uint32_t)pos, a.bt_inv)) : pos / a.bt;
    const int slot = pos - entry * a.bt;
    if (pos < 0 || t < beg || t >= end || entry >= n_tab) {
      atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
      return 0xffffffffu;
    }
    const uint32_t blk = a.tbl[tab + entry];
    if (blk >= a.pv.n_blocks || blk >= (1u << 24)) {
      atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_BLOCK);
      return 0xffffffffu;
    }
    return blk << 8 | (uint32_t)slot << 1 | (t == end - 1 ? 1u : 0u);
  }
};

template <int RMAX, bool KV>
__global__ void __launch_bounds__(SG_THREADS, RMAX == 16 ? 5 : 4) sgmv_expand_long_kernel(const __grid_constant__ SgmvArgs a, int tm, int n_ranges) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int KN = RMAX / 16, EX_VT = ex_vt(RMAX);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = blockIdx.x / n_ranges;
  int range = blockIdx.x - tile * n_ranges, j = 0;       // column ranges of all projections, one after the other
  for (; j + 1 < a.n_mats; ++j) {
    const int n = (a.d_out[j] + EX_COLS - 1) / EX_COLS;
    if (range < n) break;
    range -= n;
  }
  int seg, tok0, tok1;
  if (!find_tile(tm, a.seg_indptr, a.lora_ids, a.n_seg, tile, seg, tok0, tok1, a.all_segments != 0)) return;
  const int lid = a.lora_ids[seg];
  const int side = KV ? a.kv_side[j] : -1;   // >= 0: the result rows go into the requests' pool blocks
  const int d_out = a.d_out[j], c0 = range * EX_COLS;
  int rank = 0;
  const uint32_t sbase = smem_u32(smem), ring0 = sbase + EX_VT * RMAX * 2;
  // ---- B rows of the CTA's columns: shared memory, then fragments
  const unsigned char* rowp[RMAX <= 32 ? 1 : 2];         // row lane (and lane + 32)
  rowp[0] = nullptr;
  if (RMAX > 32) rowp[RMAX > 32 ? 1 : 0] = nullptr;
  if (lid >= 0) {
    if ((uint32_t)lid >= a.pv.dir_cap || a.pv.dir[lid].rank <= 0 || a.mat_index[j] >= a.pv.dir[lid].n_mats) return;
    const LoraEntry* e = a.pv.dir + lid;
    const LoraMat lm = e->mats[a.mat_index[j]];
    rank = min(e->rank, RMAX);
#pragma unroll
    for (int i = 0; i < (RMAX <= 32 ? 1 : 2); ++i) {
      const int r = lane + 32 * i;
      bool ok = false;
      if (r < rank) rowp[i] = lora_row(a.pv, e->table_off, lm.b_tab, lm.b_row0, lm.b_rpb, d_out, r, ok);
      if (!ok) rowp[i] = nullptr;
    }
  } else if (side < 0) {
    return;                                // no adapter and y stays where it is: nothing to do
  }
  {
    const int col = c0 + lane * 8;         // a warp copies whole rows of 512 bytes: rows warp, warp + 4, ...
#pragma unroll
    for (int i = 0; i < RMAX / 4; ++i) {
      const int r = warp + 4 * i;
      const unsigned char* src = reinterpret_cast<const unsigned char*>(
          __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(rowp[RMAX > 32 && i >= 8 ? 1 : 0]), r & 31));
      const bool have = src && col < d_out;
      cp_async16(ring0 + swz(r, lane, 32), have ? src + col * 2 : a.pv.slab, have);
    }
  }
  cp_async_commit();
  const int rows = tok1 - tok0, n_tiles = (rows + 15) / 16;
  uint32_t* const loc = reinterpret_cast<uint32_t*>(smem + EX_VT * RMAX * 2 + 4 * (EX_RING + EX_TILE));
  if (KV && side >= 0) {                   // where each row goes
    KvCursor cur;
    cur.init(a, tok0);
    for (int r = tid; r < rows; r += SG_THREADS) loc[r] = cur.find(a, tok0 + r);
  }
  cp_async_wait<0>();
  __syncthreads();
  uint32_t bf[KN][8][2];
#pragma unroll
  for (int ks = 0; ks < KN; ++ks)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      uint32_t f[4];
      ldmatrix_x4_trans(f, ring0 + swz(16 * ks + (lane & 7) + 8 * ((lane >> 3) & 1), warp * 8 + 2 * p + (lane >> 4), 32));
      bf[ks][2 * p][0] = f[0]; bf[ks][2 * p][1] = f[1];
      bf[ks][2 * p + 1][0] = f[2]; bf[ks][2 * p + 1][1] = f[3];
    }
  __syncthreads();
  // ---- y ahead: this thread's pieces are rows pr + 4 k of a tile, 16-byte chunk pc of the warp's 64 columns
  const int pr = lane >> 3, pc = lane & 7;
  const int wc = c0 + warp * 64 + pc * 8;
  const bool cok = wc < d_out;
  const uint32_t ring = ring0 + warp * EX_RING + lane * 16;
  const uint32_t term = ring0 + 4 * EX_RING + warp * EX_TILE;
  __nv_bfloat16* const ycol = a.y[j] + (size_t)(tok0 + pr) * d_out + (cok ? wc : 0);
  const size_t step4 = (size_t)4 * d_out;
  auto load_y = [&](int i) {
    const uint32_t dst = ring + (i % EX_DEPTH) * EX_TILE;
    const __nv_bfloat16* src = ycol + (size_t)(16 * i) * d_out;
    const int left = rows - 16 * i - pr;
#pragma unroll
    for (int k = 0; k < 4; ++k) cp_async16(dst + k * 512, 4 * k < left ? src + k * step4 : ycol, cok && 4 * k < left);
  };
#pragma unroll
  for (int i = 0; i < EX_DEPTH - 1; ++i) {
    if (i < n_tiles) load_y(i);
    cp_async_commit();
  }
  // Everything above reads only what was in memory before the shrink started; v is the shrink's output, so this is where a
  // dependent launch waits.
  pdl_wait();
  const size_t head_off = KV && side >= 0 ? ((size_t)(side * a.n_kv + wc / FL_HEAD_DIM) * a.bt) * (FL_HEAD_DIM * 2) + (wc % FL_HEAD_DIM) * 2 : 0;
  for (int i = 0; i < n_tiles; ++i) {
    if (i % (EX_VT / 16) == 0) {
      // ---- v of the next tokens: as the shrink left it in its final form, or slices summed, scaled, rounded to bf16
      if (i > 0) __syncthreads();
      const int v0 = 16 * i, vn = min(EX_VT, (n_tiles - i) * 16);
      for (int c = tid; c < vn * (RMAX / 8); c += SG_THREADS) {
        const int r = c / (RMAX / 8), ch = c % (RMAX / 8);
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        if (v0 + r < rows && 8 * ch < rank) {
          if (a.v16) {
            q = *reinterpret_cast<const uint4*>(a.v16 + ((size_t)j * a.n_tokens + tok0 + v0 + r) * RMAX + 8 * ch);
          } else {
            float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
            for (int sp = 0; sp < a.ksplit; ++sp) {
              const float4* src = reinterpret_cast<const float4*>(a.v + ((size_t)(j * a.ksplit + sp) * a.n_tokens + tok0 + v0 + r) * RMAX + 8 * ch);
              const float4 p0 = src[0], p1 = src[1];
              s0.x += p0.x; s0.y += p0.y; s0.z += p0.z; s0.w += p0.w;
              s1.x += p1.x; s1.y += p1.y; s1.z += p1.z; s1.w += p1.w;
            }
            q = make_uint4(pack_bf16(s0.x * a.scale, s0.y * a.scale), pack_bf16(s0.z * a.scale, s0.w * a.scale),
                           pack_bf16(s1.x * a.scale, s1.y * a.scale), pack_bf16(s1.z * a.scale, s1.w * a.scale));
          }
        }
        *reinterpret_cast<uint4*>(smem + ex_vswz<RMAX>(r, ch)) = q;
      }
      __syncthreads();
    }
    if (i + EX_DEPTH - 1 < n_tiles) load_y(i + EX_DEPTH - 1);
    cp_async_commit();
    const int vr = 16 * (i % (EX_VT / 16));
    uint32_t af[KN][4];
#pragma unroll
    for (int ks = 0; ks < KN; ++ks)
      ldmatrix_x4(af[ks], sbase + ex_vswz<RMAX>(vr + (lane & 7) + 8 * ((lane >> 3) & 1), 2 * ks + (lane >> 4)));
#pragma unroll
    for (int q = 0; q < 2; ++q) {          // 32 columns at a time
      float acc[4][4];
#pragma unroll
      for (int n = 0; n < 4; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KN; ++ks)
        if (KN == 1 || 16 * ks < rank) {
#pragma unroll
          for (int n = 0; n < 4; ++n) mma_bf16(acc[n], af[ks], bf[ks][4 * q + n][0], bf[ks][4 * q + n][1]);
        }
#pragma unroll
      for (int n = 0; n < 4; n += 2)       // 16 rows x 2 tiles of 8 columns: rows of 128 bytes, chunks swizzled
        stmatrix_x4(term + swz((lane & 7) + 8 * ((lane >> 3) & 1), 4 * q + n + (lane >> 4), 8), pack_bf16(acc[n][0], acc[n][1]),
                    pack_bf16(acc[n][2], acc[n][3]), pack_bf16(acc[n + 1][0], acc[n + 1][1]), pack_bf16(acc[n + 1][2], acc[n + 1][3]));
    }
    cp_async_wait<EX_DEPTH - 1>();
    __syncwarp();
    const uint32_t yp = ring + (i % EX_DEPTH) * EX_TILE;
    __nv_bfloat16* const yr = ycol + (size_t)(16 * i) * d_out;
    const int left = rows - 16 * i - pr;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r = pr + 4 * k;
      const uint4 base = ld_shared_v4(yp + k * 512);
      const uint4 sum = KV && lid < 0 ? base : add_bf16x8(base, ld_shared_v4(term + swz(r, pc, 8)));     // (a sum would turn -0 into 0)
      if (cok && 4 * k < left) {
        if (!KV || side < 0) {
          *reinterpret_cast<uint4*>(yr + k * step4) = sum;
        } else {
          const uint32_t l = loc[16 * i + r];
          if (l != 0xffffffffu) {
            const int slot = (l >> 1) & 127;
            unsigned char* dst = a.pv.slab + (size_t)(l >> 8) * a.pv.block_bytes + head_off + slot * (FL_HEAD_DIM * 2);
            *reinterpret_cast<uint4*>(dst) = sum;
            if (side == 1 && (l & 1u))     // V of a request's last token: clear the slots behind it
              for (int z = slot + 1; z < a.bt; ++z)
                *reinterpret_cast<uint4*>(dst + (z - slot) * (FL_HEAD_DIM * 2)) = make_uint4(0u, 0u, 0u, 0u);
          }
        }
      }
    }
    __syncwarp();
  }
  cp_async_wait<0>();
}

int pick_ksplit(int n_tokens) {
  // decode-sized batches have few token tiles: slice d_in so that enough CTAs stream adapter rows
  const int tiles = n_tokens / 16 + 1;
  int ks = 592 / tiles;
  if (ks < 1) ks = 1;
  if (ks > KSPLIT_MAX) ks = KSPLIT_MAX;
  return ks;
}

// Columns per expand CTA.  Every CTA pays a prologue of dependent look-ups (its tile, the adapter's directory
// entry and row tables, the v fragments, the K/V destinations) that wider CTAs spread over more sub-tiles; the
// widest slice that still leaves about ten CTAs per SM in the grid wins.
int pick_expand_cols(const SgmvArgs& a, int tiles) {
  int cols = EXPAND_COLS_MAX;
  for (; cols > EXPAND_COLS_MIN; cols /= 2) {
    long ctas = 0;
    for (int j = 0; j < a.n_mats; ++j) ctas += (long)tiles * ((a.d_out[j] + cols - 1) / cols);
    if (ctas >= 1480) break;
  }
  return cols;
}

template <int RMAX>
int launch_expand_long(fl_pool* p, const SgmvArgs& a, cudaStream_t st) {
  static bool configured[16] = {};
  if (!configured[p->device & 15]) {
    FL_CUDA(p, cudaFuncSetAttribute(sgmv_expand_long_kernel<RMAX, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ex_smem(RMAX)));
    FL_CUDA(p, cudaFuncSetAttribute(sgmv_expand_long_kernel<RMAX, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ex_smem(RMAX)));
    configured[p->device & 15] = true;
  }
  int n_ranges = 0;
  for (int j = 0; j < a.n_mats; ++j) n_ranges += (a.d_out[j] + EX_COLS - 1) / EX_COLS;
  // Tokens per CTA: the rounds of CTAs over the SMs times what a CTA costs, its prologue being worth about 48 tokens (of 256,
  // 128 and 64 tokens, q of 8747 tokens on 7B takes 67, 69 and 71 us in one, two and four rounds; q of 4391 tokens 31 us at
  // 128 in one round and 35 us at 64 in two).
  const long slots = (RMAX == 16 ? 5L : 4L) * p->sm_count;
  int tm = EX_TM;
  long best = -1;
  for (int t = EX_TM; t >= 64; t /= 2) {
    const long cost = ((long)(a.n_tokens / t + 1) * n_ranges + slots - 1) / slots * (t + 48);
    if (best < 0 || cost < best) { best = cost; tm = t; }
  }
  const unsigned grid = (unsigned)((a.n_seg + a.n_tokens / tm) * n_ranges);
  if (a.all_segments) FL_CUDA(p, launch_pdl(sgmv_expand_long_kernel<RMAX, true>, dim3(grid), dim3(SG_THREADS), ex_smem(RMAX), st, a, tm, n_ranges));
  else FL_CUDA(p, launch_pdl(sgmv_expand_long_kernel<RMAX, false>, dim3(grid), dim3(SG_THREADS), ex_smem(RMAX), st, a, tm, n_ranges));
  return FL_OK;
}

template <int RMAX>
int launch_expand_short(fl_pool* p, SgmvArgs& a, int tiles, int d_out_max, cudaStream_t st) {
  const int smem = expand_smem_bytes(RMAX);     // two stages of (y, B) + the LoRA-term tile
  static bool configured[16] = {};
  if (!configured[p->device & 15]) {
    FL_CUDA(p, cudaFuncSetAttribute(sgmv_expand_kernel<RMAX, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    FL_CUDA(p, cudaFuncSetAttribute(sgmv_expand_kernel<RMAX, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    configured[p->device & 15] = true;
  }
  a.expand_cols = pick_expand_cols(a, tiles);
  const dim3 grid(tiles * a.n_mats, (d_out_max + a.expand_cols - 1) / a.expand_cols);
  if (a.all_segments) FL_CUDA(p, launch_pdl(sgmv_expand_kernel<RMAX, true>, grid, dim3(SG_THREADS), smem, st, a));
  else FL_CUDA(p, launch_pdl(sgmv_expand_kernel<RMAX, false>, grid, dim3(SG_THREADS), smem, st, a));
  return FL_OK;
}

// Whether the kernel behind finds a place for all its CTAs while `ctas` of a shrink with `smem` bytes each are there, as many on an SM as fit.
// (Clusters do not fill every SM; the shares are those that tell the measured sides apart.)
constexpr int SM_SMEM = 228 * 1024, CTA_SMEM = 1024;       // an SM's shared memory, and what each CTA takes beside its own
bool has_room(const sgmv::Follower& f, int ctas, int smem, int sms) {
  return f.ctas <= (sms - (double)ctas / (SM_SMEM / (smem + CTA_SMEM))) * (f.cluster == 1 ? 1 : f.cluster == 2 ? 0.9255 : f.cluster == 3 ? 0.8677 : 0.91);
}
// Whether the shrink in tiles of 16 tokens has more of its stages in flight: where the projection's CTAs have no room beside the shallow one either,
// or room beside the deeper one as well, on the same SMs, and where the deeper one's clusters run at once (15 of eight, one CTA per SM).
// Decode steps (a graph of q, k, v with the KV store, attention over 512 keys, o; 13B up and down too, so that W comes from HBM), shallow everywhere,
// deeper everywhere and with this rule, us:  rank 64, 4 requests with an adapter each, 13B 143.5, 137.1, 137; 34B 90.9, 92.0, 86; 12 of them
// 34B 124.1, 125.1, 122; 13B 194.5, 191.0, 183; 16 of them 34B 129.9, 144.7, 130; 7B 97.0, 106.5, 97.  Rank 32, 4 of them 34B 77.3, 84.9,
// 77; 13B 115.4, 128.6, 115; 12 13B 174.1, 164.9, 166.  Rank 16, one 7B 46.6, 45.9, 46; 8 13B 130.6, 143.2, 131; 37 7B 115.4, 112.3, 112.
// 294 such steps: 1 % less than with a bound on the number of the deeper one's CTAs alone, 2 % less than with four stages; the worst, 16 adapters
// of rank 64 on 13B, 2 % more than the former.  Not above 128 tokens (rank 16, 200 tokens in one segment, 13B 187 us, shallow 175; 34B 115.5, 111.4).  (The same calls back to back, with W in L2, order themselves quite differently.)
bool deeper(const fl_pool* p, const SgmvArgs& a, int rmax, int tiles, const sgmv::Follower* next) {
  const int slice = (p->mats[a.mat_index[0]].d_in + KS * a.ksplit - 1) / (KS * a.ksplit);       // stages
  if (!a.v16 || slice <= SH_STAGES) return false;
  // behind it a GEMM on all SMs (rank 16: shallow and deeper within 1 us of 16 to 110, but 900 tokens in 45 segments on 7B, o, 38 and 35)
  if (!next) return tiles * a.n_mats * a.ksplit <= p->sm_count * (rmax == 64 ? 1.1 : rmax == 32 ? 2 : 3);
  const int sums = KSPLIT_MAX * 16 * rmax * 4, shallow = shrink_pipe_bytes(16, rmax, SH_STAGES) + sums, deep = shrink_pipe_bytes(16, rmax, deep_stages(rmax)) + sums;
  const int each = a.n_mats * a.ksplit, few = std::max(a.n_seg, (a.n_tokens + 15) / 16) * each;            // CTAs with a tile, at least
  const int most = next->cluster == 1 ? few : (a.n_seg + std::max(0, a.n_tokens - a.n_seg) / 16) * each;      // and at most
  if (few > p->sm_count * 13 / 16 * (SM_SMEM / (deep + CTA_SMEM)) || a.n_tokens > 128) return false;
  if (!has_room(*next, most, shallow, p->sm_count)) return true;
  return next->cluster > 1 && (int)next->smem + deep + 2 * CTA_SMEM <= SM_SMEM && has_room(*next, most * 3 / 2, deep, p->sm_count);
}

template <int TM, int RMAX, int STAGES>
int launch_shrink(fl_pool* p, const SgmvArgs& a, int tiles, cudaStream_t st) {
  static bool configured[16] = {};
  const int smem_max = shrink_pipe_bytes(TM, RMAX, STAGES) + (TM == 16 ? KSPLIT_MAX * 16 * RMAX * 4 : 0);
  const int smem = a.v16 ? smem_max : shrink_pipe_bytes(TM, RMAX, STAGES);      // + every slice's sums
  if (!configured[p->device & 15]) {
    FL_CUDA(p, cudaFuncSetAttribute(sgmv_shrink_kernel<TM, RMAX, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    configured[p->device & 15] = true;
  }
  FL_CUDA(p, launch_pdl_cluster(sgmv_shrink_kernel<TM, RMAX, STAGES>, dim3(tiles * a.n_mats, a.ksplit), dim3(1, a.v16 ? a.ksplit : 1),
                                dim3(SG_THREADS), smem, st, a));
  return FL_OK;
}

template <int TM, int RMAX>
int launch_pair(fl_pool* p, SgmvArgs& a, int tiles, int d_out_max, cudaStream_t st, bool shrink_only, const sgmv::Follower* next) {
  if (TM == 64 && p->sgmv_shrink_kind == 0 && a.n_mats <= 3 && a.tc_ksplit > 0) {
    // long segments: the shrink on tcgen05 tensor cores, tiles of 128 tokens, its own number of d_in slices
    a.ksplit = a.tc_ksplit;
    sgmv::TcShrinkArgs t;
    t.pv = a.pv;
    t.ksplit = a.ksplit;
    t.n_mats = a.n_mats;
    for (int j = 0; j < 3; ++j) t.mat_index[j] = a.mat_index[j < a.n_mats ? j : 0];
    t.seg_indptr = a.seg_indptr;
    t.lora_ids = a.lora_ids;
    t.n_seg = a.n_seg;
    t.n_tokens = a.n_tokens;
    t.d_in = p->mats[a.mat_index[0]].d_in;
    t.scale = a.scale;
    t.v16 = a.v16 = reinterpret_cast<__nv_bfloat16*>(a.v);
    const int rc = sgmv::shrink_tc(p, t, a.x, RMAX, st);
    if (rc != FL_OK) return rc;
  } else if (TM == 64 && RMAX == 16 && a.n_mats == 3) {      // at higher ranks the three accumulators cost too many registers
    // three stages (43 KB) put five CTAs on an SM, four stages three: 46 against 57 us for 19770 tokens on 7B, where 340 tiles
    // in two slices are one round of five per SM and two rounds of three; with fewer CTAs the deeper pipeline is the better one
    static bool configured3[16] = {};
    const int smem_of[2] = {3 * (64 + 3 * RMAX) * 128, 4 * (64 + 3 * RMAX) * 128};
    if (!configured3[p->device & 15]) {
      FL_CUDA(p, cudaFuncSetAttribute(sgmv_shrink3_kernel<RMAX, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_of[0]));
      FL_CUDA(p, cudaFuncSetAttribute(sgmv_shrink3_kernel<RMAX, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_of[1]));
      configured3[p->device & 15] = true;
    }
    if (tiles * a.ksplit > 3 * p->sm_count)
      FL_CUDA(p, launch_pdl(sgmv_shrink3_kernel<RMAX, 3>, dim3(tiles, a.ksplit), dim3(SG_THREADS), smem_of[0], st, a));
    else
      FL_CUDA(p, launch_pdl(sgmv_shrink3_kernel<RMAX, 4>, dim3(tiles, a.ksplit), dim3(SG_THREADS), smem_of[1], st, a));
  } else {
    const bool deep = TM == 16 && deeper(p, a, RMAX, tiles, next);
    const int rc = deep ? launch_shrink<TM, RMAX, TM == 16 ? deep_stages(RMAX) : SH_STAGES>(p, a, tiles, st) : launch_shrink<TM, RMAX, SH_STAGES>(p, a, tiles, st);
    if (rc != FL_OK) return rc;
  }
  if (shrink_only) return FL_OK;       // the caller consumes the partial sums itself
  return TM == 64 ? launch_expand_long<RMAX>(p, a, st) : launch_expand_short<RMAX>(p, a, tiles, d_out_max, st);
}

int rmax_of(const fl_pool* p) { return p->max_rank <= 16 ? 16 : (p->max_rank <= 32 ? 32 : 64); }

}  // namespace

extern "C" {

size_t fl_lora_sgmv_workspace(int n_tokens, int n_mats) {
  if (n_tokens <= 0 || n_mats <= 0) return 256;
  return (size_t)n_mats * pick_ksplit(n_tokens) * (size_t)n_tokens * FL_MAX_RANK * sizeof(float) + 256;
}

}  // extern "C"

namespace {

struct KvDest {      // where K and V results go when they are appended to the pool by the projection itself
  int k_slot, v_slot;           // positions of the K and V projections in the call's list
  const int32_t* req_indptr;
  const int32_t* tbl_indptr;
  const uint32_t* tbl;
  const int32_t* prefix_lens;
  int n_req, n_kv;
};

int sgmv_common(fl_pool* p, fl_bf16* const* ys, const fl_bf16* x, const int* mat_indices, int n_mats,
                const int32_t* seg_indptr, const int32_t* lora_ids, int n_seg, int n_tokens,
                float scale, void* workspace, size_t workspace_bytes, fl_stream stream, const KvDest* kv,
                sgmv::ShrinkInfo* shrink_only = nullptr, bool scaled = false, const sgmv::Follower* next = nullptr) {
  if (!p || n_mats < 1 || n_mats > FL_MAX_MATS || n_seg < 0 || n_tokens < 0 || !ys || !mat_indices) return FL_EINVAL;
  if (n_seg == 0 || n_tokens == 0) return FL_OK;
  if (!x || !seg_indptr || !lora_ids || !workspace) return FL_EINVAL;
  if (p->n_mats == 0) return FL_EBADID;   // no adapter registered
  SgmvArgs a;
  a.pv = p->view();
  a.x = reinterpret_cast<const __nv_bfloat16*>(x);
  int d_out_max = 0;
  for (int j = 0; j < n_mats; ++j) {
    const int mi = mat_indices[j];
    if (mi < 0 || mi >= p->n_mats || (!ys[j] && !shrink_only)) return FL_EINVAL;
    if (p->mats[mi].d_in != p->mats[mat_indices[0]].d_in) return FL_EINVAL;   // the projections share x
    a.y[j] = reinterpret_cast<__nv_bfloat16*>(ys[j]);
    a.mat_index[j] = mi;
    d_out_max = d_out_max > p->mats[mi].d_out ? d_out_max : p->mats[mi].d_out;
  }
  for (int j = 0; j < FL_MAX_MATS; ++j) {
    a.kv_side[j] = -1;
    a.d_out[j] = j < n_mats ? p->mats[mat_indices[j]].d_out : 0;
  }
  a.all_segments = 0;
  a.req_indptr = a.tbl_indptr = a.prefix_lens = nullptr;
  a.tbl = nullptr;
  a.n_req = a.n_kv = a.bt = 0;
  a.bt_inv = 0;
  if (kv) {
    const size_t per_tok = (size_t)2 * kv->n_kv * FL_HEAD_DIM * 2;
    if (kv->n_kv < 1 || kv->n_req < 1 || p->block_bytes % per_tok != 0 || kv->k_slot == kv->v_slot) return FL_EINVAL;
    if (!kv->req_indptr || !kv->tbl_indptr || !kv->tbl || !kv->prefix_lens) return FL_EINVAL;
    for (int side = 0; side < 2; ++side) {
      const int slot = side ? kv->v_slot : kv->k_slot;
      if (slot < 0 || slot >= n_mats || a.d_out[slot] != kv->n_kv * FL_HEAD_DIM) return FL_EINVAL;
      a.kv_side[slot] = side;
    }
    a.all_segments = 1;
    a.req_indptr = kv->req_indptr;
    a.tbl_indptr = kv->tbl_indptr;
    a.tbl = kv->tbl;
    a.prefix_lens = kv->prefix_lens;
    a.n_req = kv->n_req;
    a.n_kv = kv->n_kv;
    a.bt = (int)(p->block_bytes / per_tok);
    a.bt_inv = (uint32_t)(((1ull << 32) + a.bt - 1) / a.bt);
    // the expand packs a token's destination into one word: 7 bits of slot, 24 bits of block id
    if (a.bt > 128 || p->n_blocks > (1u << 24)) return FL_EINVAL;
  }
  a.n_mats = n_mats;
  a.seg_indptr = seg_indptr;
  a.lora_ids = lora_ids;
  a.n_seg = n_seg;
  a.n_tokens = n_tokens;
  a.scale = scale;
  a.v = reinterpret_cast<float*>(workspace);
  a.ksplit = pick_ksplit(n_tokens);
  if (workspace_bytes < fl_lora_sgmv_workspace(n_tokens, n_mats)) return FL_ENOMEM;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != p->device) cudaSetDevice(p->device);
  a.v16 = scaled ? reinterpret_cast<__nv_bfloat16*>(workspace) : nullptr;
  const bool small = scaled || n_tokens <= 16 * n_seg;   // average segment of at most 16 tokens: decode-like
  const int rmax = rmax_of(p);
  const cudaStream_t st = (cudaStream_t)stream;
  if (!small && rmax == 16 && a.ksplit == 1) {
    // A long-segment batch of a few thousand tokens gives the shrink about two CTAs per SM (eight warps), too few to
    // keep the loads of a rank-16 shrink in flight: two slices of d_in double them.  The scratch is sized for rank 64,
    // so at rank 16 two slices fit in what the caller already brought.
    const long shrink_ctas = (long)(n_seg + n_tokens / 64) * (n_mats == 3 ? 1 : n_mats);
    const size_t need = (size_t)n_mats * 2 * (size_t)n_tokens * rmax * sizeof(float) + 256;
    if (shrink_ctas < 592 && need <= workspace_bytes) a.ksplit = 2;
  }
  a.tc_ksplit = 0;
  if (!small && n_mats <= 3) {
    // At rank 16 the mma.sync shrink is the faster one for small batches, whose time is look-ups (shrink and expand, 7B: q, k, v of 512 tokens
    // 13.8 and 15.2 us; o of 2000 tokens 12 and 17), and where the tiles of 128 tokens take more than one round (q, k, v of 19770 tokens
    // 205 and 214); in between the tcgen05 one is (q, k, v of 3200 tokens 48 and 45, of 5600 70 and 67; on 34B 2000 tokens 32 and 28).
    const int d_in = p->mats[mat_indices[0]].d_in;
    if (rmax >= 32 || ((double)n_tokens * d_in >= (n_mats == 3 ? 8e6 : 2e7) && n_tokens / 128 + n_seg / 2 < p->sm_count))
      a.tc_ksplit = sgmv::tc_slices(p, n_seg, n_tokens, d_in, rmax, n_mats);
  }
  int rc;
  const bool so = shrink_only != nullptr;
  if (so) {
    shrink_only->ksplit = a.ksplit;
    shrink_only->rmax = rmax;
    shrink_only->final = scaled || (!small && p->sgmv_shrink_kind == 0 && a.tc_ksplit > 0);
  }
  if (small) {
    const int tiles = n_seg + n_tokens / 16;
    // slices of d_in so that all CTAs run at once: at rank 64 three of them fit on an SM, below that at least five
    if (scaled) a.ksplit = std::max(1, std::min(KSPLIT_MAX, (rmax == 64 ? 3 : 4) * p->sm_count / (tiles * n_mats)));
    rc = rmax == 16 ? launch_pair<16, 16>(p, a, tiles, d_out_max, st, so, next)
       : rmax == 32 ? launch_pair<16, 32>(p, a, tiles, d_out_max, st, so, next)
                    : launch_pair<16, 64>(p, a, tiles, d_out_max, st, so, next);
  } else {
    const int tiles = n_seg + n_tokens / 64;
    rc = rmax == 16 ? launch_pair<64, 16>(p, a, tiles, d_out_max, st, so, next)
       : rmax == 32 ? launch_pair<64, 32>(p, a, tiles, d_out_max, st, so, next)
                    : launch_pair<64, 64>(p, a, tiles, d_out_max, st, so, next);
  }
  if (prev != p->device && prev >= 0) cudaSetDevice(prev);
  return rc;
}

}  // namespace

namespace sgmv {
int shrink(fl_pool* p, const fl_bf16* x, const int* mat_indices, int n_mats, const int32_t* seg_indptr,
           const int32_t* lora_ids, int n_seg, int n_tokens, float scale, void* workspace, size_t workspace_bytes, fl_stream stream,
           ShrinkInfo* info) {
  fl_bf16* none[FL_MAX_MATS] = {};
  return sgmv_common(p, none, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace,
                     workspace_bytes, stream, nullptr, info);
}
int shrink_scaled(fl_pool* p, const fl_bf16* x, const int* mat_indices, int n_mats, const int32_t* seg_indptr,
                  const int32_t* lora_ids, int n_seg, int n_tokens, float scale, void* workspace, size_t workspace_bytes,
                  fl_stream stream, ShrinkInfo* info, const Follower* next) {
  fl_bf16* none[FL_MAX_MATS] = {};
  return sgmv_common(p, none, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace,
                     workspace_bytes, stream, nullptr, info, true, next);
}
}  // namespace sgmv

extern "C" {

int fl_lora_sgmv_multi(fl_pool* p, fl_bf16* const* ys, const fl_bf16* x, const int* mat_indices, int n_mats,
                       const int32_t* seg_indptr, const int32_t* lora_ids, int n_seg, int n_tokens,
                       float scale, void* workspace, size_t workspace_bytes, fl_stream stream) {
  return sgmv_common(p, ys, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace,
                     workspace_bytes, stream, nullptr);
}

int fl_lora_sgmv_qkv_append(fl_pool* p, fl_bf16* y_q, const fl_bf16* y_k, const fl_bf16* y_v, const fl_bf16* x,
                            int mat_q, int mat_k, int mat_v, const int32_t* seg_indptr, const int32_t* lora_ids,
                            int n_seg, int n_tokens, float scale, const int32_t* req_indptr,
                            const int32_t* kv_tbl_indptr, const uint32_t* kv_tbl, const int32_t* prefix_lens,
                            int n_req, int n_kv_heads, void* workspace, size_t workspace_bytes, fl_stream stream) {
  fl_bf16* ys[3] = {y_q, const_cast<fl_bf16*>(y_k), const_cast<fl_bf16*>(y_v)};
  const int mi[3] = {mat_q, mat_k, mat_v};
  const KvDest kv = {1, 2, req_indptr, kv_tbl_indptr, kv_tbl, prefix_lens, n_req, n_kv_heads};
  return sgmv_common(p, ys, x, mi, 3, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, workspace_bytes, stream, &kv);
}

int fl_lora_sgmv(fl_pool* p, fl_bf16* y, const fl_bf16* x, int mat_index,
                 const int32_t* seg_indptr, const int32_t* lora_ids, int n_seg, int n_tokens,
                 float scale, void* workspace, size_t workspace_bytes, fl_stream stream) {
  fl_bf16* ys[1] = {y};
  const int mi[1] = {mat_index};
  return fl_lora_sgmv_multi(p, ys, x, mi, 1, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace,
                            workspace_bytes, stream);
}

// ---------------------------------------------------------------- fl_lora_sgmv_static: no allocation anywhere
// The scratch that fl_lora_sgmv takes from its caller lives here instead, inside the library image.
// Every GPU that loads the library holds these FL_SGMV_STATIC_BYTES until the process exits.
}  // extern "C"

static __device__ __align__(256) unsigned char g_sgmv_static_scratch[FL_SGMV_STATIC_BYTES];

namespace {
constexpr int STATIC_MAX_DEVICES = 64;
void* g_static_scratch_addr[STATIC_MAX_DEVICES] = {};   // device address of the array, per device; one copy per process
}  // namespace

extern "C" {

int fl_lora_sgmv_static(fl_pool* p, fl_bf16* y, const fl_bf16* x, int mat_index,
                        const int32_t* seg_indptr, const int32_t* lora_ids, int n_seg, int n_tokens,
                        float scale, fl_stream stream) {
  if (!p || n_seg < 0 || n_tokens < 0) return FL_EINVAL;
  if (p->device < 0 || p->device >= STATIC_MAX_DEVICES) return FL_EINVAL;
  if (n_seg == 0 || n_tokens == 0) return FL_OK;      // nothing to do, as in fl_lora_sgmv
  if (fl_lora_sgmv_workspace(n_tokens, 1) > (size_t)FL_SGMV_STATIC_BYTES) return FL_ENOMEM;   // batch too large for the built-in scratch
  void* scratch = g_static_scratch_addr[p->device];
  if (!scratch) {
    // First call on this device: in host code the array's name is only a handle, so ask the runtime
    // for the array's address on the pool's device (which must be current for the query).
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != p->device) cudaSetDevice(p->device);
    const cudaError_t e = cudaGetSymbolAddress(&scratch, g_sgmv_static_scratch);
    if (prev != p->device && prev >= 0) cudaSetDevice(prev);
    if (e != cudaSuccess || !scratch) {
      p->last_cuda = (int)e;
      return FL_ECUDA;
    }
    g_static_scratch_addr[p->device] = scratch;
  }
  // Nothing in the scratch has to start at zero: the shrink kernel writes every partial sum that the
  // expand kernel reads, so whatever the previous call left behind is overwritten before use.
  return fl_lora_sgmv(p, y, x, mat_index, seg_indptr, lora_ids, n_seg, n_tokens, scale, scratch,
                      (size_t)FL_SGMV_STATIC_BYTES, stream);
}

}  // extern "C"
