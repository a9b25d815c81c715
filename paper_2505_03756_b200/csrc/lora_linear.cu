// Base projection with the LoRA branch folded in: y = x W + scale * (x A_i) B_i per segment (Eq. 1: W' = W + A B;
// Eq. 2: the same branch on the K/V projections), written once, never read back.
//
// A persistent tcgen05 GEMM.  A pair of CTAs on two neighbouring SMs (cta_group::2) walks tiles of 256 tokens x BN output
// columns: each CTA holds 128 token rows of x and half of the tile's columns of W, and the pair's tensor cores read both
// halves, so a k-step costs each SM two thirds of the shared-memory fill that a 128 x BN tile of its own would.  The
// accumulator lives in TMEM (each CTA its own rows, two buffers, so the epilogue of one tile overlaps the MMAs of the next).
// The LoRA branch is a few more k-steps into the same accumulator: the rank-rows of every adapter that overlaps the tile, 16
// to a unit and two units to a LoRA stage, against a matrix that holds in row t the shrink result of token t (slices
// summed, scaled, rounded to bf16) at the ranks of its own adapter and zeros elsewhere.  A tile thus needs no alignment with
// the segments.  The stages are spread over the second half of the tile's main stages: their place in the order of the
// sums is fixed, and a tile of many one-token segments fills its stages while the tensor cores work on.
// The kernel is also built for tiles of 128 tokens x 256 columns with a CTA each (G = 1), for batches whose second tile of 256 tokens
// would be mostly empty and cost the pairs a round.
//   warp 0       TMA producer: x tile [128 x 64] (K-major) and W tile [64 x BN/2] (N contiguous, as stored) per stage
//   warp 1       MMA issuer (of the pair's first CTA, for both)
//   warps 2-5    epilogue: TMEM -> bf16 -> y, or K and V rows straight into each token's pool block
//   warps 6-13   the V slots behind each request's last token (a share per CTA), then the LoRA stages, warps 6-9 the even ones,
//                10-13 the odd ones
// What bounds it: the tensor cores, and above them the power limit.  A layer step of 16 prompts (4907 tokens, 7B) went 737
// -> 665 us, of 4 prompts of 1024 new tokens (34B, rank 64) 1727 -> 1507 us against the tiles of 128 tokens per CTA before;
// with 28 one-token segments next to 4 prompts (7B, ranks 8 to 64) 734 -> 453 us, because a stage now takes the rank-rows of
// two to four segments and is filled side by side instead of one by one.
// Every mbarrier wait is bounded; a wait that gives up raises a sticky flag, the CTA drains its copies, meets its partner
// and frees its TMEM.  No multicast.
#include <cuda.h>
#include <string.h>
#include <algorithm>
#include "giveup.cuh"
#include "kv_tail.cuh"
#include "lora_skinny.cuh"
#include "mma_utils.cuh"
#include "pool.cuh"
#include "sgmv.cuh"
#include "tc_ptx.cuh"
#include "tmap.cuh"

namespace {

using namespace tc;

constexpr int LT_THREADS = 448;
constexpr int BM = 128;                          // token rows per CTA; a pair's tile has twice as many
constexpr int BK = 64;
constexpr int MAX_LIN = 3;                       // projections per launch (q, k, v share x)
constexpr int UNIT = 16;                         // rank-rows per entry of a tile's LoRA list: one k-step
constexpr int ER = 2 * UNIT;                     // rank-rows per LoRA stage
constexpr int MAX_UNITS = 2 * BM * (FL_MAX_RANK / UNIT);
constexpr int GROUP = 8;                         // LoRA stages whose row addresses are looked up together
constexpr int RASTER = 8;                        // token tiles that are walked together over a projection's columns
constexpr uint32_t A_BYTES = BM * BK * 2;        // x tile, K-major: 128 rows of 128 bytes
constexpr uint32_t B_GROUP = BK * 128;           // one 64-column group of a W tile: 64 k-rows of 128 bytes

template <int BN, int G>
struct Cfg {
  static constexpr int BH = BN / G;                           // columns of W this CTA loads
  static constexpr uint32_t B_BYTES = (BH / 64) * B_GROUP;
  static constexpr uint32_t STAGE = A_BYTES + B_BYTES;
  static constexpr int NS = G == 1 ? 3 : BN == 256 ? 5 : 7;
  // two LoRA stages side by side in one buffer of a main stage's layout: ranks 0-31 and 32-63 of every row
  static constexpr uint32_t OFF_EXT = NS * STAGE;
  static constexpr uint32_t OFF_ROWS = OFF_EXT + STAGE;       // B row addresses of two groups of LoRA stages
  static constexpr uint32_t OFF_LIST = OFF_ROWS + 2 * GROUP * ER * 8;
  static constexpr uint32_t OFF_BAR = OFF_LIST + MAX_UNITS * 8;
  static constexpr uint32_t SMEM = OFF_BAR + 512 + 1024;      // barriers and bookkeeping; slack for 1024-byte alignment
  static constexpr uint32_t TMEM_COLS = 2 * BN;               // two accumulators
  static_assert(TMEM_COLS == 512 || TMEM_COLS == 256, "TMEM allocations are powers of two");
  static_assert(SMEM <= 227 * 1024, "shared memory");
  static_assert(STAGE % 1024 == 0, "operand tiles start on 1024-byte boundaries");
};

struct LinArgs {
  PoolView pv;
  const float* v;              // shrink partial sums [projection][slice][token][rmax] ..
  const __nv_bfloat16* v16;    // .. or, where not null, the scaled result in bf16, [projection][token][rmax]
  int ksplit, rmax;
  float scale;
  const int32_t* seg_indptr;
  const int32_t* lora_ids;
  int n_seg, n_tokens, d_in;
  int n_mats;
  __nv_bfloat16* y[MAX_LIN];
  int wide[MAX_LIN];           // rows of y start on 32-byte boundaries
  int d_out[MAX_LIN], mat_index[MAX_LIN], n_tiles_n[MAX_LIN], tile_base[MAX_LIN + 1];
  int m_tiles;
  // K / V projections whose rows go straight into the requests' pool blocks (kv_side: -1 = rows go to y, 0 = K, 1 = V)
  int kv_side[MAX_LIN];
  const int32_t* req_indptr;
  const int32_t* tbl_indptr;
  const uint32_t* tbl;
  const int32_t* prefix_lens;
  int n_req, n_kv, bt;
};

struct LinMaps {
  CUtensorMap x;
  CUtensorMap w[MAX_LIN];
};

struct Tile {
  int j, m, n;       // projection, token tile, column tile
};
// Tiles run over the tokens first, RASTER token tiles at a time, then over the columns: the pairs' tiles in flight (74 on a
// B200) share about nine column slices of W and eight x tiles, and W is read from memory once per RASTER token tiles.
__device__ __forceinline__ Tile decode_tile(const LinArgs& a, int idx) {
  Tile t;
  t.j = 0;
  while (t.j + 1 < a.n_mats && idx >= a.tile_base[t.j + 1]) ++t.j;
  const int local = idx - a.tile_base[t.j], nt = a.n_tiles_n[t.j];
  const int g = local / (RASTER * nt), r = local - g * RASTER * nt;
  const int gm = min(RASTER, a.m_tiles - g * RASTER);
  t.n = r / gm;
  t.m = g * RASTER + (r - t.n * gm);
  return t;
}

// A LoRA unit: adapter (20 bits) | first rank / 16 (2) | rank-rows (5) | first token of the tile (9) | behind the last one (9)
__device__ __forceinline__ unsigned long long pack_unit(int lid, int q, int nr, int lo, int hi) {
  return (unsigned long long)lid << 25 | (unsigned long long)((uint32_t)q << 23 | (uint32_t)nr << 18 | (uint32_t)lo << 9 | (uint32_t)hi);
}
static_assert(FL_MAX_LORA_ID <= 1 << 20 && FL_MAX_RANK / UNIT <= 4 && 2 * BM < 512, "fields of a LoRA unit");

// Infinities and NaNs in an adapter's B rows stay out of a LoRA stage: times the zeros of the tile's other tokens they would make
// NaNs of these tokens' rows.  What they give their own token is added here to its row of the accumulator (columns from n0 on).
template <int BN, int RMAX>
__device__ __noinline__ void add_nonfinite_terms(const LinArgs& a, int j, int tok, int n0, uint32_t acc) {
  int lo = 0, hi = a.n_seg;                // first segment that ends behind tok
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a.seg_indptr[mid + 1] > tok) hi = mid; else lo = mid + 1;
  }
  const int lid = lo < a.n_seg && a.seg_indptr[lo] <= tok && tok < a.n_tokens ? a.lora_ids[lo] : -1, mat = a.mat_index[j], d_out = a.d_out[j];
  const LoraEntry* en = lid < 0 || (uint32_t)lid >= a.pv.dir_cap || mat >= a.pv.dir[lid].n_mats ? nullptr : a.pv.dir + lid;
  const int rank = en ? min(en->rank, RMAX) : 0;
  const LoraMat lm = rank > 0 ? en->mats[mat] : LoraMat{};
  for (int cb = 0; cb < BN; cb += 32) {
    uint32_t o[32];
    __syncwarp();
    tmem_ld32(acc + cb, o);
    tmem_wait_ld();
    for (int r = 0; r < rank; ++r) {
      const uint32_t gr = lm.b_row0 + r, blk = a.pv.tables[en->table_off + lm.b_tab + gr / lm.b_rpb];
      if (blk >= a.pv.n_blocks) continue;
      const uint4* b = reinterpret_cast<const uint4*>(a.pv.slab + (size_t)blk * a.pv.block_bytes + ((size_t)(gr % lm.b_rpb) * d_out + n0 + cb) * 2);
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (n0 + cb + 8 * h >= d_out) break;
        const uint4 q = b[h];
        if (nonfinite_chunk(q) == 0u) continue;
        float v = 0.f;
        if (a.v16) {
          v = __bfloat162float(a.v16[((size_t)j * a.n_tokens + tok) * RMAX + r]);
        } else {
          for (int sp = 0; sp < a.ksplit; ++sp) v += a.v[((size_t)(j * a.ksplit + sp) * a.n_tokens + tok) * RMAX + r];
          v = __bfloat162float(__float2bfloat16_rn(v * a.scale));
        }
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float bv = __uint_as_float(c & 1 ? w[c >> 1] & 0xffff0000u : w[c >> 1] << 16);
          if ((__float_as_uint(bv) & 0x7f800000u) == 0x7f800000u) o[8 * h + c] = __float_as_uint(fmaf(v, bv, __uint_as_float(o[8 * h + c])));
        }
      }
    }
    __syncwarp();
    tmem_st32(acc + cb, o);
  }
  tmem_wait_st();
}

template <int BN, int RMAX, int G>
__global__ void __launch_bounds__(LT_THREADS, 1) lora_linear_kernel(const __grid_constant__ LinArgs a, const __grid_constant__ LinMaps maps) {
  using C = Cfg<BN, G>;
  constexpr int TM = G * BM;                 // token rows of a tile
  constexpr int NS = C::NS, BH = C::BH;
  extern __shared__ unsigned char smem_raw[];
  // the swizzled operand tiles need 1024-byte alignment
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int crank = G == 2 ? (int)cluster_ctarank() : 0;
  const bool leader = crank == 0;
  enum { B_FULL = 0, B_EMPTY = NS, B_ACC_FULL = 2 * NS, B_ACC_EMPTY = B_ACC_FULL + 2, B_EFULL = B_ACC_EMPTY + 2, B_EEMPTY = B_EFULL + 2,
         B_LFULL = B_EEMPTY + 2, B_LEMPTY = B_LFULL + 2, B_IDLE = B_LEMPTY + 2, B_COUNT };
  const uint32_t bar0 = sbase + C::OFF_BAR;
  auto bar = [&](int k) { return bar0 + 8u * k; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + C::OFF_BAR + 8 * B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 8 * B_COUNT + 4);
  volatile int* n_ext_slot = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 8 * B_COUNT + 8);   // [2] LoRA stages of a tile
  int* scan = reinterpret_cast<int*>(smem + C::OFF_BAR + 8 * B_COUNT + 16);                          // [8] per filler warp
  volatile int* nonfinite_slot = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 8 * B_COUNT + 48);   // a B row held an infinity or NaN
  volatile int* partner_slot = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 8 * B_COUNT + 52);     // [2] its abort flag, its producer's stages
  static_assert(8 * B_COUNT + 16 + 32 + 16 <= 512, "bookkeeping area too small");

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(bar(B_FULL + s), 1);
      mbar_init(bar(B_EMPTY + s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar(B_ACC_FULL + b), 1);
      mbar_init(bar(B_ACC_EMPTY + b), 4 * G);      // the epilogue warps of both CTAs
      mbar_init(bar(B_EFULL + b), G);              // both CTAs' fillers
      mbar_init(bar(B_EEMPTY + b), 1);
      mbar_init(bar(B_LFULL + b), 1);
      mbar_init(bar(B_LEMPTY + b), 1);
    }
    mbar_init(bar(B_IDLE), 1);
    *abort_flag = 0;
    *nonfinite_slot = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (G == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(C::TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(C::TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (G == 2) cluster_sync();          // both CTAs' barriers exist
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Behind the shrink everything but v was finished before this kernel could start (the shrink lets it start after its own
  // wait); without one, the kernel before may still be writing x.
  if (a.n_seg == 0) pdl_wait();

  const int total = a.tile_base[a.n_mats];
  const int nk = (a.d_in + BK - 1) / BK;
  const int first = blockIdx.x / G, step = gridDim.x / G;        // pairs
  int fills = 0;                                                 // stages that this CTA's producer has issued

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (one lane): this CTA's halves; both CTAs' bytes are counted
    // on the first CTA's barrier
    if (lane == 0) {
      const uint32_t full0 = map_cluster_rank(bar(B_FULL), 0);
      int s = 0;
      uint32_t ph = 1;
      bool wrapped = false, ok = true;
      for (int idx = first; ok && idx < total; idx += step) {
        const Tile t = decode_tile(a, idx);
        const CUtensorMap* wm = &maps.w[t.j];
        const int row0 = t.m * TM + crank * BM, col0 = t.n * BN + crank * BH;
        for (int ks = 0; ks < nk; ++ks) {
          if (wrapped) ok = mbar_wait(bar(B_EMPTY + s), ph, abort_flag);
          if (!ok) break;
          if (leader) mbar_expect_tx(bar(B_FULL + s), G * C::STAGE);
          const uint32_t dst = sbase + s * C::STAGE, fb = full0 + 8u * s;
          tma_load_2d_group<G>(dst, &maps.x, fb, ks * BK, row0);
#pragma unroll
          for (int g = 0; g < BH / 64; ++g) tma_load_2d_group<G>(dst + A_BYTES + g * B_GROUP, wm, fb, col0 + g * 64, ks * BK);
          ++fills;
          if (++s == NS) { s = 0; ph ^= 1u; wrapped = true; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer: the whole warp runs converged, an elected lane issues
    if (leader) {
      constexpr uint32_t IDESC = G == 2 ? instr_desc_pair(BN, true) : instr_desc(BN, true);     // A (x, v) K-major, B (W, adapter rows) N-contiguous
      constexpr uint32_t HI = desc_hi(1024);
      auto wait_all = [&](uint32_t b, uint32_t parity) {
        if (__all_sync(0xffffffffu, mbar_try_cluster(b, parity))) return true;       // the common case: one test
        return __all_sync(0xffffffffu, mbar_wait_cluster(b, parity, abort_flag)) != 0;
      };
      const uint32_t a_lo0 = desc_lo(sbase, 16), b_lo0 = desc_lo(sbase + A_BYTES, B_GROUP);
      const uint32_t ea_lo0 = desc_lo(sbase + C::OFF_EXT, 16), eb_lo0 = desc_lo(sbase + C::OFF_EXT + A_BYTES, B_GROUP);
      int s = 0, es = 0;
      uint32_t ph = 0, eph = 0;
      bool ok = true;
      int k = 0;             // tiles of this pair so far
      const int half = nk / 2;
      for (int idx = first; ok && idx < total; idx += step, ++k) {
        const int buf = k & 1;
        if (k >= 2) ok = wait_all(bar(B_ACC_EMPTY + buf), (uint32_t)(((k >> 1) - 1) & 1));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * BN;
        int n_ext = 0, e = 0;
        for (int st = 0; st < nk; ++st) {
          ok = wait_all(bar(B_FULL + s), ph);
          if (!ok) break;
          tc_fence_after();
          const uint32_t a_lo = a_lo0 + s * (C::STAGE >> 4), b_lo = b_lo0 + s * (C::STAGE >> 4);
#pragma unroll
          for (int q = 0; q < BK / 16; ++q)
            umma_ss_group_elect<G>(d, a_lo + q * 2, HI, b_lo + q * (16 * 128 / 16), HI, IDESC, st > 0 || q > 0 ? 1u : 0u);
          umma_commit_group_elect<G>(bar(B_EMPTY + s));
          if (++s == NS) { s = 0; ph ^= 1u; }
          if (st >= half) {
            if (st == half && a.n_seg > 0) {
              ok = wait_all(bar(B_LFULL + buf), (uint32_t)((k >> 1) & 1));
              if (!ok) break;
              n_ext = n_ext_slot[buf];
              __syncwarp();
              if (lane == 0) mbar_arrive(bar(B_LEMPTY + buf));
            }
            const int due = (st - half + 1) * n_ext / (nk - half);
            for (; e < due; ++e) {
              ok = wait_all(bar(B_EFULL + es), eph);
              if (!ok) break;
              tc_fence_after();
#pragma unroll
              for (int q = 0; q < ER / 16; ++q)
                umma_ss_group_elect<G>(d, ea_lo0 + es * (ER * 2 / 16) + q * 2, HI, eb_lo0 + es * (ER * 128 / 16) + q * (16 * 128 / 16), HI, IDESC, 1u);
              umma_commit_group_elect<G>(bar(B_EEMPTY + es));
              es ^= 1;
              if (es == 0) eph ^= 1u;
            }
            if (!ok) break;
          }
        }
        if (ok) umma_commit_group_elect<G>(bar(B_ACC_FULL + buf));
      }
    }
  } else if (warp < 6) {
    // ------------------------------------------------ epilogue (128 threads; thread = token row = TMEM lane)
    const int quarter = warp & 3;            // the TMEM lanes this warp may touch
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t acc_empty0 = map_cluster_rank(bar(B_ACC_EMPTY), 0);
    bool ok = true;
    int k = 0;
    pdl_wait();
    for (int idx = first; idx < total; idx += step, ++k) {
      const Tile t = decode_tile(a, idx);
      const int buf = k & 1;
      const int tok = t.m * TM + crank * BM + row;
      const int d_out = a.d_out[t.j];
      const int n0 = t.n * BN;
      const int side = a.kv_side[t.j];
      // a K / V row belongs in its token's pool block: block and slot of the token's position, found while the
      // tile's MMAs are still running
      uint32_t kv_blk = 0;
      int kv_slot = -1;
      if (side >= 0 && tok < a.n_tokens) {
        int lo = 0, hi = a.n_req;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (a.req_indptr[mid] <= tok) lo = mid; else hi = mid;
        }
        const int pos = a.prefix_lens[lo] + (tok - a.req_indptr[lo]);
        const int entry = pos / a.bt, slot = pos - entry * a.bt;
        if (pos < 0 || tok < a.req_indptr[lo] || tok >= a.req_indptr[lo + 1] || entry >= a.tbl_indptr[lo + 1] - a.tbl_indptr[lo]) {
          atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
        } else {
          const uint32_t blk = a.tbl[a.tbl_indptr[lo] + entry];
          if (blk >= a.pv.n_blocks) {
            atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_BLOCK);
          } else {
            kv_blk = blk;
            kv_slot = slot;
          }
        }
      }
      ok = group_and(mbar_wait_cluster(bar(B_ACC_FULL + buf), (uint32_t)((k >> 1) & 1), abort_flag), 1, 128);
      if (!ok) break;
      tc_fence_after();
      __nv_bfloat16* yrow = side < 0 ? a.y[t.j] + (size_t)tok * d_out + n0 : nullptr;
      const bool wide = side < 0 && a.wide[t.j];
      // (a value of this tile's stages or of those of a tile before or behind it)
      if (__any_sync(0xffffffffu, *nonfinite_slot != 0)) add_nonfinite_terms<BN, RMAX>(a, t.j, tok, n0, lane_addr + buf * BN);
#pragma unroll 2
      for (int cb = 0; cb < BN; cb += 32) {
        uint32_t o[32];
        __syncwarp();
        tmem_ld32(lane_addr + buf * BN + cb, o);
        tmem_wait_ld();
        if (tok < a.n_tokens) {
          uint32_t pk[16];
#pragma unroll
          for (int c = 0; c < 16; ++c) pk[c] = pack_bf16(__uint_as_float(o[2 * c]), __uint_as_float(o[2 * c + 1]));
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int colg = n0 + cb + 8 * c;
            if (colg < d_out) {
              const uint4 q = make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
              if (wide) {                     // two chunks at a time: rows are whole multiples of 32 bytes
                if (!(c & 1)) st_global_v8(yrow + cb + 8 * c, pk + 4 * c);
              } else if (side < 0) {
                *reinterpret_cast<uint4*>(yrow + cb + 8 * c) = q;
              } else if (kv_slot >= 0) {
                // [K|V][kv head][slot][128] inside the block
                unsigned char* dst = a.pv.slab + (size_t)kv_blk * a.pv.block_bytes +
                                     ((size_t)(side * a.n_kv + colg / FL_HEAD_DIM) * a.bt + kv_slot) * (FL_HEAD_DIM * 2) +
                                     (colg % FL_HEAD_DIM) * 2;
                *reinterpret_cast<uint4*>(dst) = q;
              }
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8u * buf);
    }
  } else {
    // ------------------------------------------------ LoRA stages
    const int ft = tid - 192;                // 0..255
    const int et = ft & 127, slot = ft >> 7; // the buffer half (and the stages) of this group of four warps
    const uint32_t efull0 = map_cluster_rank(bar(B_EFULL), 0);
    unsigned long long* row_ptr = reinterpret_cast<unsigned long long*>(smem + C::OFF_ROWS);     // [2][GROUP * ER], 0 = no row
    unsigned long long* list = reinterpret_cast<unsigned long long*>(smem + C::OFF_LIST);
    unsigned char* as = smem + C::OFF_EXT;
    const uint32_t bs = sbase + C::OFF_EXT + A_BYTES;
    uint32_t ph = 1;                         // parity of this slot's B_EEMPTY
    bool used = false, ok = true;
    int count = 0;                           // LoRA stages of all tiles so far
    int k = 0;
    if (a.n_req > 0) clear_v_tails(a, (int)blockIdx.x, (int)gridDim.x, warp - 6, 8);       // while the shrink is still at work
    if (a.n_seg > 0) pdl_wait();             // v is the shrink's output
    for (int idx = first; a.n_seg > 0 && ok && idx < total; idx += step, ++k) {
      const Tile t = decode_tile(a, idx);
      const int tok0 = t.m * TM, tok1 = min(a.n_tokens, tok0 + TM);
      // ---- the tile's units, in segment order
      int lo_s = 0, hi_s = a.n_seg;          // first segment that ends behind tok0
      while (lo_s < hi_s) {
        const int mid = (lo_s + hi_s) >> 1;
        if (a.seg_indptr[mid + 1] > tok0) hi_s = mid; else lo_s = mid + 1;
      }
      int n_units = 0;
      for (int s0 = lo_s;; s0 += 256) {
        const int s = s0 + ft;
        int lo = tok1, hi = tok1, rank = 0, lid = -1;
        if (s < a.n_seg) {
          lo = max(a.seg_indptr[s], tok0);
          hi = min(a.seg_indptr[s + 1], tok1);
          if (lo < hi) {
            lid = a.lora_ids[s];
            if (lid >= 0) {
              if ((uint32_t)lid >= a.pv.dir_cap || a.pv.dir[lid].rank <= 0 || a.mat_index[t.j] >= a.pv.dir[lid].n_mats) {
                atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
              } else {
                rank = min(a.pv.dir[lid].rank, RMAX);
              }
            }
          }
        }
        const int cnt = (rank + UNIT - 1) / UNIT;
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int o = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += o;
        }
        if (lane == 31) scan[warp - 6] = incl;
        // (this barrier also keeps a new list from the old one's last readers)
        const bool last = group_and(s >= a.n_seg || lo >= tok1, 2, 256) || s0 + 256 >= a.n_seg;
        int at = n_units + incl - cnt;
        for (int w = 0; w < 8; ++w) {
          const int v = scan[w];
          if (w < warp - 6) at += v;
          n_units += v;
        }
        for (int q = 0; q < cnt; ++q, ++at)
          if (at < MAX_UNITS) list[at] = pack_unit(lid, q, min(UNIT, rank - UNIT * q), lo - tok0, hi - tok0);
        asm volatile("bar.sync 2, 256;" ::: "memory");
        if (last) break;
      }
      n_units = min(n_units, MAX_UNITS);      // (overlapping segments, which the interface rules out, could exceed it)
      const int n_ext = (n_units + 1) / 2;
      if (leader && ft == 0) {
        if (k >= 2) mbar_wait(bar(B_LEMPTY + (k & 1)), (uint32_t)(((k >> 1) - 1) & 1), abort_flag);
        n_ext_slot[k & 1] = n_ext;
        mbar_arrive(bar(B_LFULL + (k & 1)));
      }
      const int d_out = a.d_out[t.j], col0 = t.n * BN + crank * BH;
      const int mat = a.mat_index[t.j];
      // Addresses of a group's B rows, looked up side by side a group ahead of their use, and their columns asked into L2.
      auto find_rows = [&](int g) {
        for (int i = ft; i < GROUP * ER; i += 256) {
          const int u = 2 * (g * GROUP + i / ER) + (i % ER) / UNIT, r = i % UNIT;
          unsigned long long at = 0;
          if (u < n_units) {
            const unsigned long long x = list[u];
            if (r < (int)(x >> 18 & 31)) {
              const LoraEntry* en = a.pv.dir + (x >> 25);
              const LoraMat lm = en->mats[mat];
              const uint32_t gr = lm.b_row0 + (uint32_t)(x >> 23 & 3) * UNIT + r;
              const uint32_t blk = a.pv.tables[en->table_off + lm.b_tab + gr / lm.b_rpb];
              if (blk >= a.pv.n_blocks) {
                atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_BLOCK);
              } else if (col0 < d_out) {
                const unsigned char* p = a.pv.slab + (size_t)blk * a.pv.block_bytes + ((size_t)(gr % lm.b_rpb) * d_out + col0) * 2;
                at = reinterpret_cast<unsigned long long>(p);
                asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
#pragma unroll
                for (int g = 1; g < BH / 64; ++g)
                  if (col0 + 64 * g < d_out) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 128 * g));
              }
            }
          }
          row_ptr[(g & 1) * GROUP * ER + i] = at;
        }
      };
      if (n_ext > 0) find_rows(0);
      const int vrow = et >> 2, vch = et & 3;            // rows vrow + 32 i, ranks 8 vch .. of the stage's 32
      for (int e = 0; e < n_ext; ++e) {
        if (e % GROUP == 0) {
          // rows of this group are there (and nobody reads the other buffer any more)
          asm volatile("bar.sync 2, 256;" ::: "memory");
          if (e + GROUP < n_ext) find_rows(e / GROUP + 1);
        }
        if (((count + e) & 1) != slot) continue;
        if (used) ok = mbar_wait_cluster(bar(B_EEMPTY + slot), ph, abort_flag) && ok;
        used = true;
        ph ^= 1u;
        ok = group_and(ok, 3 + slot, 128);
        const unsigned long long* rp = row_ptr + (e % (2 * GROUP)) * ER;
        constexpr int CPR = BH / 8;                      // 16-byte chunks per row
#pragma unroll
        for (int i = 0; i < ER * CPR / 128; ++i) {
          const int c = et + 128 * i, r = c / CPR, ch = c % CPR;
          const unsigned long long at = ok ? rp[r] : 0ull;
          const bool have = at && col0 + ch * 8 < d_out;
          cp_async16(bs + (ch >> 3) * B_GROUP + (ER * slot + r) * 128 + (((ch & 7) ^ (r & 7)) << 4),
                     have ? reinterpret_cast<const unsigned char*>(at) + ch * 16 : a.pv.slab, have);
        }
        cp_async_commit();
        // shrink results of this CTA's 128 rows at the stage's ranks
        const int u = 2 * e + (vch >> 1);
        const unsigned long long x = u < n_units ? list[u] : 0ull;
        const int lo = (int)(x >> 9 & 511), hi = (int)(x & 511), r0 = (int)(x >> 23 & 3) * UNIT + 8 * (vch & 1);
        const bool live = 8 * (vch & 1) < (int)(x >> 18 & 31);
        if (a.v16) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int row = vrow + 32 * i, rt = crank * BM + row;
            const bool mine = live && rt >= lo && rt < hi;
            cp_async16(sbase + C::OFF_EXT + row * 128 + (((4 * slot + vch) ^ (row & 7)) << 4),
                       mine ? a.v16 + ((size_t)t.j * a.n_tokens + tok0 + rt) * RMAX + r0 : a.v16, mine);
          }
        } else {
          float4 f[4][2];
#pragma unroll
          for (int i = 0; i < 4; ++i) f[i][0] = f[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int sp = 0; sp < a.ksplit; ++sp) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int rt = crank * BM + vrow + 32 * i;
              if (live && rt >= lo && rt < hi) {
                const float4* src = reinterpret_cast<const float4*>(
                    a.v + ((size_t)(t.j * a.ksplit + sp) * a.n_tokens + tok0 + rt) * RMAX + r0);
                const float4 p = src[0], q = src[1];
                f[i][0].x += p.x; f[i][0].y += p.y; f[i][0].z += p.z; f[i][0].w += p.w;
                f[i][1].x += q.x; f[i][1].y += q.y; f[i][1].z += q.z; f[i][1].w += q.w;
              }
            }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int row = vrow + 32 * i;
            uint4 q;
            q.x = pack_bf16(f[i][0].x * a.scale, f[i][0].y * a.scale);
            q.y = pack_bf16(f[i][0].z * a.scale, f[i][0].w * a.scale);
            q.z = pack_bf16(f[i][1].x * a.scale, f[i][1].y * a.scale);
            q.w = pack_bf16(f[i][1].z * a.scale, f[i][1].w * a.scale);
            *reinterpret_cast<uint4*>(as + row * 128 + (((4 * slot + vch) ^ (row & 7)) << 4)) = q;
          }
        }
        cp_async_commit();
        cp_async_wait<1>();                              // the B rows; v16 may still be on its way
        // infinities and NaNs out of them (this thread's own pieces; add_nonfinite_terms has the reason)
        uint32_t found = 0;
#pragma unroll
        for (int i = 0; i < ER * CPR / 128; ++i) {
          const int c = et + 128 * i, r = c / CPR, ch = c % CPR;
          found |= nonfinite_chunk(ld_shared_v4(bs + (ch >> 3) * B_GROUP + (ER * slot + r) * 128 + (((ch & 7) ^ (r & 7)) << 4)));
        }
        if (found) {
          for (int i = 0; i < ER * CPR / 128; ++i) {
            const int c = et + 128 * i, r = c / CPR, ch = c % CPR;
            const uint32_t at = bs + (ch >> 3) * B_GROUP + (ER * slot + r) * 128 + (((ch & 7) ^ (r & 7)) << 4);
            const uint4 q = ld_shared_v4(at);
            st_shared_v4(at, make_uint4(finite_part(q.x), finite_part(q.y), finite_part(q.z), finite_part(q.w)));
          }
          // both CTAs' rows meet these columns
          *nonfinite_slot = 1;
          if (G == 2) st_cluster_u32(map_cluster_rank(smem_u32(const_cast<int*>(nonfinite_slot)), (uint32_t)(crank ^ 1)), 1u);
        }
        cp_async_wait<0>();
        fence_async_smem();                              // the tensor core reads shared memory through the async proxy
        asm volatile("bar.sync %0, 128;" ::"r"(3 + slot) : "memory");
        if (et == 0 && ok) mbar_arrive_cluster(efull0 + 8u * slot);
      }
      count += n_ext;
      ok = group_and(ok, 2, 256);
    }
    cp_async_wait<0>();
  }
  // ------------------------------------------------ teardown: neither CTA leaves while the other's MMAs or arrivals need it
  tc_fence_before();
  __syncthreads();
  if (G == 2) {
    if (tid == 0) {
      const uint32_t to = map_cluster_rank(smem_u32(const_cast<int*>(partner_slot)), (uint32_t)(crank ^ 1));
      st_cluster_u32(to, (uint32_t)*abort_flag);
      st_cluster_u32(to + 4, (uint32_t)fills);
    }
    __syncwarp();
    cluster_sync();
  }
  if (*abort_flag || (G == 2 && partner_slot[0])) {      // the same answer in both CTAs
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_WAIT_GAVE_UP);
    // Copies and MMAs still in flight use both CTAs' shared memory and TMEM; the first CTA's barriers count them all.
    if (leader && warp == 1) umma_commit_group_elect<G>(bar(B_IDLE));
    if (leader && tid == 0) {
      const long long armed = giveup::settle_pair(fills, G == 2 ? partner_slot[1] : fills, NS, [&](int s) { mbar_expect_tx(bar(B_FULL + s), C::STAGE); },
                                                  [&](int s) { mbar_complete_tx(bar(B_FULL + s), C::STAGE); });
      giveup::drain(armed, NS, [&](int s, uint32_t parity) { return mbar_try_cluster(bar(B_FULL + s), parity); });
      giveup::drain(1, 1, [&](int, uint32_t parity) { return mbar_try_cluster(bar(B_IDLE), parity); });
    }
    __syncthreads();
    if (G == 2) cluster_sync();
  }
  if (warp == 1) {
    tc_fence_after();
    if constexpr (G == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS) : "memory");
  }
}

template <int BN, int RMAX, int G>
int launch_linear(fl_pool* p, const LinArgs& a, const LinMaps& maps, cudaStream_t st) {
  using C = Cfg<BN, G>;
  static bool configured[16] = {};
  if (!configured[p->device & 15]) {
    FL_CUDA(p, cudaFuncSetAttribute(lora_linear_kernel<BN, RMAX, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    configured[p->device & 15] = true;
  }
  const int total = a.tile_base[a.n_mats];
  const unsigned groups = (unsigned)std::min(total, p->sm_count / G);
  FL_CUDA(p, launch_pdl_cluster(lora_linear_kernel<BN, RMAX, G>, dim3(G * groups), dim3(G), dim3(LT_THREADS), C::SMEM, st, a, maps));
  FL_CUDA(p, cudaGetLastError());
  return FL_OK;
}

template <int BN, int G>
int launch_rank(fl_pool* p, const LinArgs& a, const LinMaps& maps, cudaStream_t st, int rmax) {
  return rmax == 16 ? launch_linear<BN, 16, G>(p, a, maps, st)
       : rmax == 32 ? launch_linear<BN, 32, G>(p, a, maps, st) : launch_linear<BN, 64, G>(p, a, maps, st);
}
int launch_width(fl_pool* p, const LinArgs& a, const LinMaps& maps, cudaStream_t st, int bn, int group, int rmax) {
  return group == 1 ? launch_rank<256, 1>(p, a, maps, st, rmax)
       : bn == 256 ? launch_rank<256, 2>(p, a, maps, st, rmax) : launch_rank<128, 2>(p, a, maps, st, rmax);
}

}  // namespace

extern "C" {

size_t fl_lora_linear_workspace(int n_tokens, int n_mats) {
  if (n_tokens <= 0 || n_mats <= 0) return 256;
  return fl_lora_sgmv_workspace(n_tokens, n_mats);      // the shrink's results
}

}  // extern "C"

namespace {

struct LinKv {        // K and V projections of the call whose rows go into pool blocks
  int k_slot, v_slot;
  const int32_t* req_indptr;
  const int32_t* tbl_indptr;
  const uint32_t* tbl;
  const int32_t* prefix_lens;
  int n_req, n_kv;
  fl_bf16* tmp_k;     // [n_tokens, n_kv * 128] each: needed by batches of short segments only
  fl_bf16* tmp_v;
};

int linear_common(fl_pool* p, fl_bf16* const* ys_in, const fl_bf16* x, const fl_bf16* const* ws, const int* mat_indices,
                  int n_mats, const int32_t* seg_indptr, const int32_t* lora_ids, int n_seg, int n_tokens,
                  float scale, void* workspace, size_t workspace_bytes, fl_stream stream, const LinKv* kv) {
  if (!p || n_mats < 1 || n_mats > MAX_LIN || n_seg < 0 || n_tokens < 0 || !ys_in || !ws || !mat_indices) return FL_EINVAL;
  fl_bf16* ys[MAX_LIN] = {};
  for (int j = 0; j < n_mats; ++j) ys[j] = ys_in[j];
  if (n_tokens == 0) return FL_OK;
  if (!x || !workspace || (n_seg > 0 && (!seg_indptr || !lora_ids))) return FL_EINVAL;
  if (p->n_mats == 0) return FL_EBADID;           // the projection shapes come with the first registered adapter
  const size_t v_bytes = fl_lora_linear_workspace(n_tokens, n_mats);
  if (workspace_bytes < v_bytes) return FL_ENOMEM;
  LinArgs a;
  memset(&a, 0, sizeof(a));
  a.pv = p->view();
  for (int j = 0; j < n_mats; ++j) {
    const int mi = mat_indices[j];
    const bool to_pool = kv && (j == kv->k_slot || j == kv->v_slot);
    if (mi < 0 || mi >= p->n_mats || (!ys[j] && !to_pool) || !ws[j]) return FL_EINVAL;
    if (p->mats[mi].d_in != p->mats[mat_indices[0]].d_in) return FL_EINVAL;   // the projections share x
    a.y[j] = reinterpret_cast<__nv_bfloat16*>(ys[j]);
    a.mat_index[j] = mi;
    a.d_out[j] = p->mats[mi].d_out;
  }
  a.d_in = p->mats[mat_indices[0]].d_in;
  a.n_mats = n_mats;
  a.seg_indptr = seg_indptr;
  a.lora_ids = lora_ids;
  a.n_seg = n_seg;
  a.n_tokens = n_tokens;
  a.scale = scale;
  a.v = reinterpret_cast<const float*>(workspace);
  // Up to 256 tokens another kernel may be the faster one, which streams W once for all of them (skinny::serves).
  // Segments of a few tokens each (a large decode batch): a tile would take a LoRA stage per segment or two, each for a
  // handful of rows.  Then the GEMM computes x W alone and the segmented projection adds the LoRA term to y afterwards.
  // A batch of one tile takes up to 16 stages all the same, and is rounded once.
  const int rank_max = p->max_rank <= 16 ? 16 : (p->max_rank <= 32 ? 32 : 64);
  const bool few = skinny::serves(p, a.d_out, n_mats, a.d_in, n_tokens, n_seg, rank_max);
  const bool hybrid = !few && n_seg > 0 && n_tokens <= 16 * n_seg && (n_tokens > 2 * BM || n_seg * rank_max > 16 * ER);
  if (hybrid) a.n_seg = 0;
  for (int j = 0; j < MAX_LIN; ++j) a.kv_side[j] = -1;
  if (kv) {
    const size_t per_tok = (size_t)2 * kv->n_kv * FL_HEAD_DIM * 2;
    if (kv->n_kv < 1 || kv->n_req < 1 || p->block_bytes % per_tok != 0 || kv->k_slot == kv->v_slot) return FL_EINVAL;
    if (!kv->req_indptr || !kv->tbl_indptr || !kv->tbl || !kv->prefix_lens) return FL_EINVAL;
    for (int side = 0; side < 2; ++side) {
      const int slot = side ? kv->v_slot : kv->k_slot;
      if (slot < 0 || slot >= n_mats || a.d_out[slot] != kv->n_kv * FL_HEAD_DIM) return FL_EINVAL;
      if (n_seg > 0 && n_tokens <= 16 * n_seg && !(side ? kv->tmp_v : kv->tmp_k)) return FL_EINVAL;   // whichever kernel serves the batch
      if (hybrid) {      // x W goes to a scratch row first; the segmented projection then stores base + LoRA term in the pool
        fl_bf16* tmp = side ? kv->tmp_v : kv->tmp_k;
        ys[slot] = tmp;
        a.y[slot] = reinterpret_cast<__nv_bfloat16*>(tmp);
      } else {
        a.kv_side[slot] = side;
      }
    }
    a.req_indptr = kv->req_indptr;
    a.tbl_indptr = kv->tbl_indptr;
    a.tbl = kv->tbl;
    a.prefix_lens = kv->prefix_lens;
    a.n_req = hybrid ? 0 : kv->n_req;       // (0: no row of this kernel goes into a block)
    a.n_kv = kv->n_kv;
    a.bt = (int)(p->block_bytes / per_tok);
  }
  // Tiles of 256 or 128 columns per pair of CTAs, or 128 tokens x 256 columns per CTA: the one whose rounds over the SMs cost less.  All are
  // bound by the 64 bytes per clock that an SM gets from L2: 32 KB per k-step for a pair's 256 columns, 24 KB for its 128 (a round of
  // d_in 4096 takes 20 and 16.5 us), 48 KB for a CTA by itself.  That one is for batches of 257 to 384 tokens, whose second tile of 256
  // is mostly empty but costs the pairs a second round (q, k, v of 300 tokens, one adapter of rank 16: 34B 90 -> 78 us, 7B 52 -> 47).
  int bn = 256, group = 2;
  {
    auto rounds = [&](int rows, int w, int slots) {
      long t = 0;
      for (int j = 0; j < n_mats; ++j) t += (long)((n_tokens + rows - 1) / rows) * ((a.d_out[j] + w - 1) / w);
      return (t + slots - 1) / slots;
    };
    const int pairs = std::max(1, p->sm_count / 2);
    const long wide = rounds(2 * BM, 256, pairs) * 100, narrow = rounds(2 * BM, 128, pairs) * 82, single = rounds(BM, 256, p->sm_count) * 150;
    if (narrow < wide) bn = 128;
    if (single < std::min(wide, narrow)) { bn = 256; group = 1; }
  }
  a.m_tiles = (n_tokens + group * BM - 1) / (group * BM);
  for (int j = 0; j < n_mats; ++j) a.wide[j] = (reinterpret_cast<uintptr_t>(a.y[j]) & 31) == 0 && a.d_out[j] % 16 == 0;
  a.tile_base[0] = 0;
  for (int j = 0; j < n_mats; ++j) {
    a.n_tiles_n[j] = (a.d_out[j] + bn - 1) / bn;
    a.tile_base[j + 1] = a.tile_base[j] + a.m_tiles * a.n_tiles_n[j];
  }
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != p->device) cudaSetDevice(p->device);
  const cudaStream_t st = (cudaStream_t)stream;
  int rc = FL_OK;
  do {
    if (few) {
      skinny::Args k;
      memset(&k, 0, sizeof(k));
      k.pv = a.pv;
      k.v = reinterpret_cast<const __nv_bfloat16*>(a.v);
      k.seg_indptr = seg_indptr;
      k.lora_ids = lora_ids;
      k.n_seg = n_seg;
      k.n_tokens = n_tokens;
      k.d_in = a.d_in;
      k.n_mats = n_mats;
      for (int j = 0; j < n_mats; ++j) {
        k.y[j] = a.y[j];
        k.d_out[j] = a.d_out[j];
        k.mat_index[j] = a.mat_index[j];
        k.kv_side[j] = a.kv_side[j];
      }
      k.req_indptr = a.req_indptr;
      k.tbl_indptr = a.tbl_indptr;
      k.tbl = a.tbl;
      k.prefix_lens = a.prefix_lens;
      k.n_req = a.n_req;
      k.n_kv = a.n_kv;
      k.bt = a.bt;
      k.rmax = n_seg > 0 ? rank_max : 16;
      sgmv::ShrinkInfo info = {1, k.rmax, false};
      if (n_seg > 0) {
        // Above rank 16 and on wide layers the tcgen05 shrink is the faster one for segments above a few tokens (q, k, v of 128 tokens, one
        // segment: rank 64 7B 34.0 and 27.2 us, 34B 53 and 45; rank 32 28.4 and 27.5, 46 and 44; 40 tokens 25.8 and 25.2, 43 and 42;
        // but on a layer of 1024 values, 112 tokens, 19.4 and 20.5).
        const bool tc = rank_max > 16 && p->sgmv_shrink_kind == 0 && n_tokens > 16 * n_seg && a.d_in >= 2048;
        const sgmv::Follower next = skinny::footprint(p, k);
        rc = tc ? sgmv::shrink(p, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, v_bytes, stream, &info)
                : sgmv::shrink_scaled(p, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, v_bytes, stream, &info, &next);
        if (rc != FL_OK) break;
      }
      rc = skinny::launch(p, k, x, reinterpret_cast<const void* const*>(ws), st);
      break;
    }
    alignas(64) LinMaps maps;
    {
      const uint64_t dims[2] = {(uint64_t)a.d_in, (uint64_t)n_tokens};
      const uint64_t strides[1] = {(uint64_t)a.d_in * 2};
      const uint32_t box[2] = {BK, BM};
      rc = tmap::encode_bf16(&maps.x, x, 2, dims, strides, box);
      if (rc != FL_OK) break;
    }
    for (int j = 0; j < n_mats && rc == FL_OK; ++j) {
      const uint64_t dims[2] = {(uint64_t)a.d_out[j], (uint64_t)a.d_in};
      const uint64_t strides[1] = {(uint64_t)a.d_out[j] * 2};
      const uint32_t box[2] = {64, BK};
      rc = tmap::encode_bf16(&maps.w[j], ws[j], 2, dims, strides, box);
    }
    for (int j = n_mats; j < MAX_LIN; ++j) maps.w[j] = maps.w[0];
    if (rc != FL_OK) break;
    sgmv::ShrinkInfo info = {1, rank_max, false};
    if (hybrid) {
      // y = x W from the GEMM alone, then the segmented projection adds the LoRA term to it
      a.ksplit = 1;
      a.rmax = info.rmax;
      rc = launch_width(p, a, maps, st, bn, group, info.rmax);
      if (rc != FL_OK) break;
      if (kv && n_mats == 3 && kv->k_slot == 1 && kv->v_slot == 2)
        rc = fl_lora_sgmv_qkv_append(p, ys[0], ys[1], ys[2], x, mat_indices[0], mat_indices[1], mat_indices[2], seg_indptr,
                                     lora_ids, n_seg, n_tokens, scale, kv->req_indptr, kv->tbl_indptr, kv->tbl,
                                     kv->prefix_lens, kv->n_req, kv->n_kv, workspace,
                                     v_bytes, stream);
      else if (kv)
        rc = FL_EINVAL;
      else
        rc = fl_lora_sgmv_multi(p, ys, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace,
                                v_bytes, stream);
      break;
    }
    if (n_seg > 0) {
      // Two shrinks, in tiles of 16 tokens and of 64 or 128 tokens.  Above rank 16 and on wide layers, where the second one runs on tcgen05, it is the
      // better one for all but segments of a few tokens (q, k, v on 7B, rank 64: 320 tokens, 40 per segment 53 and 35 us; 512, 64 per segment 92
      // and 60; 1920, 80 per segment 148 and 138; rank 32, 512 tokens, 64 per segment 61 and 53; 1024 tokens and more the same).  At rank 16 the
      // second one reads the adapters' rows less often, but where it leaves fp32 slices of d_in a LoRA stage that sums them takes 5600
      // cycles instead of 1500: the first one is the better one as long as a segment's x and the rows that it reads again are few
      // (7B, 288 tokens, 20 per segment 64 and 67 us, 72 per segment 59 and 54; 1000 tokens of 1024 values, 100 per segment 23 and 25).
      // On layers of 1024 values so it is at higher ranks (a layer step, rank 32, 200 tokens in one segment 42.4 and 47.3 us, 512 in four 43.6 and
      // 47.1; rank 64, 256 in four 50.3 and 55.4, but 512 in one 65 and 56).
      const bool tc = rank_max > 16 && p->sgmv_shrink_kind == 0 && a.d_in >= 2048;
      const bool final = n_tokens <= 16 * n_seg || (!tc && (double)n_tokens / n_seg * a.d_in <= (rank_max == 16 ? 1.7e5 : rank_max == 32 ? 3e5 : 1.32e5));
      rc = final ? sgmv::shrink_scaled(p, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, v_bytes,
                                       stream, &info, nullptr)
                 : sgmv::shrink(p, x, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, v_bytes, stream, &info);
      if (rc != FL_OK) break;
      if (info.final) a.v16 = reinterpret_cast<const __nv_bfloat16*>(workspace);
    }
    a.ksplit = info.ksplit;
    a.rmax = info.rmax;
    rc = launch_width(p, a, maps, st, bn, group, info.rmax);
  } while (0);
  if (prev != p->device && prev >= 0) cudaSetDevice(prev);
  return rc;
}

}  // namespace

extern "C" {

int fl_lora_linear_multi(fl_pool* p, fl_bf16* const* ys, const fl_bf16* x, const fl_bf16* const* ws, const int* mat_indices,
                         int n_mats, const int32_t* seg_indptr, const int32_t* lora_ids, int n_seg, int n_tokens,
                         float scale, void* workspace, size_t workspace_bytes, fl_stream stream) {
  return linear_common(p, ys, x, ws, mat_indices, n_mats, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace,
                       workspace_bytes, stream, nullptr);
}

int fl_lora_linear_qkv_append(fl_pool* p, fl_bf16* y_q, const fl_bf16* x, const fl_bf16* w_q, const fl_bf16* w_k,
                              const fl_bf16* w_v, int mat_q, int mat_k, int mat_v, const int32_t* seg_indptr,
                              const int32_t* lora_ids, int n_seg, int n_tokens, float scale, const int32_t* req_indptr,
                              const int32_t* kv_tbl_indptr, const uint32_t* kv_tbl, const int32_t* prefix_lens, int n_req,
                              int n_kv_heads, fl_bf16* scratch_k, fl_bf16* scratch_v, void* workspace,
                              size_t workspace_bytes, fl_stream stream) {
  fl_bf16* ys[3] = {y_q, nullptr, nullptr};
  const fl_bf16* ws[3] = {w_q, w_k, w_v};
  const int mi[3] = {mat_q, mat_k, mat_v};
  const LinKv kv = {1, 2, req_indptr, kv_tbl_indptr, kv_tbl, prefix_lens, n_req, n_kv_heads, scratch_k, scratch_v};
  return linear_common(p, ys, x, ws, mi, 3, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, workspace_bytes,
                       stream, &kv);
}

int fl_lora_linear(fl_pool* p, fl_bf16* y, const fl_bf16* x, const fl_bf16* w, int mat_index,
                   const int32_t* seg_indptr, const int32_t* lora_ids, int n_seg, int n_tokens,
                   float scale, void* workspace, size_t workspace_bytes, fl_stream stream) {
  fl_bf16* ys[1] = {y};
  const fl_bf16* ws[1] = {w};
  const int mi[1] = {mat_index};
  return fl_lora_linear_multi(p, ys, x, ws, mi, 1, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace,
                              workspace_bytes, stream);
}

}  // extern "C"
