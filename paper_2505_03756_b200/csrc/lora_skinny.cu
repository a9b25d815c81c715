// y = x W + scale * (x A_i) B_i (Eq. 1, Eq. 2) for batches of at most 256 tokens: decode steps and short prompts.
//
// Such a call is bound by streaming W once and, with many adapters, their B rows.  One CTA owns 128 output columns for
// ALL tokens (one or two row tiles of 128) and a slice of d_in; the CTAs of a column tile form a cluster that adds its
// partial sums through distributed shared memory, so that narrow projections still use every SM and no partial sum goes
// through global memory.
//   warp 0      TMA producer: x tile [tokens x 64] and W tile [64 x 128] per stage, ring of as many stages as fit
//   warp 1      MMA issuer of x W
//   warps 2-5   list of the LoRA stages, a share of them, a share of the V slots to clear, then the epilogue (thread = token row)
//   up to 8 more the other LoRA stages, four warps to a stage
//   last warp   MMA issuer of the LoRA term, into an accumulator of its own
// The LoRA term is one more product over a long, sparse k: the rank-rows of every adapter of the batch one after the
// other, 64 to a stage, against a matrix that holds in row t the shrink result of token t at the ranks of its own adapter
// and zeros elsewhere.  A stage has the layout of a main stage: B rows through the block table in place of W rows,
// shrink results in place of x, both by cp.async (a masked copy writes the zeros).  A batch whose every token uses
// another adapter is thus no special case, and since the two accumulators have one issuer each, the order of either's
// sums does not depend on which stage is ready first.
// Launched behind the shrink, the kernel streams W and B rows while the shrink still runs: the shrink lets it start only
// after everything before the shrink is done, and only v is waited for.
// Tokens are the tensor core's rows although most of its 128 rows may be empty: with W as the row operand and the tokens
// as columns an MMA step took about 170 cycles however few the tokens, against 64 here.
// What bounds it: W.  Of one 7B layer's projections the W stream alone takes 18.6 us (q, k, v) and 8.3 us (o) when nothing
// is computed, the calls take 25 and 17 us; before, with the GEMM for long batches followed by the segmented projection,
// they took 44 and 32 us.  The rest is the shrink's chain of look-ups in front and the sum over the cluster behind.
// Every mbarrier wait is bounded; a wait that gives up raises a sticky flag and the CTA still meets its cluster's
// barriers, where it tells the others that its part of the sum is missing (none of them stores anything then), drains its copies
// and frees its TMEM.  No multicast.
#include <cuda.h>
#include <string.h>
#include <algorithm>
#include "giveup.cuh"
#include "kv_tail.cuh"
#include "lora_skinny.cuh"
#include "mma_utils.cuh"
#include "tc_ptx.cuh"
#include "tmap.cuh"

namespace {

using namespace tc;

constexpr int FILLERS = 3;                         // groups of four warps that fill LoRA stages
constexpr int MAX_THREADS = 96 + 128 * FILLERS;    // a launch brings one group per slot of the LoRA ring and no more: fewer
                                                   // registers let the CTA start beside CTAs of the shrink

constexpr int BN = 128, BK = 64;                   // columns per CTA; d_in (or rank-rows) per stage
constexpr uint32_t W_BYTES = BK * BN * 2, W_GROUP = BK * 128;      // two groups of 64 columns
constexpr int MAX_NS = 12, MAX_NE = FILLERS;
constexpr int UNIT = 16;                           // rank-rows per entry of the LoRA list: one k-step
constexpr int UNITS_PER_TOKEN = FL_MAX_RANK / UNIT;      // every token its own adapter of the highest rank
constexpr int GROUP = 4;                           // LoRA stages whose row addresses a group of warps looks up together
constexpr int MAX_SPLIT = 8;
// Not all of an SM's 227 KB: what is left lets the CTA start beside CTAs of the shrink before it (a decode step of one token:
// 57 us a layer at 180 KB, 61 at 227 KB, 59 at 113 KB; of 48 tokens the same at 180 and 227 KB, 2 % more at 113 KB).
// Above 128 tokens a stage is mostly x, and the ring needs all of it.
constexpr uint32_t SMEM_LIMIT = 180 * 1024, SMEM_MAX = 227 * 1024;

struct LoraUnit {        // 16 rank-rows of one segment's adapter
  uint16_t lo, hi;       // the segment's tokens
  uint16_t r0, nr;       // first rank, rank-rows (1..16; 0 = padding of the last stage)
  uint32_t tab, row0;    // first table entry of the stream the B rows are in, row of rank r0 inside it
};

struct KArgs {
  skinny::Args s;
  int tile_base[skinny::MAX_LIN + 1];
  int npad, ns, ne, split;        // tokens rounded up to 16, stages of the two rings, CTAs per column tile
  uint32_t tmem_cols;
};
struct Maps {
  CUtensorMap x;
  CUtensorMap w[skinny::MAX_LIN];
};

enum { B_FULL = 0, B_EMPTY = MAX_NS, B_EFULL = 2 * MAX_NS, B_EEMPTY = B_EFULL + MAX_NE, B_LIST = B_EEMPTY + MAX_NE, B_ACC, B_IDLE, B_COUNT };
// behind the two rings: barriers and bookkeeping | B row addresses, two sets of stages per group of warps | list of LoRA units
constexpr uint32_t BOOK_BYTES = 512, ROWS_BYTES = FILLERS * 2 * GROUP * BK * 8;
static_assert(8 * B_COUNT + 48 <= BOOK_BYTES, "bookkeeping area too small");
static_assert(sizeof(LoraUnit) == 16, "one 16-byte shared-memory access per unit");

// The product of the LoRA stages takes every token through every unit of a stage, times zeros where the unit is another adapter's: an
// infinity or NaN in that adapter's B rows makes a NaN of them.  Where a stage held such a value, the sums that came out as one are
// taken again here, over the units of this CTA's stages that are the token's own, and put back into the accumulator.  The fillers
// look for the values while v is on its way; looked for in the sums, by the epilogue, they cost a decode step of one token 49.0 ->
// 50.2 us.
__device__ __noinline__ void redo_lora_sums(const skinny::Args& a, const LoraUnit* list, uint32_t rpb, int crank, int split, int n_stages,
                                            int j, int t, int n0, uint32_t acc) {
  const __nv_bfloat16* v = a.v + ((size_t)j * a.n_tokens + t) * a.rmax;
  const int d_out = a.d_out[j];
  for (int c = 0; c < BN; c += 16) {
    uint32_t l[16];
    __syncwarp();
    tmem_ld16(acc + c, l);
    tmem_wait_ld();
    uint32_t top = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) top = max(top, l[q] & 0x7fffffffu);
    if (t < a.n_tokens && top >= 0x7f800000u) {
      float f[16] = {};
      for (int i = 0; i < 4 * n_stages; ++i) {
        const LoraUnit u = list[4 * (crank + (i >> 2) * split) + (i & 3)];
        if (t < u.lo || t >= u.hi) continue;
        for (int r = 0; r < u.nr; ++r) {
          const uint32_t gr = u.row0 + r, blk = a.pv.tables[u.tab + gr / rpb];
          if (blk >= a.pv.n_blocks) continue;                     // (left out of the product too)
          const uint4* b = reinterpret_cast<const uint4*>(a.pv.slab + (size_t)blk * a.pv.block_bytes + ((size_t)(gr % rpb) * d_out + n0 + c) * 2);
          const float s = __bfloat162float(v[u.r0 + r]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (n0 + c + 8 * h >= d_out) continue;
            const uint4 w = b[h];
            const float2 p[4] = {unpack_bf16(w.x), unpack_bf16(w.y), unpack_bf16(w.z), unpack_bf16(w.w)};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              f[8 * h + 2 * e] = fmaf(s, p[e].x, f[8 * h + 2 * e]);
              f[8 * h + 2 * e + 1] = fmaf(s, p[e].y, f[8 * h + 2 * e + 1]);
            }
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 16; ++q) l[q] = __float_as_uint(f[q]);
    }
    __syncwarp();
    tmem_st16(acc + c, l);
  }
  tmem_wait_st();
}

__global__ void __launch_bounds__(MAX_THREADS, 1) lora_skinny_kernel(const __grid_constant__ KArgs ka, const __grid_constant__ Maps maps) {
  const skinny::Args& a = ka.s;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ns = ka.ns, ne = ka.ne, npad = ka.npad, split = ka.split;
  const int mt = npad > 128 ? 2 : 1;                                // row tiles
  const uint32_t x_bytes = (uint32_t)npad * 128, stage_bytes = x_bytes + W_BYTES;      // [x rows][W rows]
  const uint32_t off_ext = ns * stage_bytes, off_book = off_ext + ne * stage_bytes;
  const uint32_t bar0 = sbase + off_book;
  auto bar = [&](int k) { return bar0 + 8u * k; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + off_book + 8 * B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + off_book + 8 * B_COUNT + 4);
  volatile int* n_stage_slot = reinterpret_cast<volatile int*>(smem + off_book + 8 * B_COUNT + 8);
  int* scan = reinterpret_cast<int*>(smem + off_book + 8 * B_COUNT + 16);      // [4], one per filler warp
  volatile int* rpb_slot = reinterpret_cast<volatile int*>(smem + off_book + 8 * B_COUNT + 12);
  volatile int* nonfinite_slot = reinterpret_cast<volatile int*>(smem + off_book + 8 * B_COUNT + 36);  // a B row of a stage holds an infinity or NaN
  volatile int* told_slot = reinterpret_cast<volatile int*>(smem + off_book + 8 * B_COUNT + 32);       // a CTA of the cluster has no part of the sum
  unsigned long long* row_ptr = reinterpret_cast<unsigned long long*>(smem + off_book + BOOK_BYTES);     // [group][2][GROUP * BK], 0 = no row
  LoraUnit* list = reinterpret_cast<LoraUnit*>(smem + off_book + BOOK_BYTES + ROWS_BYTES);
  const int max_units = npad * UNITS_PER_TOKEN;

  const int crank = blockIdx.x % split;            // clusters are `split` consecutive CTAs
  const int tile = blockIdx.x / split;
  int j = 0;
  while (j + 1 < a.n_mats && tile >= ka.tile_base[j + 1]) ++j;
  const int n0 = (tile - ka.tile_base[j]) * BN;
  const int d_out = a.d_out[j];
  const int nk = (a.d_in + BK - 1) / BK;
  const int k0 = crank * nk / split, k1 = (crank + 1) * nk / split;

  if (tid == 0) {
    for (int s = 0; s < ns; ++s) {
      mbar_init(bar(B_FULL + s), 1);
      mbar_init(bar(B_EMPTY + s), 1);
    }
    for (int e = 0; e < ne; ++e) {
      mbar_init(bar(B_EFULL + e), 128);
      mbar_init(bar(B_EEMPTY + e), 1);
    }
    mbar_init(bar(B_LIST), 1);
    mbar_init(bar(B_ACC), 2);            // both issuers
    mbar_init(bar(B_IDLE), 2);
    *abort_flag = 0;
    *told_slot = 0;
    *nonfinite_slot = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(ka.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tmem_lora = tmem + mt * BN;
  // Behind the shrink everything but v was finished before this kernel could start (the shrink lets it start after its own
  // wait); without one, the kernel before may still be writing x.
  if (a.n_seg == 0) pdl_wait();

  constexpr uint32_t IDESC = instr_desc(BN, true);       // A (x, v) K-major, B (W, adapter rows) N-contiguous
  constexpr uint32_t HI = desc_hi(1024);
  // four k-steps of one stage into the accumulators at d
  auto issue_stage = [&](uint32_t stage, uint32_t d, bool first, int steps) {
    const uint32_t a_lo = desc_lo(stage, 16), b_lo = desc_lo(stage + x_bytes, W_GROUP);
    for (int m = 0; m < mt; ++m) {
#pragma unroll
      for (int q = 0; q < BK / 16; ++q)
        if (q < steps)
          umma_ss_elect(d + m * BN, a_lo + m * (128 * 128 / 16) + q * 2, HI, b_lo + q * (16 * 128 / 16), HI, IDESC, first && q == 0 ? 0u : 1u);
    }
  };
  auto wait_all = [&](uint32_t b, uint32_t parity) {
    if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;       // the common case: one test
    return __all_sync(0xffffffffu, mbar_wait(b, parity, abort_flag)) != 0;
  };

  bool ok = true;
  int fills = 0;                           // stages that the producer has armed
  int n_stages = 0;                        // LoRA stages of this CTA (known to the LoRA roles)
  const int filler = (warp - 2) >> 2;      // group of four warps
  const int et = (tid - 64) & 127;         // thread of its group; of the first: epilogue thread
  if (warp == 0) {
    // ------------------------------------------------ TMA producer
    if (lane == 0) {
      const CUtensorMap* wm = &maps.w[j];
      int s = 0;
      uint32_t ph = 1;
      for (int ks = k0; ks < k1; ++ks) {
        if (ks - k0 >= ns && !mbar_wait(bar(B_EMPTY + s), ph, abort_flag)) break;
        mbar_expect_tx(bar(B_FULL + s), stage_bytes);
        const uint32_t dst = sbase + s * stage_bytes;
        tma_load_2d(dst + x_bytes, wm, bar(B_FULL + s), n0, ks * BK);
        tma_load_2d(dst + x_bytes + W_GROUP, wm, bar(B_FULL + s), n0 + 64, ks * BK);
        tma_load_2d(dst, &maps.x, bar(B_FULL + s), ks * BK, 0);
        ++fills;
        if (++s == ns) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer of x W
    int s = 0;
    uint32_t ph = 0;
    for (int ks = k0; ks < k1; ++ks) {
      if (!(ok = wait_all(bar(B_FULL + s), ph))) break;
      tc_fence_after();
      issue_stage(sbase + s * stage_bytes, tmem, ks == k0, BK / 16);
      umma_commit_elect(bar(B_EMPTY + s));
      if (++s == ns) { s = 0; ph ^= 1u; }
    }
    if (ok) umma_commit_elect(bar(B_ACC));
  } else if (warp == 2 + 4 * ne) {
    // ------------------------------------------------ MMA issuer of the LoRA term
    ok = wait_all(bar(B_LIST), 0);
    if (ok) n_stages = *n_stage_slot;
    int s = 0;
    uint32_t ph = 0;
    for (int i = 0; ok && i < n_stages; ++i) {
      if (!(ok = wait_all(bar(B_EFULL + s), ph))) break;
      tc_fence_after();
      issue_stage(sbase + off_ext + s * stage_bytes, tmem_lora, i == 0, BK / 16);
      umma_commit_elect(bar(B_EEMPTY + s));
      if (++s == ne) { s = 0; ph ^= 1u; }
    }
    if (ok) umma_commit_elect(bar(B_ACC));
  } else {
    uint32_t rpb = 1;
    if (filler == 0) {
      // ------------------------------------------------ list of the LoRA units, in segment order
      int n_units = 0;
      for (int s0 = 0; s0 < a.n_seg; s0 += 128) {
        const int s = s0 + et;
        int lo = 0, hi = 0, rank = 0;
        uint32_t tab = 0, row0 = 0;
        if (s < a.n_seg) {
          lo = max(a.seg_indptr[s], 0);
          hi = min(a.seg_indptr[s + 1], a.n_tokens);
          const int lid = a.lora_ids[s];
          if (lid >= 0 && hi > lo) {
            if ((uint32_t)lid >= a.pv.dir_cap || a.pv.dir[lid].rank <= 0 || a.mat_index[j] >= a.pv.dir[lid].n_mats) {
              atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
            } else {
              const LoraEntry* en = a.pv.dir + lid;
              rank = min(en->rank, a.rmax);
              const LoraMat lm = en->mats[a.mat_index[j]];
              tab = en->table_off + lm.b_tab;
              row0 = lm.b_row0;
              rpb = lm.b_rpb;          // the same for every adapter: they share the projection's shape
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
        if (lane == 31) scan[warp - 2] = incl;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        int at = n_units + incl - cnt;
        for (int w = 0; w < 4; ++w) {
          const int t = scan[w];
          if (w < warp - 2) at += t;
          n_units += t;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        for (int r0 = 0; r0 < rank; r0 += UNIT, ++at)
          if (at < max_units) {
            LoraUnit u;
            u.lo = (uint16_t)lo;
            u.hi = (uint16_t)hi;
            u.r0 = (uint16_t)r0;
            u.nr = (uint16_t)min(UNIT, rank - r0);
            u.tab = tab;
            u.row0 = row0 + r0;
            list[at] = u;
          }
      }
      n_units = min(n_units, max_units);           // (overlapping segments, which the interface rules out, could exceed it)
      const int all_stages = (n_units + 3) / 4;
      if (et < all_stages * 4 - n_units) {
        LoraUnit none = {};
        list[n_units + et] = none;
      }
      {
        const uint32_t m = __reduce_max_sync(0xffffffffu, rpb);
        if (lane == 0) scan[warp - 2] = (int)m;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        for (int w = 0; w < 4; ++w) rpb = max(rpb, (uint32_t)scan[w]);
      }
      // stages are dealt round robin over the cluster
      n_stages = all_stages > crank ? (all_stages - crank + split - 1) / split : 0;
      // the v rows of the ring start at zero
      if (n_stages > 0)
        for (int e = 0; e < ne; ++e)
          for (int c = et; c < npad * 8; c += 128)
            *reinterpret_cast<uint4*>(smem + off_ext + e * stage_bytes + c * 16) = make_uint4(0u, 0u, 0u, 0u);
      fence_async_smem();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (et == 0) {
        *n_stage_slot = n_stages;
        *rpb_slot = (int)rpb;
        mbar_arrive(bar(B_LIST));
      }
    } else {
      ok = mbar_wait(bar(B_LIST), 0, abort_flag);
      if (ok) {
        n_stages = *n_stage_slot;
        rpb = (uint32_t)*rpb_slot;
      }
      ok = group_and(ok, 1 + filler, 128);
      if (!ok) n_stages = 0;
    }
    // ------------------------------------------------ fill the LoRA stages
    // Addresses of the B rows of this group's next stages, looked up side by side ahead of their use, and their 256 bytes asked
    // into L2: under the stream of W a load takes 2 us, and a stage that had to wait for its table entry and then for its rows
    // took 3.5 us (decode step of 48 tokens and 35 adapters of rank 32, d_out 15360).  Issuing a stage's copies takes four
    // warps about 3000 cycles, most of them in the load/store unit's queue, hence three groups.
    unsigned long long* const my_rows = row_ptr + filler * (2 * GROUP * BK);
    // One group per slot of the ring: a group then knows, from the stage it filled before, that the slot's use before last is
    // over, and a parity wait tells the last one from it.
    const int n_mine = n_stages > filler ? (n_stages - filler + ne - 1) / ne : 0;     // stages filler, filler + ne, ..
    auto units_of = [&](int k) { return list + 4 * (crank + (filler + k * ne) * split); };
    auto find_rows = [&](int g) {
#pragma unroll
      for (int i = 0; i < GROUP * BK / 128; ++i) {
        const int c = et + 128 * i, k = g * GROUP + c / BK, r = c % BK;
        unsigned long long at = 0;
        if (k < n_mine) {
          const LoraUnit x = units_of(k)[r / UNIT];
          if (r % UNIT < x.nr) {
            const uint32_t gr = x.row0 + r % UNIT;
            const uint32_t blk = a.pv.tables[x.tab + gr / rpb];
            if (blk >= a.pv.n_blocks) {
              atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_BLOCK);
            } else {
              const unsigned char* p = a.pv.slab + (size_t)blk * a.pv.block_bytes + ((size_t)(gr % rpb) * d_out + n0) * 2;
              at = reinterpret_cast<unsigned long long>(p);
              asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
              if (n0 + 64 < d_out) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 128));
            }
          }
        }
        my_rows[(g & 1) * GROUP * BK + c] = at;
      }
    };
    const int row = et >> 4, ch = et & 15;               // B rows row + 8 i, 16-byte chunk ch of the 128 columns
    const int vrow = et >> 3, vch = et & 7;              // v rows vrow + 16 i, ranks 8 vch .. of the stage's 64
    const bool col_ok = n0 + ch * 8 < d_out;
    auto range_of = [](const LoraUnit* u, int& lo, int& hi) {      // tokens of a stage: segments come in token order
      lo = u[0].lo;
      hi = u[0].hi;
#pragma unroll
      for (int q = 1; q < 4; ++q)
        if (u[q].nr) hi = max(hi, (int)u[q].hi);
    };
    if (n_mine > 0) find_rows(0);
    for (int k = 0; k < n_mine; ++k) {
      if (k > 0) ok = mbar_wait(bar(B_EEMPTY + filler), (uint32_t)((k - 1) & 1), abort_flag);
      ok = group_and(ok, 1 + filler, 128);               // (also makes the addresses visible that were looked up before)
      if (!ok) break;
      const LoraUnit* u = units_of(k);
      const unsigned long long* rp = my_rows + (k % (2 * GROUP)) * BK;
      const uint32_t vb = sbase + off_ext + filler * stage_bytes, bb = vb + x_bytes;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int r = row + 8 * q;
        const unsigned long long at = rp[r];
        cp_async16(bb + (ch >> 3) * W_GROUP + r * 128 + (((ch & 7) ^ (r & 7)) << 4),
                   at ? reinterpret_cast<const unsigned char*>(at) + ch * 16 : a.pv.slab, at && col_ok);
      }
      cp_async_commit();
      if (k == 0) pdl_wait();                            // v is the shrink's output
      {
        const LoraUnit x = u[vch >> 1];
        const int r = x.r0 + 8 * (vch & 1);
        const bool live = 8 * (vch & 1) < x.nr;
        const __nv_bfloat16* src = a.v + ((size_t)j * a.n_tokens) * a.rmax + r;
        // Only the rows of the stage's own tokens are written, and zeros over those of the stage before it in this slot (a
        // decode step: four rows each instead of all).
        int lo, hi;
        range_of(u, lo, hi);
        for (int t = lo + vrow; t < hi; t += 16) {
          const bool mine = live && t >= x.lo && t < x.hi;
          cp_async16(vb + t * 128 + ((vch ^ (t & 7)) << 4), mine ? src + (size_t)t * a.rmax : a.v, mine);
        }
        if (k > 0) {
          int lo0, hi0;
          range_of(units_of(k - 1), lo0, hi0);
          for (int t = lo0 + vrow; t < hi0; t += 16)
            if (t < lo || t >= hi) cp_async16(vb + t * 128 + ((vch ^ (t & 7)) << 4), a.v, false);
        }
      }
      cp_async_commit();
      if (k % GROUP == 0 && k + GROUP < n_mine) find_rows(k / GROUP + 1);
      cp_async_wait<1>();                                // the B rows; v is still on its way
      uint32_t found = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int r = row + 8 * q;
        found |= nonfinite_chunk(ld_shared_v4(bb + (ch >> 3) * W_GROUP + r * 128 + (((ch & 7) ^ (r & 7)) << 4)));
      }
      if (found) *nonfinite_slot = 1;
      cp_async_wait<0>();
      fence_async_smem();
      mbar_arrive(bar(B_EFULL + filler));
    }
    cp_async_wait<0>();
    if (n_mine == 0) pdl_wait();
  }

  // ------------------------------------------------ epilogue: this thread's token row(s)
  const int quarter = warp & 3;
  const int lrow = quarter * 32 + lane;                       // row of the tile = TMEM lane
  const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
  const bool epi = filler == 0;
  const int side = a.kv_side[j];
  uint32_t kv_blk[2] = {0, 0};
  int kv_slot[2] = {-1, -1};
  if (epi) {
    if (a.n_req > 0) clear_v_tails(a, (int)blockIdx.x, (int)gridDim.x, warp - 2, 4);
    if (side >= 0) {                                          // where K / V rows go
      for (int m = 0; m < mt; ++m) {
        const int t = m * 128 + lrow;
        if (t >= a.n_tokens) continue;
        int lo = 0, hi = a.n_req;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (a.req_indptr[mid] <= t) lo = mid; else hi = mid;
        }
        const int pos = a.prefix_lens[lo] + (t - a.req_indptr[lo]);
        const int entry = pos / a.bt, slot = pos - entry * a.bt;
        if (pos < 0 || t < a.req_indptr[lo] || t >= a.req_indptr[lo + 1] || entry >= a.tbl_indptr[lo + 1] - a.tbl_indptr[lo]) {
          atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
          continue;
        }
        const uint32_t b = a.tbl[a.tbl_indptr[lo] + entry];
        if (b >= a.pv.n_blocks) {
          atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_BLOCK);
          continue;
        }
        kv_blk[m] = b;
        kv_slot[m] = slot;
      }
    }
    if (ok) ok = mbar_wait(bar(B_ACC), 0, abort_flag);
    ok = group_and(ok, 1, 128);
    tc_fence_after();
  }
  __syncwarp();
  pdl_launch_dependents();
  if (epi && ok && n_stages > 0 && *nonfinite_slot)
    for (int m = 0; m < mt; ++m) redo_lora_sums(a, list, (uint32_t)*rpb_slot, crank, split, n_stages, j, m * 128 + lrow, n0, tmem_lora + m * BN + lane_addr);
  // columns of the tile that each CTA of the cluster finishes; partial sums as [sender][token][share + 4] floats
  const int share = split > 1 ? (BN / 16 + split - 1) / split * 16 : BN;
  const int pitch = share + 4;
  const int c0 = min(crank * share, BN), c1 = min(c0 + share, BN);
  if (split > 1) {
    cluster_sync();                                           // every CTA of the cluster is done with its rings
    if (tid == 64)
      giveup::tell_cluster(ok, crank, split, [&](int p) { st_cluster_u32(map_cluster_rank(smem_u32(const_cast<int*>(told_slot)), (uint32_t)p), 1u); });
    if (epi && ok) {
      for (int p = 0; p < split; ++p) {
        if (p == crank) continue;
        const uint32_t slot = (uint32_t)(crank < p ? crank : crank - 1);
        const uint32_t dst = map_cluster_rank(sbase + slot * (uint32_t)(npad * pitch) * 4u, (uint32_t)p);
        const int p0 = min(p * share, BN), p1 = min(p0 + share, BN);
        for (int m = 0; m < mt; ++m)
          for (int c = p0; c < p1; c += 16) {
            uint32_t o[16], l[16];
            __syncwarp();
            tmem_ld16(tmem + m * BN + lane_addr + c, o);
            if (n_stages > 0) tmem_ld16(tmem_lora + m * BN + lane_addr + c, l);
            tmem_wait_ld();
            const int t = m * 128 + lrow;
            if (t < a.n_tokens) {
              const uint32_t at = dst + (uint32_t)(t * pitch + c - p0) * 4u;
#pragma unroll
              for (int q = 0; q < 16; q += 4) {
                float4 f = make_float4(__uint_as_float(o[q]), __uint_as_float(o[q + 1]), __uint_as_float(o[q + 2]), __uint_as_float(o[q + 3]));
                if (n_stages > 0) {
                  f.x += __uint_as_float(l[q]); f.y += __uint_as_float(l[q + 1]);
                  f.z += __uint_as_float(l[q + 2]); f.w += __uint_as_float(l[q + 3]);
                }
                st_cluster_f32x4(at + 4 * q, f);
              }
            }
          }
      }
    }
    __syncwarp();
    cluster_sync();
    ok = giveup::may_store(ok, *told_slot);
  }
  if (epi && ok) {
    // The finished rows as bf16 through shared memory (behind the partial sums; pitch an odd number of 16-byte chunks), so that
    // they go out a whole row piece at a time: stored by the thread that owns the row, 16 bytes of 32 rows per instruction,
    // the rows of a decode batch of 128 took up to 18 us.
    const int nch = (c1 - c0) / 8, row_bytes = share * 2 + 16;
    unsigned char* out = smem + (size_t)(split - 1) * npad * pitch * 4;
    for (int m = 0; m < mt; ++m) {
      const int t = m * 128 + lrow;
      for (int c = c0; c < c1; c += 16) {
        uint32_t o[16], l[16];
        __syncwarp();
        tmem_ld16(tmem + m * BN + lane_addr + c, o);
        if (n_stages > 0) tmem_ld16(tmem_lora + m * BN + lane_addr + c, l);
        tmem_wait_ld();
        if (t >= a.n_tokens) continue;
        float f[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) f[q] = __uint_as_float(o[q]) + (n_stages > 0 ? __uint_as_float(l[q]) : 0.f);
        for (int p = 0; p + 1 < split; ++p) {
          const float4* part = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(smem) + (size_t)(p * npad + t) * pitch + (c - c0));
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 v = part[q];
            f[4 * q] += v.x; f[4 * q + 1] += v.y; f[4 * q + 2] += v.z; f[4 * q + 3] += v.w;
          }
        }
        uint4* dst = reinterpret_cast<uint4*>(out + t * row_bytes + (c - c0) * 2);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          dst[h] = make_uint4(pack_bf16(f[8 * h], f[8 * h + 1]), pack_bf16(f[8 * h + 2], f[8 * h + 3]),
                              pack_bf16(f[8 * h + 4], f[8 * h + 5]), pack_bf16(f[8 * h + 6], f[8 * h + 7]));
      }
      if (side >= 0 && t < a.n_tokens) {
        // a column tile is one KV head: [K|V][kv head][slot][128] inside the block
        unsigned long long at = 0;
        if (kv_slot[m] >= 0)
          at = reinterpret_cast<unsigned long long>(a.pv.slab + (size_t)kv_blk[m] * a.pv.block_bytes +
                                                    ((size_t)(side * a.n_kv + n0 / FL_HEAD_DIM) * a.bt + kv_slot[m]) * (FL_HEAD_DIM * 2));
        row_ptr[t] = at;
      }
    }
    static_assert(BN == FL_HEAD_DIM && skinny::MAX_TOKENS * 8 <= ROWS_BYTES, "rows of one head, their addresses where the B rows' were");
    asm volatile("bar.sync 1, 128;" ::: "memory");
    for (int i = et; i < a.n_tokens * nch; i += 128) {
      const int t = i / nch, ch = i - t * nch;
      const uint4 q = *reinterpret_cast<const uint4*>(out + t * row_bytes + ch * 16);
      const int col = n0 + c0 + 8 * ch;
      if (side < 0) {
        if (col < d_out) *reinterpret_cast<uint4*>(a.y[j] + (size_t)t * d_out + col) = q;
      } else if (const unsigned long long at = row_ptr[t]) {
        *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(at) + (c0 + 8 * ch) * 2) = q;
      }
    }
    tc_fence_before();
  }
  // ------------------------------------------------ teardown
  __syncthreads();
  if (*abort_flag) {
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_WAIT_GAVE_UP);
    // copies and MMAs still in flight use this CTA's shared memory and TMEM
    if (warp == 1 || warp == 2 + 4 * ne) umma_commit_elect(bar(B_IDLE));
    if (tid == 0) {
      giveup::drain(fills, ns, [&](int s, uint32_t parity) { return mbar_try(bar(B_FULL + s), parity); });
      giveup::drain(1, 1, [&](int, uint32_t parity) { return mbar_try(bar(B_IDLE), parity); });
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ka.tmem_cols) : "memory");
  }
}

// As many CTAs per column tile as the SMs hold at once (clusters above two do not fill every SM), every one with at least four
// stages of d_in.
int cluster_split(const fl_pool* p, int tiles, int nk) {
  int split = 1;
  for (int s = 2; s <= MAX_SPLIT; ++s)
    if (tiles * s <= (s == 2 ? p->sm_count : p->sm_count * 9 / 10) && nk / s >= 4) split = s;
  return split;
}

// Tiles, split of d_in, rings and shared memory of a call.
void layout(const fl_pool* p, const skinny::Args& a, KArgs* out, uint32_t* smem) {
  KArgs& ka = *out;
  memset(&ka, 0, sizeof(ka));
  ka.s = a;
  ka.npad = (a.n_tokens + 15) / 16 * 16;
  int tiles = 0;
  for (int j = 0; j < a.n_mats; ++j) {
    ka.tile_base[j] = tiles;
    tiles += (a.d_out[j] + BN - 1) / BN;
  }
  for (int j = a.n_mats; j <= skinny::MAX_LIN; ++j) ka.tile_base[j] = tiles;
  ka.tmem_cols = ka.npad > 128 ? 512 : 256;
  const uint32_t fixed = BOOK_BYTES + ROWS_BYTES + ka.npad * UNITS_PER_TOKEN * sizeof(LoraUnit) + 1024;
  const uint32_t stage = W_BYTES + (uint32_t)ka.npad * 128;
  const int nk = (a.d_in + BK - 1) / BK;
  ka.split = cluster_split(p, tiles, nk);
  // The two rings share the memory as a CTA's main stages and LoRA stages (at most; ranks may be lower) share its work: both
  // are bound by the bytes they have in flight.
  const int lora = (a.n_seg * ((a.rmax + UNIT - 1) / UNIT) + 3) / 4;
  const int lora_cta = (lora + ka.split - 1) / ka.split, main_cta = nk / ka.split;
  const int fit = (int)(((ka.npad > 32 || lora_cta >= 8 ? SMEM_MAX : SMEM_LIMIT) - fixed) / stage);
  const int by_work = (fit * lora_cta + (lora_cta + main_cta) / 2) / (lora_cta + main_cta);
  ka.ne = std::max(1, std::min({FILLERS, fit - 4, by_work}));
  ka.ns = std::min(MAX_NS, fit - ka.ne);
  // the partial sums and the finished rows have to fit in the ring that they reuse
  for (; ka.split > 1; --ka.split) {
    const int share = (BN / 16 + ka.split - 1) / ka.split * 16;
    if ((uint32_t)(ka.npad * ((ka.split - 1) * (share + 4) * 4 + share * 2 + 16)) <= ka.ns * stage) break;
  }
  *smem = fixed + (ka.ns + ka.ne) * stage;
}

}  // namespace

namespace skinny {

// Up to 128 tokens always.  Above that a CTA brings 48 KB of x and W per stage for 128 columns where one of the GEMM for long batches
// brings 32 KB for as many, while the GEMM takes a tile's LoRA stages (up to 32 ranks each) one after the other.
//  - More than 16 such stages: here.  q, k, v of 230 tokens, twelve segments of rank 64, here and there: 7B 62 and 64 us; o 33 and 39.
//  - d_in split over at least two CTAs of 16 stages each (o): the GEMM leaves half of the SMs idle.  Here up to 208 tokens; beyond, the sum
//    over the cluster wants 24 stages to be small against.  o of 176 tokens, four segments: 7B 24 and 27 us, 13B 25 and 32, 34B 38 and 50; of
//    256 29 and 28, 29 and 32, 45 and 50.
//  - Otherwise (q, k, v; narrow layers): here for more than eight stages up to 176 tokens.  q, k, v of a decode step of 150 tokens, rank 16, 32
//    segments: 7B 47 and 51 us, 13B 61 and 60, 34B 64 and 68, a layer of 1024 values 26 and 30; 12 segments: 41 and 40, 54 and 51, 61 and
//    60, 23 and 22; one segment of 256 tokens 50 and 40, 66 and 54, 71 and 52, 33 and 20.
// More than 512 ranks over short segments: the two-step way (q, k, v and o of 160 tokens on 13B, 75 adapters of rank 32: 173 us here, 141).
// Over 1284 batches of 130 to 256 tokens the choice is 0.5 % behind the better of the two kernels.
bool serves(const fl_pool* p, const int* d_out, int n_mats, int d_in, int n_tokens, int n_seg, int rank_max) {
  if (n_tokens <= 128) return true;
  if (n_tokens > MAX_TOKENS || (n_seg * rank_max > 8 * 64 && n_tokens <= 16 * n_seg)) return false;
  if (n_seg * rank_max > 16 * 32) return true;
  int tiles = 0;
  for (int j = 0; j < n_mats; ++j) tiles += (d_out[j] + BN - 1) / BN;
  const int nk = (d_in + BK - 1) / BK, split = cluster_split(p, tiles, nk);
  if (split >= 2 && nk / split >= 16) return n_tokens <= 208 || nk / split >= 24;
  return n_seg * rank_max > 8 * 32 && n_tokens <= 176;
}

sgmv::Follower footprint(const fl_pool* p, const Args& a) {
  KArgs ka;
  uint32_t smem;
  layout(p, a, &ka, &smem);
  return {ka.tile_base[a.n_mats] * ka.split, ka.split, smem};
}

int launch(fl_pool* p, const Args& a, const void* x, const void* const* w, cudaStream_t st) {
  KArgs ka;
  uint32_t smem;
  layout(p, a, &ka, &smem);
  const unsigned ctas = (unsigned)(ka.tile_base[a.n_mats] * ka.split);
  Maps maps;
  {
    const uint64_t dims[2] = {(uint64_t)a.d_in, (uint64_t)a.n_tokens};
    const uint64_t strides[1] = {(uint64_t)a.d_in * 2};
    const uint32_t box[2] = {BK, (uint32_t)ka.npad};
    const int rc = tmap::encode_bf16(&maps.x, x, 2, dims, strides, box);
    if (rc != FL_OK) return rc;
  }
  for (int j = 0; j < MAX_LIN; ++j) {
    if (j >= a.n_mats) { maps.w[j] = maps.w[0]; continue; }
    const uint64_t dims[2] = {(uint64_t)a.d_out[j], (uint64_t)a.d_in};
    const uint64_t strides[1] = {(uint64_t)a.d_out[j] * 2};
    const uint32_t box[2] = {64, BK};
    const int rc = tmap::encode_bf16(&maps.w[j], w[j], 2, dims, strides, box);
    if (rc != FL_OK) return rc;
  }
  static bool configured[16] = {};
  if (!configured[p->device & 15]) {
    FL_CUDA(p, cudaFuncSetAttribute(lora_skinny_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
    configured[p->device & 15] = true;
  }
  FL_CUDA(p, launch_pdl_cluster(lora_skinny_kernel, dim3(ctas), dim3((unsigned)ka.split), dim3((unsigned)(96 + 128 * ka.ne)), smem, st, ka, maps));
  FL_CUDA(p, cudaGetLastError());
  return FL_OK;
}

}  // namespace skinny
