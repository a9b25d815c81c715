// Prefill attention, two query tiles per CTA sharing one K/V stream, persistent CTAs (Section 2.1 / 4.2:
// attention over the reused prefix KV plus the new tokens, read in place from pool blocks).
//
// One CTA per SM.  A work unit is 2 x 128 query rows of one (request, KV head): with grouped heads the two
// tiles are two query heads over the same 128 new tokens, otherwise two consecutive 128-token tiles of
// one head.  Both tiles read the same K/V tiles, so every pool page is staged into shared memory once
// for 256 query rows.  CTAs take units from a counter in device memory until none is left; the loads of
// the next unit start while the current one is still in its last tiles and its epilogue.
//   warps 0-3   softmax of tile A (thread = query row = TMEM lane)      warp 8   TMA producer, unit fetch
//   warps 4-7   softmax of tile B                                        warp 9   MMA issuer of the scores, TMEM owner
//                                                                        warps 10, 11   MMA issuers of P V, a tile each
//   K_j / V_j (128 keys = 8 pool pages each, one 4 KiB TMA box per page) -> two rings of 32 KiB slots, 128-byte swizzle;
//   a page lands as [8-key group][64-value half][8 keys][64 values], so a tile's 8-key groups are 2 KiB apart
//   S   = Q_X K_j^T     tcgen05.mma 128x128x16 (x8) into TMEM columns that both tiles use in turn
//   P_X = exp2(S - m) -> bf16 pairs in TMEM columns of tile X's own
//   O_X += P_X V_j      tcgen05.mma with the A operand read from TMEM, V MN-major as stored
// A softmax warp takes its 128 scores into registers at once, so the next scores, the other tile's, go into the same columns while it
// is at its exponentials: TMEM holds one S, two P and two O, and a tile's next scores are there when its softmax comes back for them.
// Until then S_X(j+1) waited for PV_X(j), whose P lay in its columns, and one warp issued everything, which left the tensor pipe idle
// during that warp's barrier tests (see the issuers).  A step of two tiles takes 3040 cycles, a unit's start and end included (34B,
// 4 x 1024 new tokens behind 3072), of which the MMAs need 2048.  What bounds it is the power limit as much as the chain of hand-offs:
// 16 x 1024 new tokens behind 3072, 34B, first launches on a cool chip 1500 -> 1450 us, run after run at 1000 W 1728 -> 1687 us (1540 MHz
// now, 1580 before); 64 prompts of U{128..1024} tokens, half of them cached, 7B 317 -> 307 us.
// P of a step comes in two halves of 64 keys, and PV of the first runs while the softmax is at the last quarter of its
// exponentials.
// O is rescaled only when a row maximum grew by more than 2^8.  Every mbarrier wait is bounded; a wait
// that gives up raises a sticky flag, the CTA drains its copies and frees its TMEM.
#include <cuda.h>
#include <math.h>
#include <string.h>
#include <algorithm>
#include "attention.cuh"
#include "attention_roles.cuh"
#include "giveup.cuh"
#include "mma_utils.cuh"
#include "tc_ptx.cuh"
#include "tmap.cuh"

namespace attn {
namespace {

using namespace tc;

constexpr int T2_THREADS = 384;                        // three warpgroups: softmax A, softmax B, {TMA, MMA x 3}
constexpr int KT2 = 128;                               // keys per tile
constexpr uint32_t HALF_BYTES = 128 * 128;             // [128 rows][64 bf16], swizzled
constexpr uint32_t TILE_BYTES = 2 * HALF_BYTES;        // a Q, K or V tile
constexpr uint32_t PAGE_BYTES = BT * 128 * 2;          // K or V of one head of one block: [2 groups][2 halves][8 tokens][64 bf16]
constexpr uint32_t GROUP_BYTES = PAGE_BYTES / 2;       // stride between 8-key groups of a K/V tile
constexpr uint32_t OFF_Q2 = 0;                         // Q_A, Q_B
constexpr uint32_t OFF_K = 2 * TILE_BYTES;
constexpr uint32_t OFF_V = OFF_K + K_SLOTS * TILE_BYTES;
constexpr uint32_t OFF_BAR2 = OFF_V + V_SLOTS * TILE_BYTES;
constexpr uint32_t T2_SMEM = OFF_BAR2 + 512;           // barriers, TMEM address, abort flag, two unit descriptors
constexpr uint32_t T2_TMEM_COLS = 512;                 // S (128 columns) | P_A | P_B (64 each) | O_A | O_B (128 each)
constexpr uint32_t TM_P = 128, TM_O = 256;
constexpr float RESCALE_LOG2 = 8.f;

enum { C_QFULL = 0, C_QEMPTY = 1, C_KFULL = 2, C_KEMPTY = C_KFULL + K_SLOTS, C_VFULL = C_KEMPTY + K_SLOTS, C_VEMPTY = C_VFULL + V_SLOTS,
       C_SFULL = C_VEMPTY + V_SLOTS, C_SFREE = C_SFULL + 2,
       C_PFULL = C_SFREE + 1, C_PHALF = C_PFULL + 2, C_PVDONE = C_PHALF + 2, C_UFULL = C_PVDONE + 2, C_UEMPTY = C_UFULL + 2, C_IDLE = C_UEMPTY + 2, C_COUNT };
constexpr int UNIT_READERS = 11;                       // three MMA issuers + 8 softmax warps

struct Unit {           // what a CTA works on at one time
  int tok0[2];          // first token row (in the packed q / out tensors) of each tile
  int hq[2];            // query head of each tile
  int rows[2];          // valid query rows (0 = tile unused)
  int lim0[2];          // last visible key of row 0 of each tile
  int n_kt[2];          // K/V tiles each tile takes part in
  int n_kt_max, n_pages, tbl0, h;
  int valid;            // 0: the unit's table is too short for its keys (skipped by every role)
  int index;            // -1 = no more work
};

// Unit u = (plan tile u / heads_per_item, head slot u % heads_per_item), decoded once by the producer and handed
// to the other roles through shared memory.
__device__ __forceinline__ Unit decode_unit(const AttnArgs& a, int u, int heads_per_item) {
  Unit t;
  const int item = u / heads_per_item, hslot = u % heads_per_item;
  const int2 it = a.prefill_list[item];
  const int i = it.x, q0 = it.y;
  const int n_new = a.new_lens[i], prefix = a.prefix_lens[i], ctx = prefix + n_new;
  const int group = a.n_q / a.n_kv;
  if (group % 2 == 0) {
    t.hq[0] = 2 * hslot; t.hq[1] = 2 * hslot + 1;
    t.h = t.hq[0] / group;
    t.tok0[0] = t.tok0[1] = a.req_indptr[i] + q0;
    t.rows[0] = t.rows[1] = min(128, n_new - q0);
    t.lim0[0] = t.lim0[1] = prefix + q0;
  } else {
    t.hq[0] = t.hq[1] = hslot;
    t.h = hslot / group;
    t.tok0[0] = a.req_indptr[i] + q0; t.tok0[1] = t.tok0[0] + 128;
    // a request with an odd number of 128-row tiles has its first tile alone (the plan starts its pairs at token 128)
    const bool lone = q0 == 0 && (((n_new + 127) / 128) & 1);
    t.rows[0] = min(128, n_new - q0); t.rows[1] = lone ? 0 : max(0, min(128, n_new - q0 - 128));
    t.lim0[0] = prefix + q0; t.lim0[1] = prefix + q0 + 128;
  }
#pragma unroll
  for (int x = 0; x < 2; ++x) t.n_kt[x] = t.rows[x] > 0 ? (t.lim0[x] + t.rows[x] + KT2 - 1) / KT2 : 0;
  t.n_kt_max = max(t.n_kt[0], t.n_kt[1]);
  const int kv_end = min(ctx, t.n_kt_max * KT2);
  t.tbl0 = a.tbl_indptr[i];
  t.n_pages = (kv_end + BT - 1) / BT;
  t.valid = t.rows[0] >= 1 && t.n_pages >= 1 && t.n_pages <= a.tbl_indptr[i + 1] - t.tbl0;
  t.index = u;
  return t;
}

__global__ void __launch_bounds__(T2_THREADS, 1)
attn_prefill_tc2_kernel(const AttnArgs a, const __grid_constant__ CUtensorMap kv_map, const __grid_constant__ CUtensorMap q_map,
                        int heads_per_item, int wide_out) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {   // the swizzled operand tiles need 1024-byte alignment
    if (threadIdx.x == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_WAIT_GAVE_UP);
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar0 = sbase + OFF_BAR2;
  auto bar = [&](int k) { return bar0 + 8u * k; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + OFF_BAR2 + 8 * C_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + OFF_BAR2 + 8 * C_COUNT + 4);
  Unit* unit_slot = reinterpret_cast<Unit*>(smem + OFF_BAR2 + 8 * C_COUNT + 8);   // [2]
  static_assert(8 * C_COUNT + 8 + 2 * sizeof(Unit) <= 512, "barrier area too small");

  if (tid == 0) {
    mbar_init(bar(C_QFULL), 1);
    mbar_init(bar(C_QEMPTY), 1);
    for (int s = 0; s < K_SLOTS; ++s) {
      mbar_init(bar(C_KFULL + s), 1);
      mbar_init(bar(C_KEMPTY + s), 1);
    }
    for (int s = 0; s < V_SLOTS; ++s) {
      mbar_init(bar(C_VFULL + s), 1);
      mbar_init(bar(C_VEMPTY + s), 2);      // one arrival per tile
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(bar(C_SFULL + x), 1);
      mbar_init(bar(C_PFULL + x), 4);
      mbar_init(bar(C_PHALF + x), 4);
      mbar_init(bar(C_PVDONE + x), 1);
      mbar_init(bar(C_UFULL + x), 1);
      mbar_init(bar(C_UEMPTY + x), UNIT_READERS);
    }
    mbar_init(bar(C_SFREE), 4);
    mbar_init(bar(C_IDLE), 3);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(T2_TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // everything above touched only this CTA's shared memory and TMEM; the plan (and q, K, V) are the work of the
  // kernels before this one
  pdl_wait();
  pdl_launch_dependents();    // the decode kernel works beside this one, on the SMs whose CTAs have no unit (any more)
  const int n_units = a.hdr->n_prefill * heads_per_item;   // a CTA beyond the last unit finds no work and tears down
  const int n_ctas = min((int)gridDim.x, a.hdr->prefill_ctas);

  // Readers take the k-th unit of this CTA from slot k & 1 (index -1 = no more work) and release the slot.

  int k_fills = 0, v_fills = 0, q_fills = 0;       // ring slots and Q buffers that the producer has armed

  // the softmax warpgroups keep 128 scores per thread in registers: they take the registers the third
  // warpgroup does not need
  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp == 8) {
      // ------------------------------------------------ unit fetch + TMA producer
      // The whole warp runs the loop; lane 0 fetches units and does the waiting, lanes 0-7 each own one of a tile's eight
      // pages (their block-id loads and their TMA issues run side by side).
      RingPos<K_SLOTS> k_pos;
      RingPos<V_SLOTS> v_pos;
      int n_valid = 0;                 // units whose Q tiles were loaded so far
      bool ok = true;
      for (int k = 0; ok; ++k) {
        if (lane == 0) {
          Unit t;
          t.index = -1;
          t.valid = 0;
          if (k < 2 || mbar_wait(bar(C_UEMPTY + (k & 1)), ((k >> 1) - 1) & 1, abort_flag)) {
            const int u = (int)blockIdx.x >= n_ctas ? n_units : k == 0 ? (int)blockIdx.x : n_ctas + atomicAdd(&a.hdr->next_unit, 1);
            if (u < n_units) t = decode_unit(a, u, heads_per_item);
          }
          unit_slot[k & 1] = t;
          mbar_arrive(bar(C_UFULL + (k & 1)));
        }
        __syncwarp();
        const Unit* up = unit_slot + (k & 1);
        if (up->index < 0) break;
        if (!up->valid) {
          if (lane == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
          continue;
        }
        const int n_kt_max = up->n_kt_max, n_pages = up->n_pages, tbl0 = up->tbl0, h = up->h;
        const int rows_b = up->rows[1];
        // Q buffers are free once the previous unit's last S MMA has completed
        if (lane == 0) {
          if (n_valid > 0) ok = mbar_wait(bar(C_QEMPTY), (n_valid - 1) & 1, abort_flag);
          if (ok) {
            mbar_expect_tx(bar(C_QFULL), rows_b > 0 ? 2 * TILE_BYTES : TILE_BYTES);
            ++q_fills;
          }
        }
        ++n_valid;
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        if (!ok) break;
        if (lane < 4 && (lane < 2 || rows_b > 0)) {          // lane = 2 * tile + half
          const int x = lane >> 1, half = lane & 1;
          tma_load_3d(sbase + OFF_Q2 + x * TILE_BYTES + half * HALF_BYTES, &q_map, bar(C_QFULL), 64 * half, up->hq[x], up->tok0[x]);
        }
        // this lane's page of the tile (pages behind the last needed key are masked anyway: re-read the last
        // valid page); K_j and V_j come from the same blocks
        // lane = page: eight lanes issue one 4 KiB box each
        uint32_t blk = 0;
        auto fill = [&](int side, uint32_t slot, uint32_t full, uint32_t empty, uint32_t parity, int& fills) {
          if (lane == 0) {
            ok = mbar_wait(empty, parity, abort_flag);
            if (ok) {
              mbar_expect_tx(full, TILE_BYTES);
              ++fills;
            }
          }
          ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;     // the transaction count is armed before any copy is issued
          if (ok && lane < KT2 / BT) tma_load_5d(slot + lane * PAGE_BYTES, &kv_map, full, 0, 0, 0, 2 * (side * a.n_kv + h), (int)blk);
          return ok;
        };
        load_tiles(n_kt_max, k_pos, v_pos,
                   [&](int j) {
                     if (lane < KT2 / BT) {
                       blk = a.tbl[tbl0 + min(j * (KT2 / BT) + lane, n_pages - 1)];
                       if (blk >= a.pv.n_blocks) {
                         atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_BLOCK);
                         blk = 0;
                       }
                     }
                   },
                   [&](RingPos<K_SLOTS> p) { return fill(0, sbase + OFF_K + p.s * TILE_BYTES, bar(C_KFULL + p.s), bar(C_KEMPTY + p.s), p.ph ^ 1u, k_fills); },
                   [&](RingPos<V_SLOTS> p) { return fill(1, sbase + OFF_V + p.s * TILE_BYTES, bar(C_VFULL + p.s), bar(C_VEMPTY + p.s), p.ph ^ 1u, v_fills); });
      }
    } else {
      // ------------------------------------------------ MMA issuers: warp 9 the scores of both tiles, warps 10 and 11 P V of one each
      // The tensor pipe's queue is an instruction or two deep, and a barrier test takes an issuer 100 to 250 cycles even where the
      // phase is long over, so with one warp for everything the pipe stood still for a third of a step while that warp looked at its
      // seven barriers.  Nothing orders the three warps but the barriers.  Their loops are kept lean: the whole warp runs converged and
      // an elected lane issues a tile's eight MMAs as one block, descriptors are a fixed high word and a low word that steps by
      // constants, ring slot and phase are running counters, and a barrier is tested once before the bounded wait loop is entered.
      constexpr uint32_t IDESC = instr_desc(128, false);        // S: both operands K-major
      constexpr uint32_t IDESC_PV = instr_desc(D, true);        // O: V is MN-major
      constexpr uint32_t HI_Q = desc_hi(1024), HI_KV = desc_hi(GROUP_BYTES);
      auto wait_all = [&](uint32_t b, uint32_t parity) {
        if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;       // the common case: one test
        return __all_sync(0xffffffffu, mbar_wait(b, parity, abort_flag)) != 0;
      };
      RingPos<K_SLOTS> k_pos;          // of warp 9
      RingPos<V_SLOTS> v_pos;          // of warps 10 and 11
      const int x = warp - 10;         // the tile of warps 10 and 11
      uint32_t ph_q = 0;               // parity of the next unit's Q (C_QFULL)
      uint32_t ph_s = 1;               // parity of the score tile before (C_SFREE); true at once before the first one
      uint32_t ph_p = 0;               // parity of the next P tile (C_PFULL)
      bool ok = true;
      for (int k = 0; ok; ++k) {
        if (!wait_all(bar(C_UFULL + (k & 1)), (k >> 1) & 1)) break;
        const int u_index = unit_slot[k & 1].index, u_valid = unit_slot[k & 1].valid;
        const int n_kt = unit_slot[k & 1].n_kt_max, nA = unit_slot[k & 1].n_kt[0], nB = unit_slot[k & 1].n_kt[1];
        __syncwarp();
        if (lane == 0 && u_index >= 0) mbar_arrive(bar(C_UEMPTY + (k & 1)));
        if (u_index < 0) break;
        if (!u_valid) continue;
        if (warp == 9) {
          ok = wait_all(bar(C_QFULL), ph_q);
          ph_q ^= 1u;
          if (ok)
            ok = issue_scores(n_kt, nA, nB, k_pos, ph_s,
                              [&](RingPos<K_SLOTS> p) { return wait_all(bar(C_KFULL + p.s), p.ph); },
                              [&](uint32_t ph) { return wait_all(bar(C_SFREE), ph); },
                              [&](int t, RingPos<K_SLOTS> p) {
                                tc_fence_after();
                                umma_s_tile_elect(tmem, desc_lo(sbase + OFF_Q2 + t * TILE_BYTES, 16), desc_lo(sbase + OFF_K, 16) + (uint32_t)p.s * (TILE_BYTES >> 4),
                                                  HI_Q, HI_KV, IDESC, bar(C_SFULL + t));
                              },
                              [&](RingPos<K_SLOTS> p) { umma_commit_elect(bar(C_KEMPTY + p.s)); },
                              [&] { umma_commit_elect(bar(C_QEMPTY)); });
        } else {
          ok = issue_pv(n_kt, x == 0 ? nA : nB, v_pos, ph_p,
                        [&](RingPos<V_SLOTS> p) { return wait_all(bar(C_VFULL + p.s), p.ph); },
                        [&](int half, uint32_t ph) { return wait_all(bar((half == 0 ? C_PHALF : C_PFULL) + x), ph); },
                        [&](int half, RingPos<V_SLOTS> p, bool first) {
                          tc_fence_after();
                          umma_pv_half_elect(tmem + TM_O + x * 128, tmem + TM_P + x * 64 + 32 * half,
                                             desc_lo(sbase + OFF_V, 1024) + (uint32_t)p.s * (TILE_BYTES >> 4) + half * (TILE_BYTES >> 5), HI_KV, IDESC_PV,
                                             first && half == 0 ? 0u : 1u);
                        },
                        [&] { umma_commit_elect(bar(C_PVDONE + x)); },
                        [&](RingPos<V_SLOTS> p) { umma_commit_elect(bar(C_VEMPTY + p.s)); });
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    // ------------------------------------------------ softmax of tile x: thread = query row = TMEM lane
    const int x = warp >> 2, row = tid & 127;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t p_addr = lane_addr + TM_P + x * 64, o_addr = lane_addr + TM_O + x * 128;
    const float sl2 = a.scale_log2;
    int steps = 0;      // S tiles of this tile taken so far (phase of C_SFULL)
    auto vote = [](bool v) { return __all_sync(0xffffffffu, v) != 0; };
    auto wait = [&](int k, int parity) { return seen_by_all([&] { return mbar_wait(bar(k), (uint32_t)parity, abort_flag); }, vote, tc_fence_after); };
    for (int k = 0;; ++k) {
      // this tile's few fields straight from the published descriptor
      if (!vote(mbar_wait(bar(C_UFULL + (k & 1)), (k >> 1) & 1, abort_flag))) break;
      const Unit* up = unit_slot + (k & 1);
      const int u_index = up->index, u_valid = up->valid;
      const int rows = up->rows[x], nk = up->n_kt[x], lim0 = up->lim0[x], out_tok0 = up->tok0[x], out_hq = up->hq[x];
      __syncwarp();
      if (lane == 0 && u_index >= 0) mbar_arrive(bar(C_UEMPTY + (k & 1)));
      if (u_index < 0) break;
      if (!u_valid || nk == 0) continue;
      const int lim = row < rows ? lim0 + row : -1;
      float m_used = 0.f, m_run = -INFINITY, l = 0.f;
      bool ok = true;
      for (int j = 0; j < nk; ++j) {
        ok = wait(C_SFULL + x, steps & 1);
        if (!ok) break;
        uint32_t s[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(lane_addr + 32 * c, s[c]);
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(C_SFREE));
        const int u0 = j * KT2;
        if (u0 + KT2 - 1 > lim) {     // a tile that reaches past this row's last visible key
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (u0 + 32 * c + e > lim) s[c][e] = 0xff800000u;   // -inf
        }
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int e = 0; e < 32; e += 2)
            mx[(e >> 1) & 3] = max3(mx[(e >> 1) & 3], __uint_as_float(s[c][e]), __uint_as_float(s[c][e + 1]));
        m_run = fmaxf(m_run, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])));
        bool rescale = false;
        float alpha = 1.f;
        if (j == 0) {
          m_used = m_run == -INFINITY ? 0.f : m_run;
        } else if ((m_run - m_used) * sl2 > RESCALE_LOG2) {
          rescale = true;
          alpha = ex2_approx((m_used - m_run) * sl2);
          m_used = m_run;
        }
        // P_X and O_X may be touched once PV_X(j-1) is complete
        bool pv_done = j == 0;
        if (__any_sync(0xffffffffu, rescale)) {
          ok = wait(C_PVDONE + x, (steps - 1) & 1);
          if (!ok) break;
          pv_done = true;
#pragma unroll
          for (int cb = 0; cb < D; cb += 32) {
            uint32_t o[32];
            tmem_ld32(o_addr + cb, o);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
            tmem_st32(o_addr + cb, o);
          }
          l *= alpha;
        }
        // (as a rule it is by the time the first P is there: the answer of a test ahead of the exponentials costs nothing, one behind them 220 cycles)
        if (!pv_done) pv_done = seen_by_all([&] { return mbar_test(bar(C_PVDONE + x), (steps - 1) & 1); }, vote, tc_fence_after);
        const float2 sc2 = make_float2(sl2, sl2);
        const float nm = -m_used * sl2;
        const float2 nm2 = make_float2(nm, nm);
        float2 sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int c = 0; c < 4; ++c) {      // 32 keys -> 16 bf16 pairs -> TMEM columns 16c .. 16c+15 of this tile
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float2 arg = __ffma2_rn(make_float2(__uint_as_float(s[c][2 * e]), __uint_as_float(s[c][2 * e + 1])), sc2, nm2);
            const float2 p = make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
            sum[e & 1] = __fadd2_rn(sum[e & 1], p);
            pk[e] = pack_bf16(p.x, p.y);
          }
          if (c == 0 && !pv_done) ok = wait(C_PVDONE + x, (steps - 1) & 1);
          if (c == 2) {                    // the stores of the first 64 keys have long landed
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(C_PHALF + x));
          }
          tmem_st16(p_addr + 16 * c, pk);
        }
        if (!ok) break;
        ++steps;
        l += (sum[0].x + sum[0].y) + (sum[1].x + sum[1].y);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(C_PFULL + x));
      }
      // ---- epilogue: O / l -> bf16, each thread stores its own row (8 x 32 bytes, contiguous)
      if (ok) ok = wait(C_PVDONE + x, (steps - 1) & 1);
      if (!ok) break;
      const float inv = l > 0.f ? 1.f / l : 0.f;
      uint4* orow = reinterpret_cast<uint4*>(a.out + ((size_t)(out_tok0 + row) * a.n_q + out_hq) * D);
#pragma unroll
      for (int cb = 0; cb < D; cb += 32) {
        uint32_t o[32];
        tmem_ld32(o_addr + cb, o);
        tmem_wait_ld();
        if (row < rows) {
          uint32_t pk[16];
#pragma unroll
          for (int c = 0; c < 16; ++c) pk[c] = pack_bf16(__uint_as_float(o[2 * c]) * inv, __uint_as_float(o[2 * c + 1]) * inv);
          if (wide_out) {                              // 32 bytes per lane: half as many store instructions per row
            st_global_v8(orow + (cb >> 3), pk);
            st_global_v8(orow + (cb >> 3) + 2, pk + 8);
          } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) orow[(cb >> 3) + c] = make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
          }
        }
      }
      tc_fence_before();
    }
  }
  // ------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_WAIT_GAVE_UP);
    // copies and MMAs still in flight use this CTA's shared memory and TMEM
    if (warp >= 9) umma_commit_elect(bar(C_IDLE));
    if (warp == 8 && lane == 0) {
      giveup::drain(k_fills, K_SLOTS, [&](int s, uint32_t parity) { return mbar_try(bar(C_KFULL + s), parity); });
      giveup::drain(v_fills, V_SLOTS, [&](int s, uint32_t parity) { return mbar_try(bar(C_VFULL + s), parity); });
      giveup::drain(q_fills, 1, [&](int, uint32_t parity) { return mbar_try(bar(C_QFULL), parity); });
      giveup::drain(1, 1, [&](int, uint32_t parity) { return mbar_try(bar(C_IDLE), parity); });
    }
    __syncthreads();
  }
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T2_TMEM_COLS) : "memory");
  }
}

}  // namespace

int launch_prefill_tc2(fl_pool* p, const AttnArgs& a, int n_tokens, int max_items, cudaStream_t st) {
  const CUtensorMap* kv = nullptr;
  alignas(64) CUtensorMap qmap;
  int rc = tmap::kv_pages(p, a.n_kv, &kv);
  if (rc != FL_OK) return rc;
  {   // q as [token][head][128]: box = 64 elements x 128 tokens of one head
    const uint64_t dims[3] = {(uint64_t)D, (uint64_t)a.n_q, (uint64_t)n_tokens};
    const uint64_t strides[2] = {(uint64_t)D * 2, (uint64_t)a.n_q * D * 2};
    const uint32_t box[3] = {64, 1, 128};
    rc = tmap::encode_bf16(&qmap, a.q, 3, dims, strides, box);
    if (rc != FL_OK) return rc;
  }
  static bool configured[16] = {};
  if (!configured[p->device & 15]) {
    FL_CUDA(p, cudaFuncSetAttribute(attn_prefill_tc2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T2_SMEM));
    configured[p->device & 15] = true;
  }
  const int heads_per_item = tc2_heads_per_item(a.n_q, a.n_kv);
  // one CTA per SM (shared memory and TMEM allow no more); a CTA beyond the plan's unit count finds no work and tears down
  const long long units = (long long)max_items * heads_per_item;
  const unsigned grid = (unsigned)std::min<long long>(units, p->sm_count);
  if (grid == 0) return FL_OK;
  FL_CUDA(p, launch_pdl(attn_prefill_tc2_kernel, dim3(grid), dim3(T2_THREADS), T2_SMEM, st, a, *kv, qmap, heads_per_item,
                     (reinterpret_cast<uintptr_t>(a.out) & 31) == 0 ? 1 : 0));   // 32-byte stores where the output allows them
  FL_CUDA(p, cudaGetLastError());
  return FL_OK;
}

}  // namespace attn
