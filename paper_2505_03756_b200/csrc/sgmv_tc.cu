// The shrink v = x A_i of the segmented LoRA projection (Eq. 1, Eq. 2; Section 2.1) for long segments, on the
// 5th-generation tensor cores.
//
// A CTA takes a tile of 128 tokens of one segment and a slice of d_in:
//   warp 0       TMA producer: x tile [128 tokens x 64] per stage (K-major, 128-byte swizzle)
//   warp 1       MMA issuer: D[128 x (projections * RMAX)] += x tile * adapter rows^T, tcgen05.mma 128 x N x 16
//   warps 2-9    adapter rows (row p of A is d_in contiguous values in a pool block, found through the adapter's block
//                table) by 16-byte cp.async into the stage, in the operand's swizzled layout; two groups of four warps take the stages
//                in turn, and the copies themselves arrive on the stage's barrier when they have landed
//   warps 10-13  epilogue: TMEM -> v in its final form, scaled and rounded to bf16, [projection][token][RMAX], rows of the segment only
// Two ways to fill the SMs.  With one slice CTAs stay and go through the tiles, the accumulator is double buffered in TMEM and a tile's
// epilogue overlaps the next one's stages.  With more (SLICED) the slices of a tile are the CTAs of a cluster: each leaves its sums in its
// own shared memory, and all threads of a CTA read a share of the columns from all of them and add in the slices' order.  (Sent to the CTA
// that adds them, by the thread that owns a row, 16 bytes of 32 rows at a time, the sums of three projections at rank 64 took 11 us of 24.)
// Every mbarrier wait is bounded; a wait that gives up raises a sticky flag and the CTA tears down (its cluster told, its copies
// drained, its TMEM freed).  No multicast.
#include <cuda.h>
#include <algorithm>
#include "giveup.cuh"
#include "mma_utils.cuh"
#include "pool.cuh"
#include "sgmv.cuh"
#include "tc_ptx.cuh"
#include "tmap.cuh"

namespace {

using namespace tc;

constexpr int COPY_GROUPS = 2;
constexpr int ST_THREADS = 64 + 128 * COPY_GROUPS + 128;
constexpr int TM = 128, BK = 64;
constexpr uint32_t X_BYTES = TM * BK * 2;

template <int N>
struct Cfg {
  static constexpr uint32_t B_BYTES = N * 128;
  static constexpr uint32_t STAGE = X_BYTES + ((B_BYTES + 1023) / 1024) * 1024;
  static constexpr int NS = (220 * 1024) / STAGE < 8 ? (220 * 1024) / STAGE : 8;      // ring slots: what fits, at most 8
  static constexpr uint32_t OFF_BAR = NS * STAGE;
  static constexpr uint32_t SMEM = OFF_BAR + 256 + 1024;
  static constexpr uint32_t TMEM_COLS = 2 * N <= 32 ? 32 : 2 * N <= 64 ? 64 : 2 * N <= 128 ? 128 : 2 * N <= 256 ? 256 : 512;
  static_assert(2 * N <= 512, "two accumulators must fit in TMEM");
  static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Columns of a tile that each of the `ks` CTAs of a cluster finishes; row pitch of a CTA's sums in shared memory, in floats.
__host__ __device__ constexpr int share_of(int n, int ks) { return (n / 16 + ks - 1) / ks * 16; }
__host__ __device__ constexpr int sum_pitch(int n) { return n + 4; }

struct Unit {
  int seg, tok0, tok1, lid, kb, n_it, split;
  bool ok;
};

// Unit u -> token tile and slice of d_in; the whole warp takes part (the tile search is a warp scan).
__device__ __forceinline__ Unit decode_unit(const sgmv::TcShrinkArgs& a, int u) {
  Unit t;
  const int tile = u / a.ksplit;
  t.split = u - tile * a.ksplit;
  t.ok = sgmv::find_tile<TM>(a.seg_indptr, a.lora_ids, a.n_seg, tile, t.seg, t.tok0, t.tok1);
  t.lid = -1;
  t.kb = t.n_it = 0;
  if (!t.ok) return t;
  t.lid = a.lora_ids[t.seg];
  bool good = t.lid >= 0 && (uint32_t)t.lid < a.pv.dir_cap && a.pv.dir[t.lid].rank > 0;
  for (int j = 0; good && j < a.n_mats; ++j) good = a.mat_index[j] < a.pv.dir[t.lid].n_mats;
  if (!good) {
    if ((threadIdx.x & 31) == 0 && t.lid >= 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
    t.ok = false;
    return t;
  }
  const int kchunk = ((a.d_in + a.ksplit * BK - 1) / (a.ksplit * BK)) * BK;
  t.kb = t.split * kchunk;
  const int ke = min(a.d_in, t.kb + kchunk);
  t.n_it = ke > t.kb ? (ke - t.kb + BK - 1) / BK : 0;
  return t;
}

__device__ __forceinline__ uint4 pack_scaled(const float* f, float scale) {
  return make_uint4(pack_bf16(f[0] * scale, f[1] * scale), pack_bf16(f[2] * scale, f[3] * scale), pack_bf16(f[4] * scale, f[5] * scale),
                    pack_bf16(f[6] * scale, f[7] * scale));
}

template <int RMAX, int NM, bool SLICED>
__global__ void __launch_bounds__(ST_THREADS, 1) sgmv_shrink_tc_kernel(const __grid_constant__ sgmv::TcShrinkArgs a, const __grid_constant__ CUtensorMap xmap,
                                                                       int n_units) {
  constexpr int N = RMAX * NM;
  using C = Cfg<N>;
  constexpr int NS = C::NS;
  static_assert(TM * sum_pitch(N) * 4 <= NS * C::STAGE, "a slice's sums must fit in the ring that they reuse");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  enum { B_FULL = 0, B_EMPTY = NS, B_ACC_FULL = 2 * NS, B_ACC_EMPTY = 2 * NS + 2, B_IDLE = 2 * NS + 4, B_COUNT };
  const uint32_t bar0 = sbase + C::OFF_BAR;
  auto bar = [&](int k) { return bar0 + 8u * k; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + C::OFF_BAR + 8 * B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 8 * B_COUNT + 4);
  volatile int* fills_slot = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 8 * B_COUNT + 8);
  volatile int* missing_slot = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 8 * B_COUNT + 12);      // this CTA has no part of the sum
  static_assert(8 * B_COUNT + 16 <= 256, "bookkeeping area too small");

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(bar(B_FULL + s), 1 + 128);     // the TMA producer's arrive (with the byte count) + the 128 threads of a copy group
      mbar_init(bar(B_EMPTY + s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar(B_ACC_FULL + b), 1);
      mbar_init(bar(B_ACC_EMPTY + b), 4);
    }
    mbar_init(bar(B_IDLE), 1);
    *abort_flag = 0;
    *missing_slot = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(C::TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();                 // x may come from the kernel right before this one
  pdl_launch_dependents();    // the kernel that consumes v may set itself up while this grid runs

  // (a sliced tile is the CTA's only one, and every warp needs it again for the sum)
  const Unit only = SLICED ? decode_unit(a, blockIdx.x) : Unit{};
  auto unit = [&](int u) { return SLICED ? only : decode_unit(a, u); };
  int fills = 0;       // x copies that the producer has issued
  int owed = 0;        // first stage that a copy thread has not signalled yet, of those of its group
  bool ok = true;
  if (warp == 0) {
    // ------------------------------------------------ TMA producer (lane 0 issues; the warp decodes units together)
    int s = 0;
    uint32_t ph = 1;
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
      const Unit t = unit(u);
      if (!t.ok) continue;
      if (lane == 0) {
        for (int it = 0; it < t.n_it; ++it) {
          ok = mbar_wait(bar(B_EMPTY + s), ph, abort_flag);
          if (!ok) break;
          mbar_expect_tx(bar(B_FULL + s), X_BYTES);
          tma_load_2d(sbase + s * C::STAGE, &xmap, bar(B_FULL + s), t.kb + it * BK, t.tok0);
          ++fills;
          if (++s == NS) { s = 0; ph ^= 1u; }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer: the whole warp runs converged, an elected lane issues
    constexpr uint32_t IDESC = instr_desc(N, false);     // both operands K-major
    constexpr uint32_t HI = desc_hi(1024);
    auto wait_all = [&](uint32_t b, uint32_t parity) {
      if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;       // the common case: one test
      return __all_sync(0xffffffffu, mbar_wait(b, parity, abort_flag)) != 0;
    };
    int s = 0, k = 0;         // k: units with work so far
    uint32_t ph = 0;
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
      const Unit t = unit(u);
      if (!t.ok || t.n_it == 0) continue;
      const int buf = k & 1;
      if (k >= 2) ok = wait_all(bar(B_ACC_EMPTY + buf), (uint32_t)(((k >> 1) - 1) & 1));
      tc_fence_after();
      for (int it = 0; ok && it < t.n_it; ++it) {
        if (!(ok = wait_all(bar(B_FULL + s), ph))) break;
        fence_async_smem();            // the adapter rows were written by the generic proxy, the tensor core reads through the async one
        tc_fence_after();
        const uint32_t a_lo = desc_lo(sbase + s * C::STAGE, 16), b_lo = desc_lo(sbase + s * C::STAGE + X_BYTES, 16);
#pragma unroll
        for (int ks = 0; ks < BK / 16; ++ks)
          umma_ss_elect(tmem + buf * N, a_lo + 2 * ks, HI, b_lo + 2 * ks, HI, IDESC, (it > 0 || ks > 0) ? 1u : 0u);
        umma_commit_elect(bar(B_EMPTY + s));
        if (++s == NS) { s = 0; ph ^= 1u; }
      }
      if (ok) umma_commit_elect(bar(B_ACC_FULL + buf));
      ++k;
    }
  } else if (warp < 2 + 4 * COPY_GROUPS) {
    // ------------------------------------------------ adapter rows: row n = projection * RMAX + rank row, 8 chunks of 16 bytes
    const int ct = (tid - 64) & 127, group = (warp - 2) >> 2;
    constexpr int RPT = N / 16;                   // rows per thread: n = ct / 8 + 16 i
    const int cc = ct & 7;
    int f = 0, s = 0;                             // stages of this CTA so far
    uint32_t ph = 1;
    owed = group;
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
      const Unit t = unit(u);
      if (!t.ok) continue;
      const LoraEntry* e = a.pv.dir + t.lid;
      const int rank = min(e->rank, RMAX);
      if (e->rank > RMAX && ct == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_LORA);
      const uint32_t table_off = e->table_off;
      const unsigned char* rowp[RPT];
      bool rok[RPT];
      sgmv::lora_rows<RPT>(a.pv, [&](int i, uint32_t& entry, uint32_t& off) {
        const int n = (ct >> 3) + 16 * i;
        const int m = n / RMAX, r = n % RMAX;
        if (m >= a.n_mats || r >= rank) return false;
        const LoraMat& lm = e->mats[a.mat_index[m]];
        sgmv::lora_row_at(table_off, lm.a_tab, lm.a_row0, lm.a_rpb, a.d_in, r, entry, off);
        return true;
      }, rowp, rok);
      const int ke = min(a.d_in, t.kb + ((a.d_in + a.ksplit * BK - 1) / (a.ksplit * BK)) * BK);
      for (int it = 0; it < t.n_it; ++it, ++f) {
        if ((f & (COPY_GROUPS - 1)) == group) {
          ok = mbar_wait(bar(B_EMPTY + s), ph, abort_flag);
          if (!ok) break;
          const int kk = t.kb + it * BK + cc * 8;
          const uint32_t bs = sbase + s * C::STAGE + X_BYTES;
#pragma unroll
          for (int i = 0; i < RPT; ++i) {
            const int n = (ct >> 3) + 16 * i;
            cp_async16(bs + n * 128 + ((cc ^ (n & 7)) << 4), rowp[i] + (size_t)kk * 2, rok[i] && kk < ke);
          }
          cp_async_arrive(bar(B_FULL + s));       // when they have landed
          owed = f + COPY_GROUPS;
        }
        if (++s == NS) { s = 0; ph ^= 1u; }
      }
    }
    cp_async_commit();
    cp_async_wait<0>();
  } else {
    // ------------------------------------------------ epilogue: thread = token row = TMEM lane
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    int k = 0;
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
      const Unit t = unit(u);
      if (!t.ok) continue;
      const int tok = t.tok0 + row;
      const bool mine = tok < t.tok1;
      const int buf = k & 1;
      ok = group_and(mbar_wait(bar(B_ACC_FULL + buf), (uint32_t)((k >> 1) & 1), abort_flag), 1, 128);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int c0 = 0; c0 < N; c0 += 16) {
        uint32_t o[16];
        __syncwarp();
        tmem_ld16(lane_addr + buf * N + c0, o);
        tmem_wait_ld();
        const int j = c0 / RMAX, col = c0 % RMAX;
        if constexpr (SLICED) {        // (behind the last MMA: nobody reads the ring any more)
#pragma unroll
          for (int q = 0; q < 16; q += 4)
            st_shared_v4(sbase + (uint32_t)(row * sum_pitch(N) + c0 + q) * 4u, make_uint4(o[q], o[q + 1], o[q + 2], o[q + 3]));
        } else if (mine && j < a.n_mats) {
          uint4* dst = reinterpret_cast<uint4*>(a.v16 + ((size_t)j * a.n_tokens + tok) * RMAX + col);
          const float* of = reinterpret_cast<const float*>(o);
          dst[0] = pack_scaled(of, a.scale);
          dst[1] = pack_scaled(of + 8, a.scale);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_ACC_EMPTY + buf));
      ++k;
    }
    if (SLICED && !ok && tid == ST_THREADS - 1) *missing_slot = 1;
  }
  __syncwarp();
  if (SLICED && only.ok) {       // (the CTAs of a cluster have a tile, or none, together)
    const int ks = a.ksplit, rank = (int)cluster_ctarank();
    cluster_sync();          // every slice's sums are there
    const int told = lane < ks ? (int)ld_cluster_u32(map_cluster_rank(smem_u32(const_cast<int*>(missing_slot)), (uint32_t)lane)) : 0;
    if (giveup::may_store(true, __any_sync(0xffffffffu, told != 0) ? 1 : 0)) {
      const int share = share_of(N, ks), c0 = min(rank * share, N), quads = (min(c0 + share, N) - c0) / 4;
      const int rows = only.tok1 - only.tok0;
      for (int i = tid; i < rows * quads; i += ST_THREADS) {
        const int row = i / quads, c = c0 + (i - row * quads) * 4;
        const uint32_t at = sbase + (uint32_t)(row * sum_pitch(N) + c) * 4u;
        float4 v[sgmv::TC_MAX_SLICES];
#pragma unroll
        for (int p = 0; p < sgmv::TC_MAX_SLICES; ++p)
          if (p < ks) v[p] = ld_cluster_f32x4(map_cluster_rank(at, (uint32_t)p));
        float4 f = v[0];
#pragma unroll
        for (int p = 1; p < sgmv::TC_MAX_SLICES; ++p)
          if (p < ks) { f.x += v[p].x; f.y += v[p].y; f.z += v[p].z; f.w += v[p].w; }
        const int j = c / RMAX, col = c % RMAX;
        if (j < a.n_mats)
          *reinterpret_cast<uint2*>(a.v16 + ((size_t)j * a.n_tokens + only.tok0 + row) * RMAX + col) =
              make_uint2(pack_bf16(f.x * a.scale, f.y * a.scale), pack_bf16(f.z * a.scale, f.w * a.scale));
      }
    }
    __syncwarp();
    cluster_sync();          // nobody leaves while its sums are still being read
  }
  // ------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_WAIT_GAVE_UP);
    // x copies and MMAs still in flight use this CTA's shared memory and TMEM (the adapter-row copies were waited for by their own
    // threads above).  A stage's phase ends with its x copy only if its copy threads signal it too; each owes at most the last
    // phase of a slot, since the one before it was over when the producer armed it.
    if (tid == 0) *fills_slot = fills;
    __syncthreads();
    if (warp >= 2 && warp < 2 + 4 * COPY_GROUPS)
      for (; owed < *fills_slot; owed += COPY_GROUPS) mbar_arrive(bar(B_FULL + owed % NS));
    if (warp == 1) umma_commit_elect(bar(B_IDLE));
    if (tid == 0) {
      giveup::drain(fills, NS, [&](int s, uint32_t parity) { return mbar_try(bar(B_FULL + s), parity); });
      giveup::drain(1, 1, [&](int, uint32_t parity) { return mbar_try(bar(B_IDLE), parity); });
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS) : "memory");
  }
}

template <int RMAX, int NM>
int launch(fl_pool* p, const sgmv::TcShrinkArgs& a, const CUtensorMap& xmap, int n_units, cudaStream_t st) {
  using C = Cfg<RMAX * NM>;
  static bool configured[16] = {};
  if (!configured[p->device & 15]) {
    FL_CUDA(p, cudaFuncSetAttribute(sgmv_shrink_tc_kernel<RMAX, NM, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    FL_CUDA(p, cudaFuncSetAttribute(sgmv_shrink_tc_kernel<RMAX, NM, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    configured[p->device & 15] = true;
  }
  if (a.ksplit > 1)
    FL_CUDA(p, launch_pdl_cluster(sgmv_shrink_tc_kernel<RMAX, NM, true>, dim3((unsigned)n_units), dim3((unsigned)a.ksplit), dim3(ST_THREADS), C::SMEM, st, a, xmap, n_units));
  else
    FL_CUDA(p, launch_pdl(sgmv_shrink_tc_kernel<RMAX, NM, false>, dim3((unsigned)std::min(n_units, p->sm_count)), dim3(ST_THREADS), C::SMEM, st, a, xmap, n_units));
  FL_CUDA(p, cudaGetLastError());
  return FL_OK;
}

}  // namespace

namespace sgmv {

int tc_slices(const fl_pool* p, int n_seg, int n_tokens, int d_in, int rmax, int n_mats) {
  // Rounds of tiles over the SMs times what a tile's slice takes, in us beside what every tile does: look-ups, ramp and end, where slices are
  // added their barriers and the sums, by rows, columns and CTAs (clusters of eight get into each other's way as well), and per stage the fill
  // of x and of the adapter rows at 60 bytes per clock.
  // Clusters of four find a place on the GPU's groups of SMs 33 times, clusters of eight 15 times (as the occupancy query says for this shared
  // memory); other sizes leave more SMs empty.  Shrink and expand with two, four and eight slices, 7B, 512 tokens: one segment of rank 64, q, k, v
  // 25.0, 21.8 and 21.9; 16 segments q, k, v 27.9, 24.5 and 33.7, o 15.5, 13.3 and 18.2; 1000 tokens in four, o 18.0, 15.8 and 16.4.  Over 356
  // batches of 300 to 9000 tokens the choice is 0.3 % behind the best (2.6 with one price for every sum and fewer tiles than segments).
  const long tiles = std::max<long>(n_seg, (n_tokens + TM - 1) / TM + n_seg / 2);
  const double rows = std::min<double>(TM, (double)n_tokens / tiles) / TM;
  const int nk = (d_in + BK - 1) / BK;
  const double stage = (X_BYTES + n_mats * rmax * 128) / 115e3;
  int best = 1;
  double least = 0;
  for (int ks = 1; ks <= TC_MAX_SLICES && (ks == 1 || nk / ks >= 4); ks *= 2) {
    const int kchunk = (nk + ks - 1) / ks;
    if ((ks - 1) * kchunk >= nk) continue;                                       // every slice of d_in must hold something
    const long at_once = ks <= 2 ? p->sm_count / ks : ks == 4 ? p->sm_count * 9 / 40 : p->sm_count * 13 / 128;
    const double sum = ks == 1 ? 0 : 4 + 0.125 * ks + rows * (n_mats * rmax * ks / 256.0 + (ks == 8 ? 0.25 * std::max(0L, tiles - 4) : 0));
    const double cost = (double)((tiles + at_once - 1) / at_once) * (6 + sum + kchunk * stage);
    if (ks == 1 || cost < least) { least = cost; best = ks; }
  }
  return best;
}

int shrink_tc(fl_pool* p, const TcShrinkArgs& a, const void* x, int rmax, cudaStream_t st) {
  if (a.n_mats < 1 || a.n_mats > 3 || a.d_in % 8 != 0 || a.ksplit < 1 || a.ksplit > TC_MAX_SLICES) return FL_EINVAL;
  alignas(64) CUtensorMap xmap;
  const uint64_t dims[2] = {(uint64_t)a.d_in, (uint64_t)a.n_tokens};
  const uint64_t strides[1] = {(uint64_t)a.d_in * 2};
  const uint32_t box[2] = {BK, TM};
  int rc = tmap::encode_bf16(&xmap, x, 2, dims, strides, box);
  if (rc != FL_OK) return rc;
  const int n_units = (a.n_seg + a.n_tokens / TM) * a.ksplit;     // upper bound of the tile count, times the slices
  const int nm = a.n_mats;
  if (rmax == 16) return nm == 1 ? launch<16, 1>(p, a, xmap, n_units, st) : nm == 2 ? launch<16, 2>(p, a, xmap, n_units, st) : launch<16, 3>(p, a, xmap, n_units, st);
  if (rmax == 32) return nm == 1 ? launch<32, 1>(p, a, xmap, n_units, st) : nm == 2 ? launch<32, 2>(p, a, xmap, n_units, st) : launch<32, 3>(p, a, xmap, n_units, st);
  if (rmax == 64) return nm == 1 ? launch<64, 1>(p, a, xmap, n_units, st) : nm == 2 ? launch<64, 2>(p, a, xmap, n_units, st) : launch<64, 3>(p, a, xmap, n_units, st);
  return FL_EINVAL;
}

}  // namespace sgmv
