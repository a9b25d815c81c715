// Paged attention over [cached prefix || new tokens] read from pool blocks (Section 2.1, Section 4.2).
//
// A plan kernel sorts the requests of a batch into two work lists: requests with at most 16 query
// rows per KV head (decode steps) are cut into chunks of keys that independent CTAs reduce
// (split-KV, merged by the last of them); the others (prefill) are cut into tiles of 64 query rows per head, or of 128 for the
// tcgen05 kernel.  A few decode requests, and small batches of any kind, are served without a plan.
// Both kernels stage KV pages (one 4 KiB contiguous piece per block, KV head and K/V side) into
// shared memory with 16-byte cp.async through the block table and run QK^T and PV on bf16 tensor
// cores with an fp32 online softmax.
#include <math.h>
#include <algorithm>
#include "mma_utils.cuh"
#include "attention.cuh"
#include "pool.cuh"

using namespace attn;

namespace {

constexpr int QT = QT_MMA;
constexpr int MAX_CHUNK = 2048;       // keys per work item of the split decode at most

__device__ __forceinline__ int block_excl_scan(int val, int* sh, int& total) {
  // exclusive scan over the 256 threads of the plan CTA
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = val;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  int wbase = 0, tot = 0;
  for (int w = 0; w < 8; ++w) {
    if (w < warp) wbase += sh[w];
    tot += sh[w];
  }
  __syncthreads();
  total = tot;
  return wbase + incl - val;
}

// What a batch with both kinds of work takes, in us, when the persistent prefill kernel has p of the SMs and the decode kernel
// the others, and all of them behind the prefill kernel's end.  The decode kernel is bound by the copy rate from DECODE_SMS SMs
// on; a prefill unit's step takes STEP_US, one fifth longer beside it.  (7B, 16 x 512 new tokens behind 512 and 48 decode requests
// of about 1400 keys: 299 us one after the other, 279, 270, 264 and 351 us with 100, 82, 70 and 50 SMs for the prefill kernel;
// 1000 prefill tokens beside 1.2 GB of decode pages: 198 us, 194, 191 and 228 us with 90, 50 and 8.  Grouped heads, one after the other
// and with the share chosen here, 34B: 16 decode requests of 2700 keys beside 1000 new tokens 144 and 97 us, beside 16 x 500 279 and 253,
// 64 of 3600 keys beside 16 x 500 393 and 383; of 75 batches on 7B, 13B and 34B one is slower, by 1 %.)
constexpr float STEP_US = 1.7f, KEY_US = 8e-5f, DECODE_SMS = 112.f;
__device__ __forceinline__ float shared_time(int p, int sms, float unit_us, int n_units, float decode_us) {
  const float pre = unit_us * (p < sms ? 1.2f : 1.f) * ((n_units + p - 1) / p);
  const float done = pre * fminf(1.f, (sms - p) / DECODE_SMS);
  return pre + fmaxf(0.f, decode_us - done);
}

__global__ void __launch_bounds__(256) attn_plan_kernel(const AttnArgs a, int chunk, int qt, int sms) {
  __shared__ unsigned steps, keys;           // 128-key steps of all prefill tiles; keys of the decode requests
  __shared__ unsigned long long best;
  __shared__ int sh[8];
  __shared__ int hist[64], cursor[64];
  pdl_wait();                 // the lists may still be read, and the request arrays written, by the kernel before
  pdl_launch_dependents();    // the prefill kernel sets itself up (barriers, TMEM) while this single CTA plans
  const int group = a.n_q / a.n_kv;
  for (int i = threadIdx.x; i < a.n_req * a.n_kv; i += 256) a.chunks_done[i] = 0u;
  if (threadIdx.x < 64) hist[threadIdx.x] = 0;
  if (threadIdx.x == 0) { steps = keys = 0; best = ~0ull; }
  __syncthreads();
  // Prefill requests are ordered by context length (in 128-key steps), longest first, so that the CTAs that take work
  // from the list finish together; the tiles of one request stay next to each other (its later tiles first), so the
  // units that read the same K/V pages run at about the same time and the second reader finds them in L2.
  auto key_of = [&](int i) { return min(63, (a.prefix_lens[i] + a.new_lens[i] + 127) / 128); };
  int base_p = 0, base_d = 0;
  for (int i0 = 0; i0 < a.n_req; i0 += 256) {
    const int i = i0 + threadIdx.x;
    int n = 0, ctx = 0, tiles = 0, chunks = 0;
    bool dec = false;
    if (i < a.n_req) {
      n = a.new_lens[i];
      ctx = a.prefix_lens[i] + n;
      if (n > 0) {
        dec = n * group <= DEC_ROWS;
        if (dec) chunks = (ctx + chunk - 1) / chunk; else tiles = (n + qt - 1) / qt;
      }
    }
    int tot_p, tot_d;
    block_excl_scan(tiles, sh, tot_p);
    const int off_d = base_d + block_excl_scan(chunks, sh, tot_d);
    if (i < a.n_req) {
      // a request whose chunks do not all fit in the list (contexts longer than the caller's n_tbl covers) gets no
      // output: the chunks that did fit only write partial slots inside the workspace and count as none of it (the
      // overflow raises FLAG_BAD_POS below)
      if (tiles > 0) {
        atomicAdd(&hist[key_of(i)], tiles);
        // a tile reads the keys up to its last row; one and a half steps more are a unit's start and end
        atomicAdd(&steps, (unsigned)((long long)tiles * (2 * (ctx - n) + n + qt + 3 * 128) / 256));
      }
      if (chunks > 0) atomicAdd(&keys, (unsigned)ctx);
      if (chunks > 0) {
        DecodeItem d;
        d.req = i;
        d.prefix = ctx - n;
        d.n_new = n;
        d.tok0 = a.req_indptr[i];
        d.tbl0 = a.tbl_indptr[i];
        d.tbl_n = a.tbl_indptr[i + 1] - d.tbl0;
        d.n_chunks = off_d + chunks > a.max_decode ? 0 : chunks;
        for (int c = 0; c < chunks; ++c) {
          d.chunk = c;
          if (off_d + c < a.max_decode) a.decode_list[off_d + c] = d;
        }
      }
    }
    base_p += tot_p;
    base_d += tot_d;
  }
  __syncthreads();
  if (base_p > 0 && threadIdx.x < 32) {        // bins from the last to the first, two per lane
    const int b = 63 - 2 * threadIdx.x;
    const int h0 = hist[b], h1 = hist[b - 1];
    int incl = h0 + h1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if ((int)threadIdx.x >= d) incl += o;
    }
    cursor[b] = incl - h0 - h1;
    cursor[b - 1] = incl - h1;
  }
  __syncthreads();
  for (int i = threadIdx.x; base_p > 0 && i < a.n_req; i += 256) {
    const int n = a.new_lens[i];
    if (n <= 0 || n * group <= DEC_ROWS) continue;
    const int tiles = (n + qt - 1) / qt;
    const int first = atomicAdd(&cursor[key_of(i)], tiles);
    // An item of 256 tokens is two 128-row tiles that share one K/V stream and costs as many key tiles as its later
    // tile needs.  With an odd number of 128-row tiles the request's FIRST tile (shortest context) goes alone and the
    // pairs start at token 128, instead of the last tile (longest context) going alone: one key tile less per pair.
    const bool lone_first = qt == 256 && (((n + 127) / 128) & 1);
    for (int t = 0; t < tiles; ++t) {
      const int u = tiles - 1 - t;      // item number in token order
      const int q0 = lone_first ? (u == 0 ? 0 : 128 + (u - 1) * 256) : u * qt;
      if (first + t < a.max_prefill) a.prefill_list[first + t] = make_int2(i, q0);
    }
  }
  if (base_p > 0 && base_d > 0) {        // the share that takes the least time, the largest of several
    const int n_units = base_p * tc2_heads_per_item(a.n_q, a.n_kv);
    for (int p = threadIdx.x + 1; p <= sms; p += 256)
      atomicMin(&best, (unsigned long long)__float_as_uint(shared_time(p, sms, STEP_US * steps / base_p, n_units, KEY_US * keys * a.n_kv)) << 32 | (unsigned)(sms - p));
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (base_p > a.max_prefill || base_d > a.max_decode) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
    a.hdr->n_prefill = min(base_p, a.max_prefill);
    a.hdr->n_decode = min(base_d, a.max_decode);
    a.hdr->next_unit = 0;
    a.hdr->prefill_ctas = base_p > 0 && base_d > 0 ? sms - (int)(unsigned)best : sms;
  }
}

// Online-softmax update for one warp: S holds NT 8-key tiles of raw scores for rows g and g+8.
// Key index of S[n][c] is u0 + 8n + 2*(lane&3) + (c&1); row g sees keys <= lim0, row g+8 keys <= lim1.
template <int NT>
__device__ __forceinline__ void softmax_step(float (&S)[NT][4], float (&O)[16][4], float (&m)[2], float (&l)[2],
                                             int u0, int lim0, int lim1, float scale_log2, uint32_t (&P)[NT / 2][4]) {
  const int t4 = threadIdx.x & 3;
  float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    const int u = u0 + 8 * n + 2 * t4;
    S[n][0] = u <= lim0 ? S[n][0] * scale_log2 : -INFINITY;
    S[n][1] = u + 1 <= lim0 ? S[n][1] * scale_log2 : -INFINITY;
    S[n][2] = u <= lim1 ? S[n][2] * scale_log2 : -INFINITY;
    S[n][3] = u + 1 <= lim1 ? S[n][3] * scale_log2 : -INFINITY;
    mx0 = fmaxf(mx0, fmaxf(S[n][0], S[n][1]));
    mx1 = fmaxf(mx1, fmaxf(S[n][2], S[n][3]));
  }
  mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
  mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
  mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
  mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
  const float mn0 = fmaxf(m[0], mx0), mn1 = fmaxf(m[1], mx1);
  // a row that has seen no key yet keeps max = -inf; use 0 as the reference so nothing becomes NaN
  const float r0 = mn0 == -INFINITY ? 0.f : mn0, r1 = mn1 == -INFINITY ? 0.f : mn1;
  const float a0 = exp2f(m[0] - r0), a1 = exp2f(m[1] - r1);
  m[0] = mn0; m[1] = mn1;
  float s0 = 0.f, s1 = 0.f;
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    S[n][0] = exp2f(S[n][0] - r0); S[n][1] = exp2f(S[n][1] - r0);
    S[n][2] = exp2f(S[n][2] - r1); S[n][3] = exp2f(S[n][3] - r1);
    s0 += S[n][0] + S[n][1];
    s1 += S[n][2] + S[n][3];
  }
  l[0] = l[0] * a0 + s0;
  l[1] = l[1] * a1 + s1;
#pragma unroll
  for (int n = 0; n < 16; ++n) {
    O[n][0] *= a0; O[n][1] *= a0; O[n][2] *= a1; O[n][3] *= a1;
  }
#pragma unroll
  for (int k = 0; k < NT / 2; ++k) {
    P[k][0] = pack_bf16(S[2 * k][0], S[2 * k][1]);
    P[k][1] = pack_bf16(S[2 * k][2], S[2 * k][3]);
    P[k][2] = pack_bf16(S[2 * k + 1][0], S[2 * k + 1][1]);
    P[k][3] = pack_bf16(S[2 * k + 1][2], S[2 * k + 1][3]);
  }
}

// S[NT] += Q(16 x 128) K^T for NT*8 keys staged as [key][128] rows (swizzled, 16 chunks per row).
template <int NT>
__device__ __forceinline__ void qk_tile(float (&S)[NT][4], const uint32_t (&qf)[8][4], uint32_t ksm) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
#pragma unroll
    for (int p = 0; p < NT / 2; ++p) {
      uint32_t bf[4];
      ldmatrix_x4(bf, ksm + swz(16 * p + (lane & 7) + 8 * (lane >> 4), 2 * ks + ((lane >> 3) & 1), 16));
      mma_bf16(S[2 * p], qf[ks], bf[0], bf[1]);
      mma_bf16(S[2 * p + 1], qf[ks], bf[2], bf[3]);
    }
  }
}

// O += P(16 x NT*8 keys) V for values staged as [key][128] rows.
template <int NT>
__device__ __forceinline__ void pv_tile(float (&O)[16][4], const uint32_t (&P)[NT / 2][4], uint32_t vsm) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int ks = 0; ks < NT / 2; ++ks) {
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      uint32_t bf[4];
      ldmatrix_x4_trans(bf, vsm + swz(16 * ks + (lane & 7) + 8 * ((lane >> 3) & 1), 2 * p + (lane >> 4), 16));
      mma_bf16(O[2 * p], P[ks], bf[0], bf[1]);
      mma_bf16(O[2 * p + 1], P[ks], bf[2], bf[3]);
    }
  }
}

__device__ __forceinline__ const unsigned char* page_ptr(const PoolView& pv, uint32_t blk, int side_head, bool& ok) {
  if (blk >= pv.n_blocks) {
    atomicOr(pv.flags, (uint32_t)FLAG_BAD_BLOCK);
    ok = false;
    return pv.slab;
  }
  ok = true;
  return pv.slab + (size_t)blk * pv.block_bytes + (size_t)side_head * PAGE_BYTES;
}

// ------------------------------------------------------------------ decode (split-KV)
constexpr int CL_OFF = 4 * DEC_ROWS * D * 4 + 4 * DEC_ROWS * 8;        // a CTA's own result, behind those of its four warps
template <bool PAST_L1>
__device__ __forceinline__ uint32_t load_word(const __nv_bfloat16* p) {
  return PAST_L1 ? __ldcg(reinterpret_cast<const uint32_t*>(p)) : *reinterpret_cast<const uint32_t*>(p);
}

// Which request's pages a CTA takes where there is no plan and a request gets as many CTAs as it has pages for: one for up to
// `part_pages`, two or four beyond, those of four first, so that a request's CTAs lie in one cluster of four.  Every warp finds
// it by itself from the requests' numbers, a request per lane, and has the numbers of its own at hand then.
__device__ __forceinline__ bool find_share(const AttnArgs& a, int slot, int n_slots, int part_pages, DecodeItem& it) {
  const int lane = threadIdx.x & 31;
  struct Request {
    int n_new, prefix, tok0, tbl0, tbl_n, log_parts;      // log_parts: -1 = no new token
  };
  auto load = [&](int i) {
    Request r = {0, 0, 0, 0, 0, -1};
    if (i < a.n_req) {
      r.n_new = a.new_lens[i];
      r.prefix = a.prefix_lens[i];
      r.tok0 = a.req_indptr[i];
      r.tbl0 = a.tbl_indptr[i];
      r.tbl_n = a.tbl_indptr[i + 1] - r.tbl0;
      const int pages = (r.prefix + r.n_new + BT - 1) / BT;
      // (a table too short for them: no output)
      if (r.n_new > 0) r.log_parts = pages <= part_pages || pages > r.tbl_n ? 0 : pages <= 2 * part_pages ? 1 : 2;
    }
    return r;
  };
  const Request first = load(lane);
  int n[3] = {0, 0, 0};
  for (int r0 = 0; r0 < a.n_req; r0 += 32) {
    const int c = r0 == 0 ? first.log_parts : load(r0 + lane).log_parts;
#pragma unroll
    for (int k = 0; k < 3; ++k) n[k] += __popc(__ballot_sync(0xffffffffu, c == k));
  }
  // (contexts longer than the caller's n_tbl covers: one CTA each)
  const bool fit = n[0] + 2 * n[1] + 4 * n[2] <= n_slots;
  if (!fit) {
    n[0] += n[1] + n[2];
    n[1] = n[2] = 0;
  }
  int behind = 0, k = 0, count = 0;
#pragma unroll
  for (int c = 2; c >= 0; --c) {
    if (slot >= behind && slot < behind + (n[c] << c)) {
      k = c;
      count = (slot - behind) >> c;
    }
    behind += n[c] << c;
  }
  if (slot >= behind) return false;
  for (int r0 = 0; r0 < a.n_req; r0 += 32) {
    const Request r = r0 == 0 ? first : load(r0 + lane);
    const uint32_t m = __ballot_sync(0xffffffffu, (!fit && r.log_parts > 0 ? 0 : r.log_parts) == k);
    if (count < __popc(m)) {
      const bool mine = (m >> lane & 1u) && __popc(m & ((1u << lane) - 1u)) == count;
      const int src = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
      it.req = r0 + src;
      it.chunk = slot & ((1 << k) - 1);
      it.n_chunks = 1 << k;
      it.n_new = __shfl_sync(0xffffffffu, r.n_new, src);
      it.prefix = __shfl_sync(0xffffffffu, r.prefix, src);
      it.tok0 = __shfl_sync(0xffffffffu, r.tok0, src);
      it.tbl0 = __shfl_sync(0xffffffffu, r.tbl0, src);
      it.tbl_n = __shfl_sync(0xffffffffu, r.tbl_n, src);
      return true;
    }
    count -= __popc(m);
  }
  return false;
}

// One CTA per (request, chunk of keys, KV head).  Rows = new tokens x query heads of the group
// (at most 16).  The four warps take pages round-robin, each with its own double buffer, and merge
// their partial (max, sum, O) through shared memory at the end.  The CTA that finishes a request's last chunk for its KV
// head combines the chunks' partial results (always in chunk order): as a kernel of its own the combination took 7 us
// behind one request of 700 keys and 15 us behind 64 requests of grouped heads, half of it launch and look-ups.
// What bounds it: reading K and V (a decode step of 256 requests runs at the copy rate); for a few requests the chain item ->
// block ids -> pages -> partial results, which is why an item holds all of a request's numbers.
// BESIDE: behind the persistent prefill kernel this one starts while that one runs.  The kernels before the prefill kernel are
// complete then (it lets this one start after its own wait) and nothing of what it writes is read here; what they wrote is
// read past L1.  One CTA more than the work needs waits for the prefill kernel's end, so that this grid does not end, and
// the kernel behind it does not start, before it.
// CLUSTER: a few decode requests and nothing else.  No plan: the CTAs of a cluster share the pages of one (request, KV head) and
// the first of them fetches the others' partial results from their shared memory.
// PACKED: the same, with clusters of four that a long request has to itself and short ones share (find_share).
constexpr int MAX_FEW_ROWS = 64;      // query rows per KV head, in all, of a batch served without a plan
constexpr int PACK = 4;
enum { PLAIN = 0, BESIDE = 1, CLUSTER = 2, PACKED = 3 };
template <int MODE>
__global__ void __launch_bounds__(ATT_THREADS) attn_decode_kernel(const AttnArgs a, int chunk, int n_slots) {
  constexpr bool NO_PLAN = MODE == CLUSTER || MODE == PACKED;
  extern __shared__ __align__(128) unsigned char smem[];
  if (MODE != BESIDE || blockIdx.x == gridDim.x - 1) pdl_wait();
  pdl_launch_dependents();    // the next call's first kernel may set itself up; it waits for this grid before it reads anything
  const int csize = MODE == CLUSTER ? chunk : MODE == PACKED ? PACK : 1;            // CTAs per cluster
  const int item = blockIdx.x / csize / a.n_kv, h = blockIdx.x / csize % a.n_kv;
  if (MODE == BESIDE && item >= a.max_decode) return;
  DecodeItem it;
  if (NO_PLAN) {
    if (MODE == PACKED) {
      if (!find_share(a, item * PACK + blockIdx.x % PACK, n_slots, chunk, it)) return;       // (a cluster's barriers do without the CTAs that have left)
    } else {
      it.req = item;
      it.chunk = blockIdx.x % csize;
      it.n_chunks = csize;
      it.n_new = a.new_lens[item];
      it.prefix = a.prefix_lens[item];
      it.tok0 = a.req_indptr[item];
      it.tbl0 = a.tbl_indptr[item];
      it.tbl_n = a.tbl_indptr[item + 1] - it.tbl0;
    }
    if (it.n_new * (a.n_q / a.n_kv) <= (int)blockIdx.y * DEC_ROWS) return;       // (the same answer in all of the request's CTAs)
    const int pages = (it.prefix + it.n_new + BT - 1) / BT;
    if (pages > it.tbl_n || it.n_new * (a.n_q / a.n_kv) > MAX_FEW_ROWS) {
      if (threadIdx.x == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
      return;
    }
    chunk = max(4, (pages + it.n_chunks - 1) / it.n_chunks) * BT;       // a page for every warp at least
  } else if (MODE == BESIDE) {
    const int4* src = reinterpret_cast<const int4*>(a.decode_list + item);
    const int4 lo = __ldcg(src), hi = __ldcg(src + 1);
    it.req = lo.x; it.chunk = lo.y; it.prefix = lo.z; it.n_new = lo.w;
    it.tok0 = hi.x; it.tbl0 = hi.y; it.tbl_n = hi.z; it.n_chunks = hi.w;
  } else {
    it = a.decode_list[item];
  }
  if (!NO_PLAN && item >= (MODE == BESIDE ? __ldcg(&a.hdr->n_decode) : a.hdr->n_decode)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const int i = it.req, c = it.chunk;
  const int n_new = it.n_new, prefix = it.prefix, ctx = prefix + n_new;
  const int group = a.n_q / a.n_kv;
  // a plan's items have at most 16 rows; where there is none, clusters further back in the grid take a request's rows from 16 on
  const int r0 = NO_PLAN ? (int)blockIdx.y * DEC_ROWS : 0;
  const int rows = min(DEC_ROWS, n_new * group - r0);
  const int tok0 = it.tok0;
  const int u_begin = c * chunk, u_end = min(ctx, u_begin + chunk);
  const int n_pages = max(0, (u_end - u_begin + BT - 1) / BT);       // (none for the last CTAs of a cluster with few pages)
  const int tbl0 = it.tbl0, tbl_n = it.tbl_n;
  const int pg0 = u_begin / BT;
  // a chunk behind the end of the table has no keys to read; the request's other chunks then never count up to all of them
  if (!NO_PLAN && pg0 + n_pages > tbl_n) {
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
    return;
  }
  // lane k holds the block of this warp's k-th page
  static_assert(MAX_CHUNK / BT <= 4 * 32, "one page per lane");
  const uint32_t my_blk = MODE == BESIDE && warp + 4 * lane < n_pages ? __ldcg(a.tbl + tbl0 + pg0 + warp + 4 * lane) : 0u;
  // query fragments: row r -> (new token (r0 + r) / group, query head h*group + (r0 + r) % group)
  uint32_t qf[8][4];
  int lim[2];
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const int r = g + 8 * hh;
    const bool ok = r < rows;
    const int j = ok ? (r0 + r) / group : 0;
    lim[hh] = ok ? prefix + j : -1;
    const __nv_bfloat16* qp = a.q + ((size_t)(tok0 + j) * a.n_q + (h * group + (ok ? (r0 + r) % group : 0))) * D;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      qf[ks][hh] = ok ? load_word<MODE == BESIDE>(qp + 16 * ks + 2 * t4) : 0u;
      qf[ks][hh + 2] = ok ? load_word<MODE == BESIDE>(qp + 16 * ks + 2 * t4 + 8) : 0u;
    }
  }
  float O[16][4];
#pragma unroll
  for (int n = 0; n < 16; ++n) O[n][0] = O[n][1] = O[n][2] = O[n][3] = 0.f;
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};

  const uint32_t wbase = smem_u32(smem) + warp * (4 * PAGE_BYTES);   // per warp: 2 stages x (K page, V page)
  auto load_page = [&](int pg, int st) {
    const uint32_t blk = MODE == BESIDE ? __shfl_sync(0xffffffffu, my_blk, pg >> 2) : a.tbl[tbl0 + pg0 + pg];
    bool ok;
    const unsigned char* kp = page_ptr(a.pv, blk, h, ok);
    const unsigned char* vp = kp + (size_t)a.n_kv * PAGE_BYTES;
    const uint32_t ks = wbase + st * 2 * PAGE_BYTES, vs = ks + PAGE_BYTES;
    // slots behind the last stored token may hold anything: their V rows are zero-filled so that a
    // zero weight times a stale non-finite value cannot reach the output
    const int valid = u_end - (u_begin + pg * BT);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int cidx = lane + 32 * q;          // 256 chunks per page: row = cidx / 16
      const int row = cidx >> 4, ch = cidx & 15;
      cp_async16(ks + swz(row, ch, 16), kp + cidx * 16, ok);
      cp_async16(vs + swz(row, ch, 16), vp + cidx * 16, ok && row < valid);
    }
  };
  if (warp < n_pages) load_page(warp, 0);
  cp_async_commit();
  int st = 0;
  for (int pg = warp; pg < n_pages; pg += 4, st ^= 1) {
    if (pg + 4 < n_pages) load_page(pg + 4, st ^ 1);
    cp_async_commit();
    cp_async_wait<1>();
    __syncwarp();
    const uint32_t ks = wbase + st * 2 * PAGE_BYTES, vs = ks + PAGE_BYTES;
    float S[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    qk_tile<2>(S, qf, ks);
    uint32_t P[1][4];
    softmax_step<2>(S, O, m, l, u_begin + pg * BT, lim[0], lim[1], a.scale_log2, P);
    pv_tile<2>(O, P, vs);
    __syncwarp();
  }
  cp_async_wait<0>();
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    l[hh] += __shfl_xor_sync(0xffffffffu, l[hh], 1);
    l[hh] += __shfl_xor_sync(0xffffffffu, l[hh], 2);
  }
  __syncthreads();
  // merge the four warps: red_o [warp][16][128], red_ml [warp][16]
  float* red_o = reinterpret_cast<float*>(smem);
  float2* red_ml = reinterpret_cast<float2*>(smem + 4 * DEC_ROWS * D * 4);
#pragma unroll
  for (int n = 0; n < 16; ++n) {
    float* p = red_o + (warp * DEC_ROWS + g) * D + 8 * n + 2 * t4;
    p[0] = O[n][0]; p[1] = O[n][1];
    p[8 * D] = O[n][2]; p[8 * D + 1] = O[n][3];
  }
  if (t4 == 0) {
    red_ml[warp * DEC_ROWS + g] = make_float2(m[0], l[0]);
    red_ml[warp * DEC_ROWS + g + 8] = make_float2(m[1], l[1]);
  }
  __syncthreads();
  for (int e = tid; e < rows * D; e += ATT_THREADS) {
    const int r = e / D, col = e % D;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < 4; ++w) M = fmaxf(M, red_ml[w * DEC_ROWS + r].x);
    const float ref = M == -INFINITY ? 0.f : M;
    float L = 0.f, o = 0.f;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float2 ml = red_ml[w * DEC_ROWS + r];
      const float sc = exp2f(ml.x - ref);
      L += ml.y * sc;
      o += red_o[(w * DEC_ROWS + r) * D + col] * sc;
    }
    if (NO_PLAN && it.n_chunks > 1) {
      float* const mine = reinterpret_cast<float*>(smem + CL_OFF);
      mine[e] = o;
      if (col == 0) reinterpret_cast<float2*>(smem + CL_OFF + DEC_ROWS * D * 4)[r] = make_float2(M, L);
    } else if (it.n_chunks == 1) {
      const int j = (r0 + r) / group, hq = h * group + (r0 + r) % group;
      a.out[((size_t)(tok0 + j) * a.n_q + hq) * D + col] = __float2bfloat16_rn(L > 0.f ? o / L : 0.f);
    } else {
      const size_t slot = ((size_t)item * a.n_kv + h) * DEC_ROWS + r;
      a.part_o[slot * D + col] = o;
      if (col == 0) a.part_ml[slot] = make_float2(M, L);
    }
  }
  if (it.n_chunks <= 1) return;
  if (NO_PLAN) {
    __syncwarp();
    cluster_sync();
    const uint32_t first = blockIdx.x % csize;       // (read by the first of the request's CTAs)
    if (c == 0)
      for (int e = tid; e < rows * (D / 4); e += ATT_THREADS) {
        const int r = e / (D / 4);
        const uint32_t po = smem_u32(smem) + CL_OFF + e * 16, pm = smem_u32(smem) + CL_OFF + DEC_ROWS * D * 4 + r * 8;
        float4 p[8];
        float2 ml[8];
        float ref = -INFINITY;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k < it.n_chunks) {
            p[k] = ld_cluster_f32x4(map_cluster_rank(po, first + k));
            ml[k] = ld_cluster_f32x2(map_cluster_rank(pm, first + k));
            ref = fmaxf(ref, ml[k].x);
          }
        if (ref == -INFINITY) ref = 0.f;
        float L = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k < it.n_chunks) {
            const float sc = exp2f(ml[k].x - ref);
            L += ml[k].y * sc;
            o.x += p[k].x * sc; o.y += p[k].y * sc; o.z += p[k].z * sc; o.w += p[k].w * sc;
          }
        const int j = (r0 + r) / group, hq = h * group + (r0 + r) % group;
        uint2 q = make_uint2(0u, 0u);
        if (L > 0.f) q = make_uint2(pack_bf16(o.x / L, o.y / L), pack_bf16(o.z / L, o.w / L));
        *reinterpret_cast<uint2*>(a.out + ((size_t)(tok0 + j) * a.n_q + hq) * D + (e % (D / 4)) * 4) = q;
      }
    __syncwarp();
    cluster_sync();              // nobody leaves while its results are still being read
    return;
  }
  // ---- the last chunk of this request and head to get here combines them all
  __shared__ int last;
  __syncthreads();
  if (tid == 0) {       // releases the whole CTA's partial results (the barrier orders them before it) and acquires the others'
    unsigned done;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(done) : "l"(&a.chunks_done[(size_t)i * a.n_kv + h]) : "memory");
    last = done == (unsigned)(it.n_chunks - 1);
  }
  __syncthreads();
  if (!last) return;
  float* row_max = reinterpret_cast<float*>(smem);           // [16]
  const size_t slot0 = ((size_t)(item - c) * a.n_kv + h) * DEC_ROWS, slot_step = (size_t)a.n_kv * DEC_ROWS;
  for (int r = warp; r < rows; r += 4) {
    float M = -INFINITY;
    for (int k = lane; k < it.n_chunks; k += 32) M = fmaxf(M, __ldcg(&a.part_ml[slot0 + k * slot_step + r]).x);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, d));
    if (M == -INFINITY) M = 0.f;
    if (lane == 0) row_max[r] = M;
  }
  __syncthreads();
  for (int e = tid; e < rows * (D / 4); e += ATT_THREADS) {
    const int r = e / (D / 4), col = (e % (D / 4)) * 4;
    const float ref = row_max[r];
    float L = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < it.n_chunks; ++k) {
      const size_t slot = slot0 + k * slot_step + r;
      const float2 ml = __ldcg(&a.part_ml[slot]);
      const float4 p = __ldcg(reinterpret_cast<const float4*>(a.part_o + slot * D + col));
      const float sc = exp2f(ml.x - ref);
      L += ml.y * sc;
      o.x += p.x * sc; o.y += p.y * sc; o.z += p.z * sc; o.w += p.w * sc;
    }
    const int j = (r0 + r) / group, hq = h * group + (r0 + r) % group;
    uint2 q = make_uint2(0u, 0u);
    if (L > 0.f) q = make_uint2(pack_bf16(o.x / L, o.y / L), pack_bf16(o.z / L, o.w / L));
    *reinterpret_cast<uint2*>(a.out + ((size_t)(tok0 + j) * a.n_q + hq) * D + col) = q;
  }
}

// ------------------------------------------------------------------ prefill (tensor-core tiles, mma.sync)
// One CTA per (request, tile of 64 new tokens, query head); warp w owns rows 16w..16w+15.
// PLANNED = false: small batches, all requests, whatever their new tokens, in one kernel.  Every warp finds its tile by itself from the
// requests' numbers, 32 requests at a time.  What such a batch takes is the chain of look-ups and launches: plan, tcgen05 prefill kernel and
// a decode kernel without work take 10 us for 4 requests of 32 new tokens behind 32 (8 heads), this one 5.
__device__ __forceinline__ bool find_query_tile(const AttnArgs& a, int item, int& req, int& q0) {
  const int lane = threadIdx.x & 31;
  for (int r0 = 0; r0 < a.n_req; r0 += 32) {
    const int tiles = r0 + lane < a.n_req ? (max(0, a.new_lens[r0 + lane]) + QT - 1) / QT : 0;
    int incl = tiles;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    const uint32_t behind = __ballot_sync(0xffffffffu, incl > item);      // the first request that ends behind the tile
    if (behind) {
      const int src = __ffs(behind) - 1;
      req = r0 + src;
      q0 = (item - __shfl_sync(0xffffffffu, incl - tiles, src)) * QT;
      return true;
    }
    item -= __shfl_sync(0xffffffffu, incl, 31);
  }
  return false;
}
// Without a plan a warp of the grid's last CTA looks for what the plan would have: more tiles than the grid has, which nobody serves, and
// contexts beyond what n_tbl covers.
__device__ __forceinline__ void check_sizes(const AttnArgs& a, int chunk) {
  const int lane = threadIdx.x & 31, group = a.n_q / a.n_kv;
  int tiles = 0, chunks = 0;
  for (int i = lane; i < a.n_req; i += 32) {
    const int n = max(0, a.new_lens[i]);
    tiles += (n + QT - 1) / QT;
    if (n > 0 && n * group <= DEC_ROWS) chunks += (a.prefix_lens[i] + n + chunk - 1) / chunk;
  }
  tiles = __reduce_add_sync(0xffffffffu, tiles);
  chunks = __reduce_add_sync(0xffffffffu, chunks);
  if (lane == 0 && (tiles > a.max_prefill || chunks > a.max_decode)) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
}
template <bool PLANNED>
__global__ void __launch_bounds__(ATT_THREADS) attn_prefill_kernel(const AttnArgs a, int chunk) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int item = blockIdx.x / a.n_q, hq = blockIdx.x % a.n_q;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  int i, q0;
  if (PLANNED) {
    if (item >= a.hdr->n_prefill) return;
    const int2 it = a.prefill_list[item];
    i = it.x;
    q0 = it.y;
  } else {
    pdl_wait();                 // q, K and V come from the kernel right before this one
    pdl_launch_dependents();
    const bool found = find_query_tile(a, item, i, q0);
    if (blockIdx.x + 1 == gridDim.x && warp == 0) check_sizes(a, chunk);       // (as a rule this CTA has no tile)
    if (!found) return;
  }
  const int n_new = a.new_lens[i], prefix = a.prefix_lens[i], ctx = prefix + n_new;
  const int h = hq / (a.n_q / a.n_kv);
  const int tok0 = a.req_indptr[i] + q0;
  const int q_rows = min(QT, n_new - q0);
  const int kv_end = min(ctx, prefix + q0 + QT);
  const int n_kt = (kv_end + KT - 1) / KT;
  const int tbl0 = a.tbl_indptr[i], tbl_n = a.tbl_indptr[i + 1] - tbl0;
  if ((kv_end + BT - 1) / BT > tbl_n) {
    if (tid == 0) atomicOr(a.pv.flags, (uint32_t)FLAG_BAD_POS);
    return;
  }
  constexpr int TILE_BYTES = KT * D * 2;     // 16 KiB
  const uint32_t qs = smem_u32(smem);        // Q tile, later the output tile
  const uint32_t kv0 = qs + QT * D * 2;      // 2 stages x (K tile, V tile)
  const int crow = tid >> 4, cch = tid & 15;
  // Q tile
#pragma unroll
  for (int r = 0; r < QT / 8; ++r) {
    const int row = crow + 8 * r;
    const bool ok = row < q_rows;
    cp_async16(qs + swz(row, cch, 16), a.q + ((size_t)(tok0 + (ok ? row : 0)) * a.n_q + hq) * D + cch * 8, ok);
  }
  auto load_kv = [&](int kt, int st) {
    const uint32_t ks = kv0 + st * 2 * TILE_BYTES, vs = ks + TILE_BYTES;
#pragma unroll
    for (int r = 0; r < KT / 8; ++r) {
      const int row = crow + 8 * r;
      const int u = kt * KT + row;
      bool ok = u < kv_end;
      const unsigned char* kp = a.pv.slab;
      if (ok) kp = page_ptr(a.pv, a.tbl[tbl0 + u / BT], h, ok);
      const unsigned char* vp = kp + (size_t)a.n_kv * PAGE_BYTES;
      const int off = (u % BT) * (D * 2) + cch * 16;
      cp_async16(ks + swz(row, cch, 16), kp + off, ok);
      cp_async16(vs + swz(row, cch, 16), vp + off, ok);
    }
  };
  load_kv(0, 0);
  cp_async_commit();

  float O[16][4];
#pragma unroll
  for (int n = 0; n < 16; ++n) O[n][0] = O[n][1] = O[n][2] = O[n][3] = 0.f;
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
  const int row0 = warp * 16 + g;
  const int lim0 = row0 < q_rows ? prefix + q0 + row0 : -1;
  const int lim1 = row0 + 8 < q_rows ? prefix + q0 + row0 + 8 : -1;
  uint32_t qf[8][4];

  for (int kt = 0; kt < n_kt; ++kt) {
    const int st = kt & 1;
    if (kt + 1 < n_kt) load_kv(kt + 1, st ^ 1);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    if (kt == 0) {
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        ldmatrix_x4(qf[ks], qs + swz(warp * 16 + (lane & 7) + 8 * ((lane >> 3) & 1), 2 * ks + (lane >> 4), 16));
    }
    const uint32_t ks = kv0 + st * 2 * TILE_BYTES, vs = ks + TILE_BYTES;
    // keys beyond every row of this warp contribute nothing: skip the tile for this warp
    if (kt * KT <= prefix + q0 + warp * 16 + 15) {
      float S[8][4];
#pragma unroll
      for (int n = 0; n < 8; ++n) S[n][0] = S[n][1] = S[n][2] = S[n][3] = 0.f;
      qk_tile<8>(S, qf, ks);
      uint32_t P[4][4];
      softmax_step<8>(S, O, m, l, kt * KT, lim0, lim1, a.scale_log2, P);
      pv_tile<8>(O, P, vs);
    }
    __syncthreads();
  }
  cp_async_wait<0>();
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    l[hh] += __shfl_xor_sync(0xffffffffu, l[hh], 1);
    l[hh] += __shfl_xor_sync(0xffffffffu, l[hh], 2);
  }
  const float inv0 = l[0] > 0.f ? 1.f / l[0] : 0.f, inv1 = l[1] > 0.f ? 1.f / l[1] : 0.f;
  // stage the output tile in the Q buffer (each warp only touches its own 16 rows), then 16-byte stores
#pragma unroll
  for (int n = 0; n < 16; ++n) {
    *reinterpret_cast<uint32_t*>(smem + swz(row0, n, 16) + 4 * t4) = pack_bf16(O[n][0] * inv0, O[n][1] * inv0);
    *reinterpret_cast<uint32_t*>(smem + swz(row0 + 8, n, 16) + 4 * t4) = pack_bf16(O[n][2] * inv1, O[n][3] * inv1);
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < QT / 8; ++r) {
    const int row = crow + 8 * r;
    if (row < q_rows)
      *reinterpret_cast<uint4*>(a.out + ((size_t)(tok0 + row) * a.n_q + hq) * D + cch * 8) =
          *reinterpret_cast<const uint4*>(smem + swz(row, cch, 16));
  }
}

int pick_chunk(int n_tbl, int n_kv) {
  // enough (chunk, head) items to fill the GPU several times over, chunks of 64..2048 keys (256 requests of up to 4096 keys on
  // 13B: the layer step takes 1906, 1877 and 1871 us with at most 1024, 1536 and 2048; longer ones leave a longer tail)
  long long c = ((long long)n_tbl * BT * n_kv + 1183) / 1184;
  c = (c + 63) / 64 * 64;
  if (c < 64) c = 64;
  if (c > MAX_CHUNK) c = MAX_CHUNK;
  return (int)c;
}

// CTAs that share the pages of a (request, KV head) where a few decode requests are served without a plan, 0 = with one.  Without it
// the contexts' lengths are not known when the grid is chosen: enough CTAs that a CTA has no more than 160 + 4 n_req pages even if one
// request had them all, more where SMs are idle and a CTA keeps eight pages; with more than one CTA each, a plan where that needs more than
// 600 CTAs.  (packed_slots then looks at the batches of one long request.)
// KV append and attention of a layer, with the plan and without.  7B: 1 request of 134 keys 12.5 and 9.4 us, of 3000 28.8 and 19.8;
// 3 of 140 14.6 and 10.5; 8 of 550 34.3 and 27.9; 16 of 130 32.5 and 20.2; 26 of 95 29.6 and 22.8; 40 of 60 29.2 and 26.5; but 8 of
// 1500 50 and 61.  34B: 3 of 2000 40.3 and 17.2, 8 of 550 21.3 and 12.2 us.  13B: 30 of 95 34.5 and 28.2; but 9 of 1200 55 and 77 us.
int cluster_size(int n_req, int n_tbl, int n_kv, int sms) {
  const long long units = (long long)n_req * n_kv;
  const int worst = 160 + 4 * n_req;
  int cs = 1;
  while (cs <= 8 && n_tbl > worst * cs) cs *= 2;
  if (cs > 8 || (cs > 1 && units * cs > 600)) return 0;
  while (cs < 8 && units * cs * 2 <= 2 * sms && n_tbl >= 16ll * cs * n_req) cs *= 2;
  return cs;
}

// A batch whose n_tbl entries may be one request's nearly all: with the same number of CTAs for every request that one would keep a warp
// busy with more than 25 to 37 pages and some more for every other request (the plan's time grows with them too).  Then a request gets
// CTAs as it has pages: `slots` of them per KV head (a request of p pages takes at most 1 + 1.5 p / part_pages), 0 = the same number for
// each, -1 = a plan.  Small parts as long as the CTAs with work run at once (three fit on an SM) and those without are not many more; where
// even large parts take twice that, the many short requests are better off with a CTA each, and from 200 pages on with a plan.  (4 requests
// of 1300 keys on 7B, a layer step of 41 us: in parts of eight pages 16 CTAs per head, 512 in all, it took 48.)
// Attention with the same number of CTAs, as here, and with the plan (of the tree that had nothing else).  One request has nearly all: 7B, 5 requests,
// 2560 keys 37, 14 and 24 us; 8, 3200 keys 30, 15, 29; 12, 2560 keys 41, 16, 26; 13B, 8, 2560 keys 42, 17, 27.  One has four times as many as the
// others: 13B, 4 requests of 600 keys 29, 15, 23; 7B, 6 22, 15, 23.  Lengths from one to eight times the shortest: 7B, 5 of 350 keys
// 13.4, 13.2, 23; 8 of 370 14.4, 13.3, 19; 16 of 180 13.3, 15.2, 20; a layer of 8 KV heads, 16 of 370 11.3, 10.6, 20.
struct Packed {
  int slots, part_pages;
};
Packed packed_slots(int n_req, int n_tbl, int n_kv, int csize, int sms) {
  const int longest = n_tbl - n_req + 1;
  if (n_req < 2 || csize >= PACK || longest <= (csize == 1 ? 100 : 150) + n_req * csize) return {0, 0};
  Packed p = {0, 0};
  for (int pages : {8, 12, 16, 24, 32, 48}) {
    p.part_pages = pages;
    p.slots = (std::min(n_req + n_tbl * 3 / (2 * pages), PACK * n_req) + PACK - 1) / PACK * PACK;
    const int alike = n_tbl <= pages * n_req ? 1 : n_tbl <= 2 * pages * n_req ? 2 : PACK;       // CTAs of a request if all are alike
    if (p.slots * n_kv <= 4 * sms && n_req * alike * n_kv <= 3 * sms) return p;
  }
  if (p.slots * n_kv > 6 * sms) p.slots = longest > 200 ? -1 : 0;
  return p;
}

// Batches that attn_prefill_kernel<false> serves by itself: contexts of at most eight blocks in the mean, 40 for the longest if the others have
// one each (the lengths themselves are not known here), and CTAs that run in three rounds at most.  A CTA takes 2.3 us
// per 64 keys, so it is contexts that the line is about.  Attention, this kernel and the three of the planned way, in us, heads / KV heads
// 8/8, 32/32, 64/8: 1 request of 32 new tokens behind 32 5.0 and 9.6, 5.1 and 10.0, 5.1 and 10.4; 4 such 5.1 and 9.9, 5.7 and 10.4, 6.1 and
// 11.4; 4 of 64 behind 64 7.3 and 10.0, 8.7 and 10.6, 9.2 and 11.9.
// Beyond: 1 request of 64 new tokens behind 192 12.0 and 11.4, 12.1 and 11.5, 12.3 and 12.8; 1 of 128 behind 384 21 and 14, 21 and 14, 25 and 16.
// One request has nearly all of the table, a decode step's keys beside prompts of 16 tokens: 14 blocks, 6 requests 10 and 10, 11 and 15, 13 and 21;
// 26 blocks 16 and 10, 17 and 16, 21 and 22; 40 blocks 22 and 11, 24 and 18, 28 and 24 (a prompt's keys 22 and 17, 24 and 18, 28 and 19), the
// most that the rule lets through is lost there; among 60 requests 24 and 23 on 8 heads.  64 blocks, 16 requests, 35 to 38 and 15 to 29.
bool small_batch(int n_req, int n_tokens, int n_tbl, int n_q, int sms) {
  return (n_tokens / QT + n_req) * (long long)n_q <= 6ll * sms && n_tbl <= 8ll * n_req && n_tbl - n_req < 40;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct WsLayout {
  size_t hdr, prefill_list, decode_list, chunks_done, part_o, part_ml, total;
  int max_prefill, max_decode, chunk;
};

WsLayout ws_layout(int n_req, int n_tokens, int n_tbl, int n_kv) {
  WsLayout w;
  w.chunk = pick_chunk(n_tbl, n_kv);
  w.max_prefill = n_tokens / QT + n_req;
  w.max_decode = (int)(((long long)n_tbl * BT) / w.chunk) + n_req;
  size_t off = 0;
  w.hdr = off; off = align256(off + sizeof(PlanHdr));
  w.prefill_list = off; off = align256(off + sizeof(int2) * (size_t)w.max_prefill);
  w.decode_list = off; off = align256(off + sizeof(DecodeItem) * (size_t)w.max_decode);
  w.chunks_done = off; off = align256(off + sizeof(unsigned) * (size_t)n_req * n_kv);
  w.part_o = off; off = align256(off + sizeof(float) * (size_t)w.max_decode * n_kv * DEC_ROWS * D);
  w.part_ml = off; off = align256(off + sizeof(float2) * (size_t)w.max_decode * n_kv * DEC_ROWS);
  w.total = off;
  return w;
}

}  // namespace

extern "C" {

size_t fl_paged_attention_workspace(int n_req, int n_tokens, int n_tbl, int n_q_heads, int n_kv_heads) {
  (void)n_q_heads;
  if (n_req <= 0 || n_tokens < 0 || n_tbl < 0 || n_kv_heads <= 0) return 256;
  return ws_layout(n_req, n_tokens, n_tbl, n_kv_heads).total;
}

int fl_paged_attention(fl_pool* p, fl_bf16* out, const fl_bf16* q, const int32_t* req_indptr,
                       const int32_t* kv_tbl_indptr, const uint32_t* kv_tbl, const int32_t* prefix_lens,
                       const int32_t* new_lens, int n_req, int n_tokens, int n_tbl,
                       int n_q_heads, int n_kv_heads, float sm_scale,
                       void* workspace, size_t workspace_bytes, fl_stream stream) {
  if (!p || n_req < 0 || n_tokens < 0 || n_tbl < 0 || n_q_heads < 1 || n_kv_heads < 1 || n_q_heads % n_kv_heads != 0)
    return FL_EINVAL;
  if (p->block_bytes != (size_t)2 * n_kv_heads * PAGE_BYTES) return FL_EINVAL;   // needs 16-token blocks
  if (n_req == 0 || n_tokens == 0) return FL_OK;
  if (!out || !q || !req_indptr || !kv_tbl_indptr || !kv_tbl || !prefix_lens || !new_lens || !workspace) return FL_EINVAL;
  const WsLayout w = ws_layout(n_req, n_tokens, n_tbl, n_kv_heads);
  if (workspace_bytes < w.total) return FL_ENOMEM;
  unsigned char* ws = reinterpret_cast<unsigned char*>(workspace);
  AttnArgs a;
  a.pv = p->view();
  a.out = reinterpret_cast<__nv_bfloat16*>(out);
  a.q = reinterpret_cast<const __nv_bfloat16*>(q);
  a.req_indptr = req_indptr;
  a.tbl_indptr = kv_tbl_indptr;
  a.tbl = kv_tbl;
  a.prefix_lens = prefix_lens;
  a.new_lens = new_lens;
  a.n_req = n_req;
  a.n_q = n_q_heads;
  a.n_kv = n_kv_heads;
  a.scale_log2 = sm_scale * 1.4426950408889634f;
  a.hdr = reinterpret_cast<PlanHdr*>(ws + w.hdr);
  a.prefill_list = reinterpret_cast<int2*>(ws + w.prefill_list);
  a.decode_list = reinterpret_cast<DecodeItem*>(ws + w.decode_list);
  a.chunks_done = reinterpret_cast<unsigned*>(ws + w.chunks_done);
  a.part_o = reinterpret_cast<float*>(ws + w.part_o);
  a.part_ml = reinterpret_cast<float2*>(ws + w.part_ml);
  a.max_prefill = w.max_prefill;
  a.max_decode = w.max_decode;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != p->device) cudaSetDevice(p->device);
  const cudaStream_t st = (cudaStream_t)stream;
  constexpr int DEC_SMEM = 4 * 4 * PAGE_BYTES;                 // 64 KiB
  constexpr int PRE_SMEM = QT * D * 2 + 2 * 2 * KT * D * 2;    // 80 KiB
  static bool configured[16] = {};
  int rc = FL_OK;
  do {
    if (!configured[p->device & 15]) {
      if (cudaFuncSetAttribute(attn_decode_kernel<PLAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, DEC_SMEM) != cudaSuccess ||
          cudaFuncSetAttribute(attn_decode_kernel<BESIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, DEC_SMEM) != cudaSuccess ||
          cudaFuncSetAttribute(attn_decode_kernel<CLUSTER>, cudaFuncAttributeMaxDynamicSharedMemorySize, DEC_SMEM) != cudaSuccess ||
          cudaFuncSetAttribute(attn_decode_kernel<PACKED>, cudaFuncAttributeMaxDynamicSharedMemorySize, DEC_SMEM) != cudaSuccess ||
          cudaFuncSetAttribute(attn_prefill_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, PRE_SMEM) != cudaSuccess ||
          cudaFuncSetAttribute(attn_prefill_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, PRE_SMEM) != cudaSuccess) {
        p->last_cuda = (int)cudaGetLastError();
        rc = FL_ECUDA;
        break;
      }
      configured[p->device & 15] = true;
    }
    // the tensor-core kernels fold sm_scale into the exponent and take row maxima of raw scores: they need sm_scale > 0
    const int kind = sm_scale > 0.f ? p->prefill_kernel : 1;
    // upper bound of the plan's tile count: full tiles plus one ragged tile per prefill request, and a
    // request is a prefill only with more than DEC_ROWS / group new tokens
    const int group = n_q_heads / n_kv_heads;
    const int max_req = std::min(n_req, n_tokens / (DEC_ROWS / group + 1));
    const int max_items = std::min(w.max_prefill, n_tokens / tc2_tile_tokens(n_q_heads, n_kv_heads) + max_req);
    // No prefill request is possible, or decode steps are meant (a request with more than 16 rows, next to some without any, takes
    // several clusters; in the grid they cost the 64 requests of 40 keys of a 7B layer what the plan does: 37 against 36 us).
    const int passes = max_items == 0 ? 1 : (n_tokens * group + DEC_ROWS - 1) / DEC_ROWS;
    const bool few = max_items == 0 || (n_tokens <= n_req && n_tokens * group <= MAX_FEW_ROWS && (long long)n_req * n_kv_heads * passes <= 6000);
    const int csize = kind == 0 && few ? cluster_size(n_req, n_tbl, n_kv_heads, p->sm_count) : 0;
    const Packed packed = csize > 0 ? packed_slots(n_req, n_tbl, n_kv_heads, csize, p->sm_count) : Packed{-1, 0};
    if (packed.slots >= 0) {
      const cudaError_t e =
          packed.slots > 0 ? launch_pdl_cluster(attn_decode_kernel<PACKED>, dim3((unsigned)(packed.slots * n_kv_heads), (unsigned)passes), dim3(PACK),
                                                dim3(ATT_THREADS), DEC_SMEM, st, a, packed.part_pages, packed.slots)
                    : launch_pdl_cluster(attn_decode_kernel<CLUSTER>, dim3((unsigned)(n_req * n_kv_heads * csize), (unsigned)passes), dim3((unsigned)csize),
                                         dim3(ATT_THREADS), DEC_SMEM, st, a, csize, 0);
      if (e != cudaSuccess) {
        p->last_cuda = (int)e;
        rc = FL_ECUDA;
      }
      break;
    }
    if (kind == 0 && small_batch(n_req, n_tokens, n_tbl, n_q_heads, p->sm_count)) {
      const cudaError_t e = launch_pdl(attn_prefill_kernel<false>, dim3((unsigned)(w.max_prefill * n_q_heads)), dim3(ATT_THREADS), PRE_SMEM, st, a, w.chunk);
      if (e != cudaSuccess) {
        p->last_cuda = (int)e;
        rc = FL_ECUDA;
      }
      break;
    }
    // every kernel of the call is a programmatic dependent launch: it may start while the one before it drains
    // and waits inside for that kernel's results
    if (launch_pdl(attn_plan_kernel, dim3(1), dim3(256), 0, st, a, w.chunk,
                   kind == 0 ? tc2_tile_tokens(n_q_heads, n_kv_heads) : QT_MMA, p->sm_count) != cudaSuccess) {
      p->last_cuda = (int)cudaGetLastError();
      rc = FL_ECUDA;
      break;
    }
    bool beside = false;       // a prefill kernel that the decode kernel works beside
    if (kind == 0) {
      rc = launch_prefill_tc2(p, a, n_tokens, max_items, st);
      if (rc != FL_OK) break;
      beside = max_items > 0;
    } else {
      attn_prefill_kernel<true><<<(unsigned)w.max_prefill * n_q_heads, ATT_THREADS, PRE_SMEM, st>>>(a, w.chunk);
    }
    cudaError_t e = launch_pdl(beside ? attn_decode_kernel<BESIDE> : attn_decode_kernel<PLAIN>, dim3((unsigned)w.max_decode * n_kv_heads + (beside ? 1u : 0u)),
                               dim3(ATT_THREADS), DEC_SMEM, st, a, w.chunk, 0);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
      p->last_cuda = (int)e;
      rc = FL_ECUDA;
    }
  } while (0);
  if (prev != p->device && prev >= 0) cudaSetDevice(prev);
  return rc;
}

}  // extern "C"
