"""The layer steps that a serving program has this library run, with their sizes, inputs and necessary work.

One case is one batch of requests taken through one layer over the unified block pool: the q, k, v projections with
the new K, V stored in the requests' blocks, attention over [cached prefix || new tokens], the o projection, and the
MLP's up and down where the layer carries adapters there.  Fields of a case:

  hidden, q_heads, kv_heads, inter   the layer (inter = 0: adapters on the attention projections only)
  n_prefill, len_lo, len_hi, cached  prompts of U{len_lo..len_hi} tokens, the share `cached` of them served from the pool
  n_decode, ctx_lo, ctx_hi           requests with one new token behind U{ctx_lo..ctx_hi} cached tokens
  adapters, rank, alpha              registered adapters, their rank (0: 8, 16, 32 and 64 mixed), Zipf exponent of their use
  plain                              requests of the batch that use no adapter
  base                               True: y = x W + s (x A) B (fl_lora_linear*); False: the adapter term is added to a y
                                     that holds x W already (fl_lora_sgmv*)
  append                             base = False only: "fused" = K, V stored by the projection, "separate" = fl_kv_append
  graph                              the step's kernels are replayed from a CUDA graph, as decode loops do
  swap                               blocks swapped out and in on side streams while the kernels run
  batch                              number of the batch: which lengths and adapters are drawn
"""
import bisect
import itertools
import math
import random

import numpy as np
import torch

from paper_2505_03756_b200 import binding as fl
from paper_2505_03756_b200.synth import LayerShape

SCALE = 2.0
_SHAPES = {  # the layers of the workloads in synth.SHAPES
    "small": dict(hidden=1024, q_heads=8, kv_heads=8, inter=0),
    "7b": dict(hidden=4096, q_heads=32, kv_heads=32, inter=0),
    "13b": dict(hidden=5120, q_heads=40, kv_heads=40, inter=13824),
    "34b": dict(hidden=8192, q_heads=64, kv_heads=8, inter=0),
}


def _case(name, shape, **kw):
    c = dict(name=name, **_SHAPES[shape], n_prefill=0, len_lo=0, len_hi=0, cached=0.0, n_decode=0, ctx_lo=0, ctx_hi=0,
             adapters=1, rank=16, alpha=1.0, plain=0, base=False, append="fused", graph=False, swap=0, batch=0)
    c.update(kw)
    return c


def listed():
    return [
        # a handful of short requests on a small layer through the elementary calls: launches and host work count
        _case("tiny_step", "small", n_prefill=4, len_lo=64, len_hi=64, cached=0.5, adapters=4, rank=8, alpha=0.0,
              append="separate"),
        # one user typing: a single token per step, every weight read once
        _case("chat_decode_7b", "7b", n_decode=1, ctx_lo=700, ctx_hi=700, base=True, graph=True),
        # an ordinary decode batch with the base projections on the path
        _case("decode_13b_base", "13b", n_decode=48, ctx_lo=512, ctx_hi=4096, adapters=128, rank=32, alpha=0.8, base=True,
              graph=True),
        # the largest decode batch: 256 requests, 12 GB of cached KV
        _case("decode_13b", "13b", n_decode=256, ctx_lo=512, ctx_hi=4096, adapters=128, rank=32, alpha=0.8, graph=True),
        # decode over grouped heads
        _case("decode_34b_base", "34b", n_decode=64, ctx_lo=512, ctx_hi=4096, adapters=16, rank=64, alpha=1.0, base=True,
              graph=True),
        # time to first token of one prompt, half of it in the cache
        _case("one_prompt_7b_base", "7b", n_prefill=1, len_lo=1021, len_hi=1021, cached=0.5, base=True),
        # an ordinary prefill batch with the base projections on the path
        _case("prefill_7b_base", "7b", n_prefill=16, len_lo=128, len_hi=1024, cached=0.5, adapters=32, base=True),
        # a large prefill batch, adapter terms and attention only (the default shape of the benchmark)
        _case("prefill_7b", "7b", n_prefill=64, len_lo=128, len_hi=1024, cached=0.5, adapters=32),
        # long prompts whose first three quarters are cached, grouped heads, the highest rank
        _case("prefill_34b_base", "34b", n_prefill=4, len_lo=4096, len_hi=4096, cached=0.75, adapters=16, rank=64, alpha=0.0,
              base=True),
        _case("prefill_34b", "34b", n_prefill=16, len_lo=4096, len_hi=4096, cached=0.75, adapters=16, rank=64, alpha=0.0),
        # continuous batching: decode and prefill requests together, ranks 8 to 64, a few requests on the bare model ...
        _case("mixed_7b_base", "7b", n_prefill=4, len_lo=128, len_hi=1024, cached=0.5, n_decode=28, ctx_lo=512, ctx_hi=4096,
              adapters=200, rank=0, alpha=1.2, plain=4, base=True),
        # ... and with blocks swapped both ways during the step
        _case("mixed_7b_swap", "7b", n_prefill=32, len_lo=128, len_hi=1024, cached=0.5, n_decode=32, ctx_lo=512, ctx_hi=4096,
              adapters=200, rank=0, alpha=1.2, swap=32),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    """One more step of the ranges above: any layer, batches from one request to the largest, odd lengths."""
    every = listed()
    most = {k: max(work(c)[k] for c in every) for k in ("bytes", "flops")}
    while True:
        shape = rng.choice(["small", "7b", "7b", "13b", "34b"])
        kind = rng.choice(["prefill", "prefill", "decode", "decode", "mixed"])
        c = _case("", shape, adapters=_log_int(rng, 1, 200), rank=rng.choice([8, 16, 16, 32, 64, 0]),
                  alpha=rng.choice([0.0, 0.8, 1.0, 1.2]), base=rng.random() < 0.5, append=rng.choice(["fused", "fused", "separate"]),
                  graph=kind == "decode" and rng.random() < 0.75, swap=rng.choice([0, 0, 0, 8, 32]) if kind == "mixed" else 0,
                  batch=rng.randrange(1 << 20))
        del c["name"]
        if kind != "decode":
            c["n_prefill"] = _log_int(rng, 1, 64 if kind == "prefill" else 32)
            c["len_hi"] = _log_int(rng, 48, 4096)
            c["len_lo"] = rng.randint(max(33, c["len_hi"] // 8), c["len_hi"])
            c["cached"] = rng.choice([0.0, 0.5, 0.5, 0.75])
        if kind != "prefill":
            c["n_decode"] = _log_int(rng, 1, 256 if kind == "decode" else 64)
            c["ctx_hi"] = _log_int(rng, 64, 4096)
            c["ctx_lo"] = rng.randint(max(1, c["ctx_hi"] // 8), c["ctx_hi"])
        if rng.random() < 0.25:
            c["plain"] = rng.randint(0, (c["n_prefill"] + c["n_decode"]) // 4)
        w = work(c)
        if all(w[k] <= most[k] for k in most):
            return c


# ------------------------------------------------------------------ the batch that a case stands for
def _shape(case):
    return LayerShape(case["hidden"], case["q_heads"], case["kv_heads"], inter=case["inter"])


def _batch(case):
    """(adapter, cached tokens, new tokens) per request, sorted by adapter as the segments need it, and all ranks."""
    rng = random.Random(case["batch"])
    n = case["n_prefill"] + case["n_decode"]
    bt = _shape(case).block_tokens
    ranks = [case["rank"] or rng.choice([8, 16, 32, 64]) for _ in range(case["adapters"])]
    cum = list(itertools.accumulate((k + 1) ** -case["alpha"] for k in range(case["adapters"])))
    if case["alpha"] == 0.0:
        lora = [i % case["adapters"] for i in range(n)]
    else:
        lora = [min(bisect.bisect(cum, rng.random() * cum[-1]), case["adapters"] - 1) for _ in range(n)]
    for i in rng.sample(range(n), case["plain"]):
        lora[i] = -1
    lens = []
    for i in range(n):
        if i < case["n_decode"]:
            lens.append((rng.randint(case["ctx_lo"], case["ctx_hi"]), 1))
        else:
            total = rng.randint(case["len_lo"], case["len_hi"])
            p = int(total * case["cached"]) // bt * bt
            lens.append((p, total - p))
    reqs = sorted(((a, p, m) for a, (p, m) in zip(lora, lens)), key=lambda r: r[0])
    return reqs, ranks


def work(case):
    """Each input read once, each output written once; multiply-adds as two operations."""
    s = _shape(case)
    reqs, ranks = _batch(case)
    T = sum(m for _, _, m in reqs)
    used = sorted({a for a, _, _ in reqs if a >= 0})
    of_rank = {a: sum(m for b, _, m in reqs if b == a) for a in used}
    n_bytes = 2 * T * s.hidden                                                    # x
    flops = 0.0
    for _, d_in, d_out in s.mats:
        n_bytes += 2 * T * d_out + (2 * d_in * d_out if case["base"] else 2 * T * d_out)      # result; W, or the y it adds to
        n_bytes += sum(2 * ranks[a] * (d_in + d_out) for a in used)
        flops += sum(2.0 * of_rank[a] * ranks[a] * (d_in + d_out) for a in used)
        flops += 2.0 * T * d_in * d_out if case["base"] else 0.0
    n_bytes += 2 * T * s.n_q_heads * s.head_dim                                   # attention output
    n_bytes += sum(p for _, p, _ in reqs) * 2 * s.n_kv_heads * s.head_dim * 2     # cached K and V
    flops += 4.0 * s.head_dim * s.n_q_heads * sum(m * p + m * (m + 1) / 2 for _, p, m in reqs)
    n_bytes += 2 * case["swap"] * s.block_bytes
    return {"bytes": float(n_bytes), "flops": flops}


# ------------------------------------------------------------------ inputs
class _Pool:
    """Owner of a pool's handle, destroyed with the last view of its slabs."""

    def __init__(self, block_bytes, n_blocks, n_host):
        self.handle = None
        self.handle = fl.fl_pool_create(block_bytes, n_blocks, max(1, n_host))
        self.n_blocks, self.n_host, self.values = n_blocks, n_host, block_bytes // 2

    def __del__(self):
        if self.handle is not None:
            torch.cuda.synchronize()
            fl.fl_pool_destroy(self.handle)
            self.handle = None


class _Slab:
    """One of a pool's two slabs as [blocks, values per block] for torch or numpy, without a copy; keeps the pool alive."""

    def __init__(self, pool, host):
        self.pool = pool
        base = (fl.fl_pool_host_base if host else fl.fl_pool_device_base)(pool.handle)
        what = {"shape": (pool.n_host if host else pool.n_blocks, pool.values), "typestr": "<i2", "version": 3, "data": (base, False)}
        setattr(self, "__array_interface__" if host else "__cuda_array_interface__", what)


class _Step:
    """Pool, adapters, index arrays and buffers of one batch, and the calls of its layer step."""

    def __init__(self, case, seed):
        self.case, self.shape = case, _shape(case)
        s, dev = self.shape, torch.device("cuda")
        reqs, ranks = _batch(case)
        mats = [(i, o) for _, i, o in s.mats]
        self.mat = {n: k for k, (n, _, _) in enumerate(s.mats)}
        bt, bb, swap = s.block_tokens, s.block_bytes, case["swap"]
        gen = torch.Generator(device=dev).manual_seed(seed)
        order = np.random.default_rng(seed)
        # blocks that the step writes come first in the slab, in random order, then the swapped ones, then the cached
        # prefixes and the adapters over the rest in random order
        first_new = [p // bt for _, p, _ in reqs]
        n_blk = [-(-(p + m) // bt) for _, p, m in reqs]
        n_new = sum(n_blk) - sum(first_new)
        used = sorted({a for a, _, _ in reqs if a >= 0})
        n_table = {a: fl.fl_lora_blocks(bb, ranks[a], mats) for a in set(used) | {0}}
        n_rest = sum(first_new) + sum(n_table.values())
        self.n_written = n_new + 2 * swap
        n_blocks = self.n_written + n_rest
        owner = _Pool(bb, n_blocks, 2 * swap)
        self.pool = owner.handle
        fl.fl_block_alloc(self.pool, n_blocks)
        slab = torch.as_tensor(_Slab(owner, host=False), device=dev).view(torch.bfloat16)
        slab.normal_(generator=gen)
        self.written = slab[:self.n_written]        # keeps the pool alive, here and in what a pass returns
        new_ids, rest = order.permutation(n_new), self.n_written + order.permutation(n_rest)
        tables, c0, w0 = [], 0, 0
        for f, n in zip(first_new, n_blk):
            tables.append(np.concatenate([rest[c0:c0 + f], new_ids[w0:w0 + n - f]]))
            c0, w0 = c0 + f, w0 + n - f
        for a in sorted(n_table):
            ids, c0 = rest[c0:c0 + n_table[a]], c0 + n_table[a]
            slab[torch.from_numpy(ids).to(dev)] *= 0.02
            fl.fl_lora_register(self.pool, a, ranks[a], mats, ids)

        def ints(v):
            return torch.from_numpy(np.asarray(v, dtype=np.int32)).to(dev)

        seg_ids = [a for a, _ in itertools.groupby(r[0] for r in reqs)]
        seg_len = [sum(m for b, _, m in reqs if b == a) for a in seg_ids]
        self.seg_indptr, self.seg_ids, self.n_seg = ints(np.cumsum([0] + seg_len)), ints(seg_ids), len(seg_ids)
        self.req_indptr = ints(np.cumsum([0] + [m for _, _, m in reqs]))
        self.prefix, self.new = ints([p for _, p, _ in reqs]), ints([m for _, _, m in reqs])
        self.tbl_indptr, self.tbl, self.n_tbl = ints(np.cumsum([0] + n_blk)), ints(np.concatenate(tables)), sum(n_blk)
        self.n_req, self.T = len(reqs), sum(m for _, _, m in reqs)
        T = self.T

        def rows(*shape, std=1.0):
            return torch.empty(*shape, dtype=torch.bfloat16, device=dev).normal_(0.0, std, generator=gen)

        self.x = rows(T, s.hidden)
        self.attn = torch.empty(T, s.n_q_heads, s.head_dim, dtype=torch.bfloat16, device=dev)
        if case["base"]:
            self.y = {n: torch.empty(T, o, dtype=torch.bfloat16, device=dev) for n, _, o in s.mats if n not in ("k", "v")}
            self.w = {n: rows(i, o, std=i ** -0.5) for n, i, o in s.mats}
            self.ws = torch.empty(fl.fl_lora_linear_workspace(T, 3), dtype=torch.uint8, device=dev)
            self.scratch_k = self.scratch_v = None
            if T <= 16 * self.n_seg:                # batches of short segments form x W for K and V in scratch rows
                self.scratch_k, self.scratch_v = (torch.empty(T, s.n_kv_heads * s.head_dim, dtype=torch.bfloat16, device=dev)
                                                  for _ in range(2))
        else:
            self.y = {n: rows(T, o) for n, _, o in s.mats}
            self.ws = torch.empty(fl.fl_lora_sgmv_workspace(T, 3), dtype=torch.uint8, device=dev)
        self.attn_ws = torch.empty(fl.fl_paged_attention_workspace(self.n_req, T, self.n_tbl, s.n_q_heads, s.n_kv_heads),
                                   dtype=torch.uint8, device=dev)
        if swap:
            ids = n_new + order.permutation(2 * swap)
            self.out_dev, self.in_dev = ids[:swap], ids[swap:]
            host = fl.fl_host_block_alloc(self.pool, 2 * swap)
            self.out_host, self.in_host = host[:swap], host[swap:]
            self.host = np.asarray(_Slab(owner, host=True))
            self.host[:] = order.integers(0, 1 << 14, self.host.shape, dtype=np.int16)
            self.side_out, self.side_in = torch.cuda.Stream(), torch.cuda.Stream()
        # y += s (x A) B on one pass and -= on the next: a program gets a new y each step, here its values stay bounded
        self.scales = [SCALE] if case["base"] else [SCALE, -SCALE]
        self.passes, self.graphs = 0, None
        if case["graph"]:
            keep = {n: v.clone() for n, v in self.y.items()}
            self.kernels(SCALE)                     # the first ordinary call configures the kernels
            torch.cuda.synchronize()
            for n, v in keep.items():
                self.y[n].copy_(v)
            self.graphs = [torch.cuda.CUDAGraph() for _ in self.scales]
            for g, scale in zip(self.graphs, self.scales):
                with torch.cuda.graph(g):
                    self.kernels(scale)

    def kernels(self, scale):
        s, y, m = self.shape, self.y, self.mat
        seg = (self.seg_indptr, self.seg_ids, self.n_seg, self.T, scale)
        kv = (self.req_indptr, self.tbl_indptr, self.tbl, self.prefix)
        if self.case["base"]:
            fl.fl_lora_linear_qkv_append(self.pool, y["q"], self.x, self.w["q"], self.w["k"], self.w["v"], m["q"], m["k"], m["v"],
                                         *seg, *kv, self.n_req, s.n_kv_heads, self.scratch_k, self.scratch_v, self.ws)
        elif self.case["append"] == "fused":
            fl.fl_lora_sgmv_qkv_append(self.pool, y["q"], y["k"], y["v"], self.x, m["q"], m["k"], m["v"], *seg, *kv,
                                       self.n_req, s.n_kv_heads, self.ws)
        else:
            fl.fl_lora_sgmv_multi(self.pool, [y["q"], y["k"], y["v"]], self.x, [m["q"], m["k"], m["v"]], *seg, self.ws)
            fl.fl_kv_append(self.pool, y["k"], y["v"], *kv, self.n_req, self.T, s.n_kv_heads)
        fl.fl_paged_attention(self.pool, self.attn, y["q"], *kv, self.new, self.n_req, self.T, self.n_tbl, s.n_q_heads,
                              s.n_kv_heads, s.head_dim ** -0.5, self.attn_ws)
        src = self.attn
        for n in ("o", "up", "down"):
            if n in m:
                if self.case["base"]:
                    fl.fl_lora_linear(self.pool, y[n], src, self.w[n], m[n], *seg, self.ws)
                else:
                    fl.fl_lora_sgmv(self.pool, y[n], src, m[n], *seg, self.ws)
                src = y[n]

    def step(self):
        if self.case["swap"]:
            fl.fl_swap_out(self.pool, self.out_dev, self.out_host, self.side_out)
            fl.fl_swap_in(self.pool, self.in_dev, self.in_host, self.side_in)
        k = self.passes % len(self.scales)
        self.passes += 1
        if self.graphs:
            self.graphs[k].replay()
        else:
            self.kernels(self.scales[k])
        out = {"attention": self.attn, "blocks": self.written, **self.y}
        if self.case["swap"]:
            out["host"] = self.host
        return out


def prepare(case, seed):
    return _Step(case, seed)


def run(state):
    return state.step()


def tolerance(case):
    """bf16 values behind fp32 sums.  The library's two prefill attention kernels and two shrinks (other tiles, other order
    of the sums) differ by at most 3.8e-3 and 2.8e-2 over the listed cases; swapped blocks are bytes and stay the same."""
    return {"rel": 1.5e-2, "max": 0.11}
