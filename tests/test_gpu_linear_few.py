"""fl_lora_linear* on batches of at most 256 tokens (W streamed once for all of them), at the sizes where its tiles end:
token counts around multiples of 16, 128 and 256 and the two ends of the range, ranks that end inside a 16-row step or a
64-row stage, widths that end inside a column tile or a k-stage, one CTA per column tile up to a cluster of eight."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.lora import lora_linear
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_adapters

RANKS = [1, 8, 5, 24, 32, 33, 64, 16]


def _workload(T, shape, per_req, n_adapters):
    """T tokens in requests of `per_req` tokens (the last one takes the rest), ranks from RANKS, every fifth request without
    an adapter."""
    n = max(1, T // per_req)
    wl = synth.make_workload("decode13b", n_req=n, len_range=(3, 40), n_adapters=n_adapters, shape=shape)
    wl.ranks[:] = [RANKS[i % len(RANKS)] for i in range(n_adapters)]
    wl.new_lens[:] = per_req
    wl.new_lens[-1] += T - n * per_req
    wl.lora_of_req[2::5] = -1
    wl.lora_of_req.sort()
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 130 * n_adapters + 64
    return wl


@pytest.mark.parametrize("T,per_req,hidden,heads", [
    (1, 1, 1024, (8, 8)), (2, 1, 4096, (32, 32)), (15, 1, 328, (3, 1)), (16, 16, 328, (3, 1)), (17, 1, 1024, (8, 8)),
    (33, 11, 200, (2, 1)), (127, 1, 1024, (8, 8)), (129, 43, 328, (3, 1)), (200, 100, 1024, (8, 2)), (255, 1, 328, (3, 1)),
    (256, 256, 1024, (8, 8)), (256, 1, 2048, (4, 1)), (257, 1, 328, (3, 1)),
    (176, 44, 4096, (8, 8)), (177, 1, 4096, (64, 8)), (209, 9, 1024, (8, 8)), (300, 100, 328, (64, 8)), (384, 128, 328, (64, 8))])
def test_linear_of_few_tokens(T, per_req, hidden, heads):
    from paper_2505_03756_b200 import binding as fl, harness as H
    wl = _workload(T, synth.LayerShape(hidden, *heads), per_req, 12)
    assert wl.n_tokens == T
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        s.fill_prefix_kv()
        dims = dict((n, o) for n, _, o in wl.shape.mats)
        seg, ids = wl.segments()
        x = wl.x("q")
        tx = H.f32_to_dev(x, s.dev)
        tw = {m: H.f32_to_dev(wl.weight(m), s.dev) for m in "qkvo"}
        want = {m: lora_linear(x, wl.weight(m), seg, ids, oracle_adapters(wl, m), wl.scale) for m in "qkv"}
        # q, k, v into y, with K and V stored afterwards; then the fused call, bit for bit the same
        ty = [torch.full((T, dims[m]), 7.0, dtype=torch.bfloat16, device=s.dev) for m in "qkv"]
        s.lora_linear(ty, tx, [tw[m] for m in "qkv"], ["q", "k", "v"])
        for m, t in zip("qkv", ty):
            assert_close(H.dev_to_f32(t), want[m], f"few tokens {T} {m}")
        blocks = sorted({int(b) for t in s.kv_tables for b in t})
        s.kv_append(ty[1], ty[2])
        torch.cuda.synchronize()
        stored = fl.device_block_bytes(s.pool, s.block_bytes, blocks)
        junk = torch.full_like(ty[1], 5.0)
        s.kv_append(junk, junk)
        y_q = torch.full_like(ty[0], -5.0)
        s.lora_linear_qkv_append(y_q, tx, tw["q"], tw["k"], tw["v"])
        torch.cuda.synchronize()
        assert torch.equal(y_q, ty[0])
        assert np.array_equal(fl.device_block_bytes(s.pool, s.block_bytes, blocks), stored)
        # one projection (narrow: more CTAs per column tile), and the LoRA term alone against its own size
        xo = wl.x("o")
        y_o = torch.full((T, hidden), 3.0, dtype=torch.bfloat16, device=s.dev)
        s.lora_linear([y_o], H.f32_to_dev(xo, s.dev), [tw["o"]], ["o"])
        assert_close(H.dev_to_f32(y_o), lora_linear(xo, wl.weight("o"), seg, ids, oracle_adapters(wl, "o"), wl.scale), f"few tokens {T} o")
        s.lora_linear([y_o], H.f32_to_dev(xo, s.dev), [torch.zeros_like(tw["o"])], ["o"])
        assert_close(H.dev_to_f32(y_o), lora_linear(xo, np.zeros_like(wl.weight("o")), seg, ids, oracle_adapters(wl, "o"), wl.scale),
                     f"few tokens {T} LoRA term")
        assert s.status()["device_flags"] == 0
    finally:
        s.close()


@pytest.mark.parametrize("long_tokens,n_one,hidden,heads,n_adapters", [
    (258, 0, 328, (3, 1), 3), (382, 1, 1024, (8, 8), 3), (258, 2, 328, (64, 8), 4), (370, 14, 200, (64, 8), 16), (500, 12, 328, (3, 1), 20), (513, 0, 4096, (3, 1), 2),
    (1024, 40, 200, (2, 1), 60), (2300, 17, 1024, (8, 2), 24)])
def test_linear_of_long_segments_next_to_one_token_segments(long_tokens, n_one, hidden, heads, n_adapters):
    """The GEMM for longer batches: tiles of 256 tokens that end in the middle of a segment, tiles with more LoRA stages than
    are looked up together, tiles without any, both column widths."""
    from paper_2505_03756_b200 import harness as H
    wl = synth.make_workload("decode13b", n_req=n_one + 2, len_range=(3, 40), n_adapters=n_adapters,
                             shape=synth.LayerShape(hidden, *heads))
    wl.ranks[:] = [RANKS[i % len(RANKS)] for i in range(n_adapters)]
    wl.lora_of_req[:] = np.sort(np.arange(n_one + 2) % n_adapters)
    wl.lora_of_req[0] = -1
    wl.new_lens[-1] = long_tokens // 3
    wl.new_lens[n_one // 2] = long_tokens - long_tokens // 3
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 130 * n_adapters + 64
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        T = wl.n_tokens
        assert T > 256 and T > 16 * s.n_seg
        dims = dict((n, o) for n, _, o in wl.shape.mats)
        seg, ids = wl.segments()
        x = wl.x("q")
        tx = H.f32_to_dev(x, s.dev)
        for scale_w in (1.0, 0.0):           # with W, and the LoRA term alone against its own size
            tw = [H.f32_to_dev(wl.weight(m), s.dev) * scale_w for m in "qkv"]
            ty = [torch.full((T, dims[m]), 7.0, dtype=torch.bfloat16, device=s.dev) for m in "qkv"]
            s.lora_linear(ty, tx, tw, ["q", "k", "v"])
            for m, t in zip("qkv", ty):
                want = lora_linear(x, wl.weight(m) * scale_w, seg, ids, oracle_adapters(wl, m), wl.scale)
                assert_close(H.dev_to_f32(t), want, f"long and one-token segments {T} {m} {scale_w}")
        assert s.status()["device_flags"] == 0
    finally:
        s.close()


@pytest.mark.parametrize("T,per_req,hidden,heads,n_adapters", [
    (1, 1, 1024, (8, 8), 2), (40, 1, 1024, (8, 8), 12), (130, 1, 4096, (8, 8), 4), (200, 1, 1024, (8, 2), 3), (256, 1, 328, (64, 8), 4),
    (300, 20, 328, (3, 1), 2), (330, 3, 328, (64, 8), 3)])
def test_v_slots_behind_a_request_are_cleared(T, per_req, hidden, heads, n_adapters):
    """K and V stored by the projection itself into blocks that hold old values behind the requests' last tokens: the same bytes as the
    projection and the KV append, whichever kernel serves the batch and whichever CTA clears the slots."""
    from paper_2505_03756_b200 import binding as fl, harness as H
    wl = _workload(T, synth.LayerShape(hidden, *heads), per_req, n_adapters)
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        s.fill_prefix_kv()
        dims = dict((n, o) for n, _, o in wl.shape.mats)
        tx = H.f32_to_dev(wl.x("q"), s.dev)
        tw = [H.f32_to_dev(wl.weight(m), s.dev) for m in "qkv"]
        ty = [torch.empty((T, dims[m]), dtype=torch.bfloat16, device=s.dev) for m in "qkv"]
        s.lora_linear(ty, tx, tw, ["q", "k", "v"])
        s.kv_append(ty[1], ty[2])
        torch.cuda.synchronize()
        blocks = sorted({int(b) for t in s.kv_tables for b in t})
        stored = fl.device_block_bytes(s.pool, s.block_bytes, blocks)
        kv, bt = wl.shape.n_kv_heads, wl.shape.block_tokens
        for r in range(wl.n_req):
            last = int(wl.prefix_lens[r] + wl.new_lens[r]) - 1
            b = int(s.kv_tables[r][last // bt])
            data = fl.fl_block_read(s.pool, b, s.block_bytes).reshape(2, kv, bt, 256).copy()
            assert not data[1, :, last % bt + 1:].any()
            data[1, :, last % bt:] = 0x55                       # the last token's own slot too: it is stored again
            fl.fl_block_write(s.pool, b, data.reshape(-1))
        y_q = torch.empty_like(ty[0])
        s.lora_linear_qkv_append(y_q, tx, *tw)
        torch.cuda.synchronize()
        assert torch.equal(y_q, ty[0])
        assert np.array_equal(fl.device_block_bytes(s.pool, s.block_bytes, blocks), stored)
        assert s.status()["device_flags"] == 0
    finally:
        s.close()
