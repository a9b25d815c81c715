"""fl_lora_sgmv* on long segments, at the sizes where the stream's pieces end: segments around multiples of 16, 96, 112, 128 and
256 tokens next to one-token segments and segments without an adapter, widths that end inside a warp's 64 or a CTA's
256 columns, ranks that end inside a 16-row step, blocks of 8 and 16 tokens."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.lora import lora_project
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_adapters


@pytest.mark.parametrize("rank,hidden,heads,lens", [
    (16, 200, (3, 1), [97, 1, 255, 16, 300]), (5, 1024, (8, 8), [1, 257, 1, 95, 111, 1]), (32, 328, (2, 1), [128, 513, 17, 40]),
    (24, 264, (2, 2), [1, 1, 700, 2]), (64, 328, (3, 1), [112, 113, 1, 256, 600]), (33, 1096, (4, 2), [224, 15, 225, 1, 1])])
@pytest.mark.parametrize("bt", [16, 8])
def test_sgmv_of_long_segments(rank, hidden, heads, lens, bt):
    from paper_2505_03756_b200 import binding as fl, harness as H
    shape = synth.LayerShape(hidden, *heads, block_tokens=bt)
    n = len(lens)
    wl = synth.make_workload("decode13b", n_req=n, len_range=(3, 40), n_adapters=n, shape=shape)
    wl.ranks[:] = [max(1, rank - i) for i in range(n)]
    wl.lora_of_req[:] = np.arange(n) - 1                  # the first request uses no adapter
    wl.new_lens[:] = lens
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + bt - 1) // bt)) + 200 * n + 64
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        T = wl.n_tokens
        assert T > 16 * s.n_seg
        seg, ids = wl.segments()
        x = wl.x("q")
        tx = H.f32_to_dev(x, s.dev)
        blocks = sorted({int(b) for t in s.kv_tables for b in t})
        for base in (1.0, 0.0):              # with a base projection in y, and the LoRA term alone against its own size
            yb = {m: (wl.y_base(m) * base).astype(np.float32) for m in "qkvo"}
            ty = [H.f32_to_dev(yb[m], s.dev) for m in "qkv"]
            s.sgmv(ty, tx, ["q", "k", "v"])
            for m, t in zip("qkv", ty):
                assert_close(H.dev_to_f32(t), lora_project(yb[m], x, seg, ids, oracle_adapters(wl, m), wl.scale), f"long {T} {m} {base}")
            s.kv_append(ty[1], ty[2])
            torch.cuda.synchronize()
            stored = fl.device_block_bytes(s.pool, s.block_bytes, blocks)
            junk = torch.full_like(ty[1], 5.0)
            s.kv_append(junk, junk)
            y_q = H.f32_to_dev(yb["q"], s.dev)
            s.sgmv_qkv_append(y_q, H.f32_to_dev(yb["k"], s.dev), H.f32_to_dev(yb["v"], s.dev), tx)
            torch.cuda.synchronize()
            assert torch.equal(y_q, ty[0])
            assert np.array_equal(fl.device_block_bytes(s.pool, s.block_bytes, blocks), stored)
        xo = wl.x("o")
        t_o = H.f32_to_dev(wl.y_base("o"), s.dev)
        s.sgmv([t_o], H.f32_to_dev(xo, s.dev), ["o"])
        assert_close(H.dev_to_f32(t_o), lora_project(wl.y_base("o"), xo, seg, ids, oracle_adapters(wl, "o"), wl.scale), f"long {T} o")
        assert s.status()["device_flags"] == 0
    finally:
        s.close()
