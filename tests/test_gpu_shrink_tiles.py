"""The shrink on tcgen05 at the sizes where its tiles and slices end: segments around multiples of 128 tokens next to one-token
segments and one without an adapter, input widths that end inside a stage of 64 values or leave the last slice short, and
batches of one to some tens of tiles, so that d_in goes to one, two, four and eight CTAs of a cluster."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.lora import lora_linear, lora_project
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_adapters


# hidden (= d_in), tokens per segment, rank
@pytest.mark.parametrize("hidden,lens,rank", [
    (2056, [127, 128, 129, 1], 33), (2048, [257, 1], 64), (4160, [40], 32), (5120, [96, 32], 64), (4096, [300, 300, 300, 300], 17), (1096, [128] * 24, 64),
    (328, [90, 700], 20), (2048, [128] * 60, 24), (7176, [255, 1, 1200], 16),
    (4104, [40] * 39, 64)])
def test_shrink_of_long_segments(hidden, lens, rank):
    from paper_2505_03756_b200 import harness as H
    shape = synth.LayerShape(hidden, 2, 2, block_tokens=16)
    n = len(lens)
    wl = synth.make_workload("decode13b", n_req=n, len_range=(3, 20), n_adapters=n, shape=shape)
    wl.ranks[:] = [max(1, rank - i % 5) for i in range(n)]
    wl.lora_of_req[:] = np.arange(n) - (1 if n > 2 else 0)        # the first of several requests uses no adapter
    wl.new_lens[:] = lens
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 260 * n + 64
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        assert wl.n_tokens > 16 * s.n_seg
        seg, ids = wl.segments()
        x = wl.x("q")
        tx = H.f32_to_dev(x, s.dev)
        ad = {m: oracle_adapters(wl, m) for m in "qkv"}
        yb = {m: wl.y_base(m) * 0 for m in "qkv"}                 # the LoRA term alone, against its own size
        out = []
        for _ in range(2):
            ty = [H.f32_to_dev(yb[m], s.dev) for m in "qkv"]
            s.sgmv(ty, tx, ["q", "k", "v"])
            one = H.f32_to_dev(yb["q"], s.dev)
            s.sgmv([one], tx, ["q"])
            out.append(ty + [one])
        assert all(torch.equal(a, b) for a, b in zip(*out))       # the slices are added in one order
        for m, t in zip("qkvq", out[0]):
            assert_close(H.dev_to_f32(t), lora_project(yb[m], x, seg, ids, ad[m], wl.scale), f"{hidden} {m}")
        w = wl.weight("q")
        lin = torch.empty_like(out[0][0])
        s.lora_linear([lin], tx, [H.f32_to_dev(w, s.dev)], ["q"])
        assert_close(H.dev_to_f32(lin), lora_linear(x, w, seg, ids, ad["q"], wl.scale), f"{hidden} linear")
        assert s.status()["device_flags"] == 0
    finally:
        s.close()


# around the lines of the shrink with more stages in flight: up to 15 clusters of eight at rank 64, twelve to twenty segments and fewer, slices of five stages
@pytest.mark.parametrize("hidden,rank,lens", [
    (4096, 64, [4] * 12), (4096, 64, [1] * 14), (4096, 64, [1] * 15), (4104, 64, [1] * 16), (8192, 64, [3] * 16), (4096, 64, [1] * 20),
    (2624, 64, [5, 1, 30, 2]), (2560, 32, [2] * 30), (2560, 32, [2] * 37), (2568, 16, [1] * 44), (2560, 16, [1] * 60)])
def test_shrink_of_decode_steps(hidden, rank, lens):
    from paper_2505_03756_b200 import harness as H
    shape = synth.LayerShape(hidden, 2, 2, block_tokens=16)
    n = len(lens)
    wl = synth.make_workload("decode13b", n_req=n, len_range=(3, 20), n_adapters=n, shape=shape)
    wl.ranks[:] = [rank - i % 3 for i in range(n)]
    wl.lora_of_req[:] = np.arange(n)
    wl.new_lens[:] = lens
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 260 * n + 64
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        seg, ids = wl.segments()
        x, w = wl.x("q"), wl.weight("q")
        tx, tw = H.f32_to_dev(x, s.dev), H.f32_to_dev(w, s.dev)
        out = []
        for _ in range(3):
            y = torch.full((wl.n_tokens, 256), float("nan"), dtype=torch.bfloat16, device=s.dev)
            s.lora_linear([y], tx, [tw], ["q"])
            out.append(y)
        assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
        assert_close(H.dev_to_f32(out[0]), lora_linear(x, w, seg, ids, oracle_adapters(wl, "q"), wl.scale), f"decode {hidden} rank {rank}")
        assert s.status()["device_flags"] == 0
    finally:
        s.close()
