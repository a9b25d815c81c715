"""fl_lora_linear* with an infinity and NaNs in one adapter's B rows: its own tokens get them, those of the other adapters and of no
adapter do not, although they share tiles, stages and clusters with it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.lora import lora_linear
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_adapters

BAD = 2                                      # the adapter
SPOTS = [(0, 0, np.inf), (3, 5, np.nan), (7, 130, -np.inf), (1, -1, np.inf), (4, 64, np.nan)]      # rank-row, column, value


def check(new_lens, lora, hidden, heads, ranks, mats="qkv"):
    from paper_2505_03756_b200 import harness as H
    wl = synth.make_workload("decode13b", n_req=len(new_lens), len_range=(3, 40), n_adapters=len(ranks), shape=synth.LayerShape(hidden, *heads))
    wl.ranks[:], wl.new_lens[:], wl.lora_of_req[:] = ranks, new_lens, lora
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 130 * len(ranks) + 64
    clean = {m: oracle_adapters(wl, m) for m in mats}
    whole = type(wl).adapter

    def poisoned(a, m):
        A, B = whole(wl, a, m)
        if a == BAD:
            B = B.copy()
            for r, c, v in SPOTS:
                B[min(r, B.shape[0] - 1), c % B.shape[1]] = v
        return A, B

    wl.adapter = poisoned
    seg, ids = wl.segments()
    T = wl.n_tokens
    own = np.zeros(T, dtype=bool)
    for k, a in enumerate(ids):
        own[seg[k]:seg[k + 1]] = a == BAD
    assert own.any() and not own.all()
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        x = wl.x("q")
        w = {m: wl.weight(m) for m in mats}
        dims = dict((n, o) for n, _, o in wl.shape.mats)
        ty = [torch.full((T, dims[m]), 7.0, dtype=torch.bfloat16, device=s.dev) for m in mats]
        s.lora_linear(ty, H.f32_to_dev(x, s.dev), [H.f32_to_dev(w[m], s.dev) for m in mats], list(mats))
        assert s.status()["device_flags"] == 0
        for m, t in zip(mats, ty):
            got, want = H.dev_to_f32(t), lora_linear(x, w[m], seg, ids, clean[m], wl.scale)
            cols = np.zeros(dims[m], dtype=bool)
            cols[[c % dims[m] for _, c, _ in SPOTS]] = True
            assert not np.isfinite(got[np.ix_(own, cols)]).any(), m
            assert_close(got[~own], want[~own], f"other tokens {m}")
            assert_close(got[np.ix_(own, ~cols)], want[np.ix_(own, ~cols)], f"own tokens, other columns {m}")
    finally:
        s.close()


@pytest.mark.parametrize("T,hidden,heads", [(24, 1024, (8, 8)), (40, 4096, (32, 32)), (128, 328, (3, 1)), (200, 1024, (8, 2))])
def test_few_tokens_of_many_adapters(T, hidden, heads):
    """One token per request: units of several adapters in a stage, stages dealt over a cluster."""
    ranks = [16, 64, 33, 8, 24, 64, 5]
    check([1] * T, np.sort(np.arange(T) % 8) - 1, hidden, heads, ranks)


@pytest.mark.parametrize("new_lens,lora,hidden,heads", [
    ([90, 1, 1, 60, 1, 1, 1, 120], [-1, 0, 1, 2, 2, 3, 4, 5], 1024, (8, 8)),      # the adapter's tokens in the middle of a tile of 256
    ([1, 200, 180, 1, 140], [1, 1, 2, 2, 3], 4096, (3, 1)),                       # in both halves of one and the start of the next
    ([300, 5, 420], [0, 2, 4], 328, (3, 1)),
    ([700, 33, 900], [-1, 2, 3], 1024, (8, 2)),
    ([120, 1, 90, 1, 101], [-1, 1, 2, 3, 4], 328, (64, 8))])                      # tiles of 128 tokens
def test_long_batches(new_lens, lora, hidden, heads):
    check(new_lens, lora, hidden, heads, [16, 64, 33, 8, 24, 64])
