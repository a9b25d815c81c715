"""fl_paged_attention of prompts with up to 128 new tokens behind long cached prefixes: units of one query tile, whose K and V tiles come
from HBM (the pool is larger than L2, which is flushed as well), the same bits each time, alone and beside decode steps (where K and V in
one ring gave other bits about once in 350 passes)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.attention import attend_request
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_context


@pytest.mark.parametrize("heads,prefix,new,passes", [
    ((32, 32), [2000] * 6 + [0, 333], [100] * 6 + [128, 65], 30), ((24, 8), [2900, 500, 1600], [97, 300, 384], 30),
    ((32, 32), [3000, 700, 2100, 1500, 448, 96, 320], [1, 1, 1, 1, 450, 101, 333], 400)])
def test_lone_tiles_behind_long_prefixes(heads, prefix, new, passes):
    from paper_2505_03756_b200 import harness as H
    wl = synth.make_workload("tiny", n_req=len(new), len_range=(0, 0), n_adapters=1, shape=synth.LayerShape(heads[0] * 128, *heads))
    wl.prefix_lens[:], wl.new_lens[:] = prefix, new
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 64
    s = H.Session(wl, adapters=[])
    try:
        s.build_batch()
        s.fill_prefix_kv()
        k_new, v_new = wl.kv_new()
        s.kv_append(H.f32_to_dev(k_new, s.dev), H.f32_to_dev(v_new, s.dev))
        q = wl.q()
        tq = H.f32_to_dev(q, s.dev)
        flush = torch.empty(256 << 20, dtype=torch.uint8, device=s.dev)
        first = None
        for n in range(passes):
            out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device=s.dev)
            if n % 3 == 0:
                flush.fill_(n % 128)
            s.attention(out, tq)
            first = out if first is None else first
            assert torch.equal(out, first)
        got = H.dev_to_f32(first)
        for i in (0, wl.n_req - 2, wl.n_req - 1):
            lo, hi = int(wl.req_indptr[i]), int(wl.req_indptr[i + 1])
            k, v = oracle_context(wl, i, k_new, v_new)
            assert_close(got[lo:hi], attend_request(q[lo:hi], k, v, prefix[i], 1.0 / math.sqrt(128)), f"lone tiles {heads} request {i}")
        assert s.status()["device_flags"] == 0
    finally:
        s.close()
