"""fl_paged_attention on batches with both kinds of work, whose decode kernel runs beside the persistent prefill kernel: shares of
one SM to all of them (a few long units beside many decode pages, one decode request beside many units), and a projection
right behind the call that reads both kernels' rows."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.attention import attend_request
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_context


@pytest.mark.parametrize("heads", [(4, 4), (8, 2)])
@pytest.mark.parametrize("prefix,new", [
    ([0, 1300], [600, 1]),                                  # long units, one decode request that ends long before them
    ([900] * 24 + [0], [1] * 24 + [17]),                    # one short unit per head beside a batch of decode steps
    ([2500] * 6 + [130, 0, 64], [1] * 6 + [700, 257, 129]),
    ([40] + [300] * 12, [1] + [130] * 12)])
def test_decode_beside_prefill(heads, prefix, new):
    from paper_2505_03756_b200 import harness as H
    wl = synth.make_workload("tiny", n_req=len(new), len_range=(0, 0), n_adapters=2, shape=synth.LayerShape(heads[0] * 128, *heads))
    wl.prefix_lens[:], wl.new_lens[:] = prefix, new
    wl.ranks[:] = 16
    wl.lora_of_req[:] = np.arange(len(new)) % 2
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 400
    s = H.Session(wl)
    try:
        s.load_adapters()
        s.build_batch()
        s.fill_prefix_kv()
        k_new, v_new = wl.kv_new()
        s.kv_append(H.f32_to_dev(k_new, s.dev), H.f32_to_dev(v_new, s.dev))
        q = wl.q()
        tq = H.f32_to_dev(q, s.dev)
        out = torch.empty(q.shape, dtype=torch.bfloat16, device=s.dev)
        y0 = H.f32_to_dev(wl.y_base("o"), s.dev)
        first = None
        for _ in range(20):
            out.fill_(float("nan"))
            y = y0.clone()
            s.attention(out, tq)
            s.sgmv([y], out, ["o"])                         # starts as soon as the call before it allows it
            torch.cuda.synchronize()
            if first is None:
                first = out.clone(), y.clone()
                got = H.dev_to_f32(out)
                for i in range(wl.n_req):
                    lo, hi = int(wl.req_indptr[i]), int(wl.req_indptr[i + 1])
                    k, v = oracle_context(wl, i, k_new, v_new)
                    assert_close(got[lo:hi], attend_request(q[lo:hi], k, v, prefix[i], 1.0 / math.sqrt(128)), f"mixed {heads} request {i}")
            assert torch.equal(out, first[0]) and torch.equal(y, first[1])
        assert s.status()["device_flags"] == 0
    finally:
        s.close()
