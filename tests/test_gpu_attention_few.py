"""fl_paged_attention of a few decode requests, served without a plan: contexts of one key to more than a page for every warp of
a cluster, clusters with CTAs that have no page, several new tokens, grouped heads, requests without a new token, a request whose
table is too short next to good ones."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.attention import attend_request
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_context


@pytest.mark.parametrize("heads,prefix,new", [
    ((4, 4), [0], [1]), ((4, 4), [15], [1]), ((4, 4), [16, 600], [1, 0]), ((2, 2), [63, 64, 65], [1, 1, 1]), ((4, 4), [40, 0], [9, 7]),
    ((8, 8), [2600], [1]), ((8, 2), [1000, 17], [1, 3]), ((8, 1), [130, 131], [1, 1]), ((16, 16), [100 + 7 * i for i in range(16)], [1] * 16),
    ((1, 1), [511, 0, 5], [3, 12, 1]), ((4, 4), [5 * i for i in range(40)], [1] * 40), ((8, 1), [700, 3, 0, 90, 16], [1, 1, 1, 2, 0]),
    ((2, 2), [30, 9] + [7] * 30, [25, 6] + [0] * 30), ((16, 2), [2000, 31, 600], [1, 1, 1]),
    # one or a few requests hold most of the pages: a request gets one, two or four CTAs, the short ones share a cluster
    ((4, 4), [4000] + [5] * 11, [1] * 12), ((16, 16), [1200, 10, 700, 31, 300] + [9] * 11, [1] * 16), ((4, 4), [2] * 39 + [2600], [1] * 40),
    ((16, 16), [383, 384, 767, 768, 1200] + [1] * 11, [1] * 16), ((32, 32), [767, 768, 1535, 1536] + [1] * 4, [1] * 8), ((8, 1), [4300, 3, 40, 700] + [3] * 11 + [20], [1, 1, 2, 1] + [0] * 11 + [1]),
    ((4, 4), [1900, 40] + [8] * 34 + [530], [2, 1] + [0, 1] * 17 + [3])])
def test_few_decode_requests(heads, prefix, new):
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
        first = None
        for _ in range(3):
            out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device=s.dev)
            s.attention(out, tq)
            first = out if first is None else first
            assert torch.equal(out, first)
        got = H.dev_to_f32(first)
        for i in range(wl.n_req):
            lo, hi = int(wl.req_indptr[i]), int(wl.req_indptr[i + 1])
            k, v = oracle_context(wl, i, k_new, v_new)
            assert_close(got[lo:hi], attend_request(q[lo:hi], k, v, prefix[i], 1.0 / math.sqrt(128)), f"few {heads} request {i}")
        assert s.status()["device_flags"] == 0
        if len(new) > 1 and prefix[-1] > 0 and new[-1] > 0:      # the last request's keys now end behind its table
            s.t_prefix[-1] += 4096
            out = torch.full(q.shape, 3.0, dtype=torch.bfloat16, device=s.dev)
            s.attention(out, tq)
            torch.cuda.synchronize()
            n = int(wl.req_indptr[-2])
            assert torch.equal(out[:n], first[:n]) and bool((out[n:] == 3.0).all())
            assert s.status(clear=True)["device_flags"] != 0
    finally:
        s.close()


def test_tables_longer_than_the_contexts():
    """Blocks allocated ahead: the tables have more entries than the batch's contexts need, and n_tbl counts those in use."""
    from paper_2505_03756_b200 import harness as H
    wl = synth.make_workload("tiny", n_req=5, len_range=(0, 0), n_adapters=1, shape=synth.LayerShape(512, 4, 4))
    wl.prefix_lens[:], wl.new_lens[:] = [100, 17, 300, 40, 15], [1, 1, 1, 1, 1]
    used = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16))
    wl.pool_blocks = used + 64
    s = H.Session(wl, adapters=[])
    try:
        s.build_batch()
        s.fill_prefix_kv()
        k_new, v_new = wl.kv_new()
        s.kv_append(H.f32_to_dev(k_new, s.dev), H.f32_to_dev(v_new, s.dev))
        q = H.f32_to_dev(wl.q(), s.dev)
        want = torch.empty(q.shape, dtype=torch.bfloat16, device=s.dev)
        s.attention(want, q)
        long_tables = [np.concatenate([t, s.alloc(7)]) for t in s.kv_tables]
        s.t_tbl_indptr = torch.from_numpy(np.cumsum([0] + [len(t) for t in long_tables]).astype(np.int32)).to(s.dev)
        s.t_tbl = torch.from_numpy(np.concatenate(long_tables).astype(np.uint32).view(np.int32)).to(s.dev)
        assert s.n_tbl == used
        out = torch.full_like(want, float("nan"))
        s.attention(out, q)
        assert torch.equal(out, want)
        assert s.status()["device_flags"] == 0
    finally:
        s.close()
