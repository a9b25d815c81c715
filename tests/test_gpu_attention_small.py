"""fl_paged_attention of small batches, served by one kernel without a plan: new tokens around a tile's 64 rows and a warp's 16,
contexts around 64 keys, requests without a new token, one-token requests among prompts, more than 32 requests, grouped heads, a
request whose table is too short, one long context among many short ones, and batches on either side of each line to the planned kernels."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.attention import attend_request
from paper_2505_03756_b200 import synth

from _util import assert_close, oracle_context


def without_plan(heads, prefix, new):
    """The rule of attention.cu: CTAs of three rounds, eight blocks a request, 40 for one if the others have one each."""
    tables = [-(-(p + n) // 16) for p, n in zip(prefix, new)]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return (sum(new) // 64 + len(new)) * heads[0] <= 6 * sms and sum(tables) <= 8 * len(new) and sum(tables) - len(new) < 40

@pytest.mark.parametrize("heads,prefix,new", [
    ((4, 4), [0], [64]), ((4, 4), [0], [65]), ((8, 8), [32] * 4, [32] * 4), ((2, 2), [0, 63, 1, 15], [63, 1, 17, 128]),
    ((8, 2), [64, 0, 16], [64, 16, 33]), ((8, 1), [17, 40], [19, 3]), ((4, 4), [0, 5, 0, 30], [127, 0, 1, 18]),
    ((2, 1), [7 * (i % 9) for i in range(40)], [1 + 5 * (i % 7) for i in range(40)]), ((4, 4), [300] + [0] * 9, [30] + [16] * 9),
    ((16, 16), [60], [68]), ((16, 16), [61], [68]), ((32, 32), [16] * 13, [64] * 13), ((32, 32), [16] * 14, [64] * 14)])
def test_small_batch(heads, prefix, new):
    check_batch(heads, prefix, new)


@pytest.mark.parametrize("heads,prefix,new,alone", [
    ((2, 1), [7 * (i % 3) for i in range(40)], [0 if 30 <= i < 34 else 1 + 3 * (i % 5) for i in range(40)], True),      # the 33rd request and on
    ((4, 4), [0] * 33, [16] * 32 + [150], True), ((2, 2), [0] * 70, [3] * 40 + [0] * 28 + [65, 7], True),
    ((32, 32), [0] * 15, [48] * 15, True), ((32, 32), [0] * 16, [48] * 16, False),                                       # the grid's line
    ((4, 4), [20] * 3, [108] * 3, True), ((4, 4), [20] * 3, [108, 108, 109], False),                                     # eight blocks each
    ((4, 4), [0] * 99 + [623], [16] * 99 + [17], True), ((4, 4), [0] * 99 + [640], [16] * 99 + [1], False)])             # the longest one's
def test_the_lines_to_the_planned_kernels(heads, prefix, new, alone):
    assert without_plan(heads, prefix, new) == alone
    check_batch(heads, prefix, new)


def check_batch(heads, prefix, new):
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
        out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device=s.dev)
        s.attention(out, tq)
        got = H.dev_to_f32(out)
        for i in range(wl.n_req):
            lo, hi = int(wl.req_indptr[i]), int(wl.req_indptr[i + 1])
            k, v = oracle_context(wl, i, k_new, v_new)
            assert_close(got[lo:hi], attend_request(q[lo:hi], k, v, prefix[i], 1.0 / math.sqrt(128)), f"small {heads} request {i}")
        assert s.status()["device_flags"] == 0
        if len(new) > 1 and new[-1] > 0:                         # the last request's keys now end behind its table
            s.t_prefix[-1] += 4096
            bad = torch.full(q.shape, 3.0, dtype=torch.bfloat16, device=s.dev)
            s.attention(bad, tq)
            torch.cuda.synchronize()
            n = int(wl.req_indptr[-2])
            assert torch.equal(bad[:n], out[:n]) and bool((bad[n:] == 3.0).all())
            assert s.status(clear=True)["device_flags"] != 0
    finally:
        s.close()


@pytest.mark.parametrize("prefix,new,n_tokens,n_tbl", [
    ([0, 0, 0, 0], [200, 8, 8, 8], 100, None),               # four tiles where n_tokens leaves room for two: one kernel without a plan
    ([0], [128], 40, None), ([0] * 40, [8] * 39 + [300], 255, None),
    ([0, 0], [2000, 8], 100, None),                          # the planned kernels
    ([0, 399], [17, 1], 18, 8), ([600, 399, 399], [700, 1, 1], 702, 25)])      # decode contexts that n_tbl does not cover, without and with a plan
def test_sizes_that_are_too_small_raise_the_status(prefix, new, n_tokens, n_tbl):
    """Too few tokens or table entries named in the call; q, out and the tables hold all the rows that the requests have."""
    from paper_2505_03756_b200 import binding as fl, harness as H
    wl = synth.make_workload("tiny", n_req=len(new), len_range=(0, 0), n_adapters=1, shape=synth.LayerShape(512, 4, 4))
    wl.prefix_lens[:], wl.new_lens[:] = prefix, new
    wl.pool_blocks = int(np.sum((wl.prefix_lens + wl.new_lens + 15) // 16)) + 64
    s = H.Session(wl, adapters=[])
    try:
        s.build_batch()
        s.fill_prefix_kv()
        k_new, v_new = wl.kv_new()
        s.kv_append(H.f32_to_dev(k_new, s.dev), H.f32_to_dev(v_new, s.dev))
        q = H.f32_to_dev(wl.q(), s.dev)
        out = torch.zeros_like(q)
        for tokens, tbl, bad in ((wl.n_tokens, s.n_tbl, False), (n_tokens, s.n_tbl if n_tbl is None else n_tbl, True)):
            ws = torch.empty(fl.fl_paged_attention_workspace(wl.n_req, wl.n_tokens, s.n_tbl, 4, 4), dtype=torch.uint8, device=s.dev)
            fl.fl_paged_attention(s.pool, out, q, s.t_req_indptr, s.t_tbl_indptr, s.t_tbl, s.t_prefix, s.t_new, wl.n_req, tokens, tbl, 4, 4, 0.1, ws)
            torch.cuda.synchronize()
            assert (s.status(clear=True)["device_flags"] != 0) == bad
    finally:
        s.close()
