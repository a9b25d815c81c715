"""The natively marshalled calls of a layer step (csrc/native.cpp) without a GPU: what they refuse before the library sees it.  With a
null pool the library refuses the rest, so nothing is launched."""
import sys
import threading
import time

import pytest

from paper_2505_03756_b200 import binding as fl

WS = 0        # workspace and stream as raw addresses


@pytest.mark.parametrize("mats", [[], [0], [0, 1], [0, 1, 2, 3]])
def test_lists_of_unequal_length_are_refused(mats):
    ys = [4096, 8192, 12288]
    with pytest.raises(ValueError):
        fl.fl_lora_sgmv_multi(None, ys, 4096, mats, 4096, 4096, 1, 1, 1.0, WS, 0)
    with pytest.raises(ValueError):
        fl.fl_lora_linear_multi(None, ys, 4096, ys, mats, 4096, 4096, 1, 1, 1.0, WS, 0)
    with pytest.raises(ValueError):
        fl.fl_lora_linear_multi(None, ys, 4096, [4096] * len(mats), [0, 1, 2], 4096, 4096, 1, 1, 1.0, WS, 0)


def test_lists_of_equal_length_reach_the_library():
    for ys in ([4096], [4096, 8192, 12288], [4096] * 20):
        mats = list(range(len(ys)))
        with pytest.raises(fl.FlError):
            fl.fl_lora_sgmv_multi(None, ys, 4096, mats, 4096, 4096, 1, 1, 1.0, WS, 0)
        with pytest.raises(fl.FlError):
            fl.fl_lora_linear_multi(None, ys, 4096, ys, mats, 4096, 4096, 1, 1, 1.0, WS, 0)


def test_other_threads_run_during_a_call():
    """With a switch interval that never ends, a thread that waits for the interpreter's lock gets it only where a call gives it up."""
    gate, ran = threading.Lock(), []
    gate.acquire()

    def other():
        with gate:
            ran.append(True)

    t = threading.Thread(target=other, daemon=True)
    t.start()
    time.sleep(0.2)                          # it waits at the gate now
    old = sys.getswitchinterval()
    sys.setswitchinterval(1000.0)
    try:
        gate.release()
        end = time.monotonic() + 10.0
        while not ran and time.monotonic() < end:
            try:
                fl.fl_kv_append(None, 4096, 4096, 4096, 4096, 4096, 4096, 1, 1, 1, 0)
            except fl.FlError:
                pass
        got = bool(ran)
    finally:
        sys.setswitchinterval(old)
    t.join()
    assert got
