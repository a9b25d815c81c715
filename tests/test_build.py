"""When the module that is built against torch counts as out of date."""
import os

from paper_2505_03756_b200 import build as b

SRC = os.path.join(b.CSRC, "native.cpp")


def test_native_module_is_rebuilt_for_another_torch_or_python(monkeypatch):
    b.build()
    assert not b._native_stale(SRC)
    tag = b._native_tag()
    for other in (tag + "1", tag[:-1], tag.replace("python 3.", "python 4.")):
        monkeypatch.setattr(b, "_native_tag", lambda: other)
        assert b._native_stale(SRC), other
