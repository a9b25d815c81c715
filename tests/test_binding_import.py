"""The functions that work on host data alone need neither torch nor the module that is built against it."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
sys.modules["torch"] = None                                  # any import of it raises
sys.modules["paper_2505_03756_b200._native"] = None
from paper_2505_03756_b200 import binding as fl
tree = fl.fl_tree_create(16)
assert fl.fl_tree_size(tree) >= 0
fl.fl_tree_destroy(tree)
assert fl.fl_lora_blocks(1 << 20, 16, [(4096, 4096)]) > 0
try:
    fl.fl_kv_append(None, 1, 1, 1, 1, 1, 1, 1, 1, 1, 0)
except ImportError:
    print("as expected")
"""


def test_host_functions_without_torch():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "as expected" in r.stdout, r.stderr
