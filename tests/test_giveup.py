"""What the kernels do when a bounded wait has given up (csrc/giveup.cuh), run on the host against a model of what they wait for: no
GPU wait has to run out for it."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_03756_b200", "csrc")


def run_model(tmp_path, source):
    """Compiles a host program around giveup.cuh and runs it; the program prints what it found wrong and counts it."""
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text("#include <cstdio>\n#include <vector>\n#include \"giveup.cuh\"\n" + source)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("n_ctas", [1, 2, 3, 8])
def test_a_sum_that_lacks_a_part_is_not_stored(tmp_path, n_ctas):
    """Every set of CTAs of a cluster whose wait gave up: before the barrier each tells the others or sends its part, behind it
    each stores or does not.  Memory that was never sent holds old bytes, here a large number."""
    run_model(tmp_path, """
int main() {
  const int n = %d;
  int wrong = 0;
  for (int failed = 0; failed < 1 << n; ++failed) {
    std::vector<int> told(n, 0);
    std::vector<std::vector<long>> part(n, std::vector<long>(n, 1000000));
    for (int c = 0; c < n; ++c) {
      const bool ok = !(failed >> c & 1);
      giveup::tell_cluster(ok, c, n, [&](int p) { told[p] = 1; });
      for (int p = 0; p < n && ok; ++p) part[p][c] = 1 << c;
    }
    for (int c = 0; c < n; ++c) {
      const bool stores = giveup::may_store(!(failed >> c & 1), told[c]);
      long sum = 0;
      for (long v : part[c]) sum += v;
      if (stores && sum != (1 << n) - 1) { printf("CTA %%d of %%d stores %%ld with %%x failed\\n", c, n, sum, failed); ++wrong; }
      if (!stores && failed == 0) { printf("CTA %%d of %%d stores nothing\\n", c, n); ++wrong; }
    }
  }
  return wrong ? 1 : 0;
}
""" % n_ctas)
