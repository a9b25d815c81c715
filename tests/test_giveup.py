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


@pytest.mark.parametrize("n_ctas", [2, 4, 8])
def test_a_sum_whose_parts_are_fetched_is_not_stored_without_one(tmp_path, n_ctas):
    """The tcgen05 shrink: a CTA leaves its part, or a word that it has none, in its own memory before the barrier; behind it each looks at
    every CTA's word, a lane each, and stores its share of the sum only if none is set.  Memory without a part holds old bytes."""
    run_model(tmp_path, """
int main() {
  const int n = %d;
  int wrong = 0;
  for (int failed = 0; failed < 1 << n; ++failed) {
    std::vector<int> missing(n, 0);
    std::vector<long> part(n, 1000000);
    for (int c = 0; c < n; ++c) {
      if (failed >> c & 1) missing[c] = 1;
      else part[c] = 1 << c;
    }
    for (int c = 0; c < n; ++c) {
      bool any = false;
      for (int lane = 0; lane < 32; ++lane) any |= (lane < n ? missing[lane] : 0) != 0;
      long sum = 0;
      for (long v : part) sum += v;
      const bool stores = giveup::may_store(true, any ? 1 : 0);
      if (stores && sum != (1 << n) - 1) { printf("CTA %%d of %%d stores %%ld with %%x failed\\n", c, n, sum, failed); ++wrong; }
      if (!stores && failed == 0) { printf("CTA %%d of %%d stores nothing\\n", c, n); ++wrong; }
    }
  }
  return wrong ? 1 : 0;
}
""" % n_ctas)


BARRIER = """
// A ring slot's barrier: a phase ends when its arrivals and its bytes have come.  A parity test is true for every phase but the
// current one of that parity, so also for the one before it.
struct Bar {
  int count = 1, left = 1, tx = 0, phase = 0;
  void step() { while (left == 0 && tx == 0) { ++phase; left = count; } }
  void arrive() { --left; step(); }
  void expect(int bytes) { tx += bytes; --left; step(); }
  void complete(int bytes) { tx -= bytes; step(); }
  bool test(unsigned parity) const { return (unsigned)(phase & 1) != parity; }
};
struct Copy { int slot, bytes, at; };        // lands at the at-th poll
struct Flight {
  std::vector<Copy> copies;
  int polls = 0;
  template <typename B> void poll(B& bars) {
    ++polls;
    for (Copy& c : copies) if (c.at == polls) bars[c.slot].complete(c.bytes);
  }
  int left() const { int n = 0; for (const Copy& c : copies) n += c.at > polls; return n; }
};
"""


@pytest.mark.parametrize("ns", [1, 2, 5, 12])
def test_the_drain_waits_for_the_last_armed_phase_of_every_slot(tmp_path, ns):
    """A producer stopped after any number of stages, the last ones' copies still on their way, in any order of landing."""
    run_model(tmp_path, BARRIER + """
int main() {
  const int ns = %d;
  int wrong = 0;
  for (int fills = 0; fills <= 4 * ns + 1; ++fills)
    for (int open = 0; open <= ns && open <= fills; ++open)
      for (int order = 0; order < 3; ++order) {
        std::vector<Bar> bars(ns);
        Flight fl;
        for (int f = 0; f < fills; ++f) {
          bars[f %% ns].expect(100);
          const int k = f - (fills - open);
          if (k < 0) bars[f %% ns].complete(100);
          else fl.copies.push_back({f %% ns, 100, 1 + (order == 0 ? 7 * k : order == 1 ? 7 * (open - k) : (k * 13) %% 29 + 3)});
        }
        const bool all = giveup::drain(fills, ns, [&](int s, uint32_t parity) { fl.poll(bars); return bars[s].test(parity); });
        if (!all || fl.left()) { printf("ring %%d, %%d stages, %%d open: %%d copies still on their way\\n", ns, fills, open, fl.left()); ++wrong; }
      }
  std::vector<Bar> bars(1);
  bars[0].expect(100);                       // nothing comes: the bound ends it
  if (giveup::drain(1, 1, [&](int, uint32_t parity) { return bars[0].test(parity); })) { printf("a copy that never comes\\n"); ++wrong; }
  return wrong ? 1 : 0;
}
""" % ns)


@pytest.mark.parametrize("ns", [1, 3, 5])
def test_a_pair_that_stopped_at_different_stages(tmp_path, ns):
    """The first CTA's barriers count both CTAs' halves.  Either may be ahead by up to a ring, and stages of both be open."""
    run_model(tmp_path, BARRIER + """
int main() {
  const int ns = %d;
  int wrong = 0;
  for (int done = 0; done <= 2 * ns + 1; ++done)         // stages both have brought and used
    for (int a = 0; a <= ns; ++a)                        // stages issued beyond them, by the first and by the second CTA
      for (int b = 0; b <= ns; ++b) {
        std::vector<Bar> bars(ns);
        Flight fl;
        for (int f = 0; f < done + a; ++f) {
          bars[f %% ns].expect(200);
          if (f < done) { bars[f %% ns].complete(100); bars[f %% ns].complete(100); }
          else fl.copies.push_back({f %% ns, 100, 1 + (f * 5) %% 17});
        }
        for (int f = done; f < done + b; ++f) fl.copies.push_back({f %% ns, 100, 1 + (f * 11) %% 23});
        const long long n = giveup::settle_pair(done + a, done + b, ns, [&](int s) { bars[s].expect(100); }, [&](int s) { bars[s].complete(100); });
        const bool all = giveup::drain(n, ns, [&](int s, uint32_t parity) { fl.poll(bars); return bars[s].test(parity); });
        if (!all || fl.left()) { printf("ring %%d, %%d stages, %%d and %%d open: %%d copies still on their way\\n", ns, done, a, b, fl.left()); ++wrong; }
      }
  return wrong ? 1 : 0;
}
""" % ns)


@pytest.mark.parametrize("ns", [2, 4])
def test_stages_that_copy_threads_signal_too(tmp_path, ns):
    """The tcgen05 shrink: a phase needs the producer's arrival with its bytes and every copy thread's.  Threads that stopped behind
    the producer make up for the last phase of a slot; threads that ran ahead of it owe nothing."""
    run_model(tmp_path, BARRIER + """
int main() {
  const int ns = %d, threads = 3;
  int wrong = 0;
  for (int used = 0; used <= 2 * ns; ++used)             // stages whose product is done: their slots may be armed again
    for (int ahead = 0; ahead <= ns; ++ahead)            // stages the producer has armed beyond them
      for (int mix = 0; mix < (ns + 1) * (ns + 1) * (ns + 1); ++mix) {
        std::vector<Bar> bars(ns);
        for (Bar& b : bars) b.count = b.left = 1 + threads;
        std::vector<long long> arrived(threads);
        Flight fl;
        const int fills = used + ahead;
        int m = mix;
        for (int t = 0; t < threads; ++t, m /= ns + 1) arrived[t] = used + m %% (ns + 1);
        for (int f = 0; f < used + ns; ++f) {
          Bar& b = bars[f %% ns];
          if (f < fills) b.expect(100);
          for (int t = 0; t < threads; ++t) if (f < arrived[t]) b.arrive();
          if (f < used) b.complete(100);
          else if (f < fills) fl.copies.push_back({f %% ns, 100, 1 + (f * 7) %% 19});
        }
        for (int t = 0; t < threads; ++t) for (; arrived[t] < fills; ++arrived[t]) bars[arrived[t] %% ns].arrive();
        const bool all = giveup::drain(fills, ns, [&](int s, uint32_t parity) { fl.poll(bars); return bars[s].test(parity); });
        if (!all || fl.left()) { printf("ring %%d, %%d used, %%d ahead, mix %%d: %%d copies\\n", ns, used, ahead, mix, fl.left()); ++wrong; }
      }
  return wrong ? 1 : 0;
}
""" % ns)
