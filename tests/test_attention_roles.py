"""The producer and the MMA issuers of the tcgen05 prefill attention kernel (csrc/attention_roles.cuh), run on the host against a model
of the barriers, the copies and the tensor pipe: copies may take any time and land in any order, as on a GPU."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_03756_b200", "csrc")

MODEL = r"""
#include <ucontext.h>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <memory>
#include <queue>
#include <vector>
#include "attention_roles.cuh"
#include "giveup.cuh"

// Fibers on a common clock: a role runs until it lets time pass.
struct Sim {
  struct Event { long at, seq; std::function<void()> run; };
  struct Later { bool operator()(const Event& a, const Event& b) const { return a.at != b.at ? a.at > b.at : a.seq > b.seq; } };
  std::priority_queue<Event, std::vector<Event>, Later> events;
  long now = 0, seq = 0;
  ucontext_t main_ctx;
  struct Fiber { ucontext_t ctx; std::vector<char> stack; std::function<void()> body; };
  std::vector<std::unique_ptr<Fiber>> fibers;
  Fiber* current = nullptr;
  static Sim* self;
  void at(long t, std::function<void()> f) { events.push({t, seq++, f}); }
  static void entry() { self->current->body(); swapcontext(&self->current->ctx, &self->main_ctx); }
  void resume(Fiber* f) { current = f; swapcontext(&main_ctx, &f->ctx); }
  void spawn(std::function<void()> body) {
    fibers.emplace_back(new Fiber);
    Fiber* f = fibers.back().get();
    f->stack.resize(1 << 16);
    f->body = body;
    getcontext(&f->ctx);
    f->ctx.uc_stack.ss_sp = f->stack.data();
    f->ctx.uc_stack.ss_size = f->stack.size();
    f->ctx.uc_link = nullptr;
    makecontext(&f->ctx, entry, 0);
    at(now, [this, f] { resume(f); });
  }
  void pass(long cycles) {
    Fiber* f = current;
    at(now + cycles, [this, f] { resume(f); });
    swapcontext(&f->ctx, &main_ctx);
  }
  void run() { self = this; while (!events.empty()) { Event e = events.top(); events.pop(); now = e.at; e.run(); } }
};
Sim* Sim::self = nullptr;

int wrong = 0;
const char* where = "";
void fault(const char* what, int slot, int want, int got) {
  if (wrong++ < 5) printf("%s: %s, slot %d, tile %d, found %d\n", where, what, slot, want, got);
}

// A phase ends when its arrivals and its bytes have come; a parity test is true for the phase before last too.
struct Bar {
  int count = 1, left = 1, tx = 0, phase = 0;
  void init(int n) { count = left = n; }
  void step() { while (left == 0 && tx == 0) { ++phase; left = count; } }
  void arrive() { if (left == 0) fault("an arrival beyond a phase's count", -1, phase, tx); else --left; step(); }
  void expect() { ++tx; arrive(); }
  void complete() { --tx; step(); }
  bool test(unsigned parity) const { return (unsigned)(phase & 1) != parity; }
};
struct Slot { int tile = -1, readers = 0, open = 0; };      // what has landed, MMAs under way on it, copies under way into it

struct Unit { int n[2]; };
constexpr long LIMIT = 60000, NEVER = 40 * LIMIT;

// One ring: K and V take turns, as the kernel had it once.  Own rings: the kernel's.
struct Shared5 : attn::RingPos<5> {
  Shared5 next() const { Shared5 r; static_cast<attn::RingPos<5>&>(r) = attn::RingPos<5>::next().next(); return r; }
};
struct Cta {
  Sim sim;
  std::vector<Slot> slots{5};           // K's, then V's; or the one ring
  std::vector<Bar> full{5}, empty{5};
  Slot q;
  Bar q_full, q_empty, s_full[2], s_free, p_half[2], p_full[2], pv_done[2];
  bool abort = false;
  std::function<long(bool is_v, int tile)> latency;
  long pipe_free = 0;
  int fills[2] = {0, 0};                // K's and V's
  bool wait(const Bar& b, unsigned parity) {
    const long from = sim.now;
    for (sim.pass(150);; sim.pass(20)) {
      if (b.test(parity)) return true;
      if (abort) return false;
      if (sim.now - from > LIMIT) { abort = true; return false; }
    }
  }
  void load(int s, bool is_v, int tile) {
    Slot& sl = slots[s];
    if (sl.readers) fault("a copy into a slot under an MMA", s, tile, sl.tile);
    if (sl.open) fault("a copy into a slot whose copy has not landed", s, tile, sl.tile);
    sl.tile = -1;
    ++sl.open;
    full[s].expect();
    ++fills[is_v];
    sim.at(sim.now + latency(is_v, tile), [this, s, tile] { slots[s].tile = tile; --slots[s].open; full[s].complete(); });
  }
  // an MMA group of one thread: the pipe takes them in the order of issue; done_at is when the thread's last one is complete
  void mma(int s, int want, long cycles, long& done_at) {
    sim.pass(60);
    Slot& sl = slots[s];
    if (sl.tile != want) fault("an MMA on a slot that does not hold its tile", s, want, sl.tile);
    ++sl.readers;
    pipe_free = std::max(pipe_free, sim.now) + cycles;
    done_at = pipe_free;
    sim.at(pipe_free, [this, s] { --slots[s].readers; });
  }
  void commit(Bar& b, long done_at) { sim.pass(10); sim.at(std::max(sim.now, done_at), [&b] { b.arrive(); }); }
};

// Runs a CTA's units; v0 is where V's slots start and its first position is v_first.
template <typename KPos, typename VPos>
void run_cta(Cta& c, const std::vector<Unit>& units, VPos v_first, int v0, int k_empty, int v_empty, int softmax) {
  for (int s = 0; s < 5; ++s) c.empty[s].init(v0 && s < v0 ? k_empty : v_empty);
  c.s_free.init(1);
  Sim& sim = c.sim;
  auto steps = [](const Unit& u) { return std::max(u.n[0], u.n[1]); };
  sim.spawn([&] {                         // producer
    KPos k;
    VPos v = v_first;
    int tile_k = 0, tile_v = 0, n = 0;
    for (const Unit& u : units) {
      if (n > 0 && !c.wait(c.q_empty, (n - 1) & 1)) return;
      ++n;
      c.q_full.expect();
      sim.at(sim.now + 1500, [&] { c.q_full.complete(); });
      if (!attn::load_tiles(steps(u), k, v, [&](int) { sim.pass(100); },
                            [&](KPos p) { if (!c.wait(c.empty[p.s], p.ph ^ 1u)) return false; c.load(p.s, false, tile_k++); return true; },
                            [&](VPos p) { if (!c.wait(c.empty[v0 + p.s], p.ph ^ 1u)) return false; c.load(v0 + p.s, true, 1000000 + tile_v++); return true; })) return;
    }
  });
  sim.spawn([&] {                         // issuer of the scores
    KPos k;
    unsigned ph_free = 1, ph_q = 0;
    long done = 0;
    int base = 0;
    for (const Unit& u : units) {
      const bool ok = c.wait(c.q_full, ph_q);
      ph_q ^= 1u;
      int at = base;
      if (!ok || !attn::issue_scores(steps(u), u.n[0], u.n[1], k, ph_free, [&](KPos p) { return c.wait(c.full[p.s], p.ph); },
                                     [&](unsigned ph) { return c.wait(c.s_free, ph); },
                                     [&](int x, KPos p) { c.mma(p.s, at, 512, done); c.commit(c.s_full[x], done); },
                                     [&](KPos p) { ++at; for (int i = 0; i < k_empty; ++i) c.commit(c.empty[p.s], done); }, [&] { c.commit(c.q_empty, done); })) return;
      base += steps(u);
    }
  });
  for (int x = 0; x < 2; ++x) {
    sim.spawn([&, x] {                    // issuer of P V
      VPos v = v_first;
      unsigned ph_p = 0;
      long done = 0;
      int at = 1000000;
      for (const Unit& u : units)
        if (!attn::issue_pv(steps(u), u.n[x], v, ph_p, [&](VPos p) { return c.wait(c.full[v0 + p.s], p.ph); },
                            [&](int half, unsigned ph) { return c.wait(half ? c.p_full[x] : c.p_half[x], ph); },
                            [&](int, VPos p, bool) { c.mma(v0 + p.s, at, 256, done); }, [&] { c.commit(c.pv_done[x], done); },
                            [&](VPos p) { ++at; c.commit(c.empty[v0 + p.s], done); })) return;
    });
    sim.spawn([&, x] {                    // softmax
      int n = 0;
      for (const Unit& u : units) {
        for (int j = 0; j < u.n[x]; ++j, ++n) {
          if (!c.wait(c.s_full[x], n & 1)) return;
          sim.pass(200);
          c.s_free.arrive();
          sim.pass(softmax / 4);
          if (j > 0 && !c.wait(c.pv_done[x], (n - 1) & 1)) return;
          sim.pass(softmax / 2);
          c.p_half[x].arrive();
          sim.pass(softmax / 4);
          c.p_full[x].arrive();
        }
        if (u.n[x] > 0) {
          if (!c.wait(c.pv_done[x], (n - 1) & 1)) return;
          sim.pass(2000);
        }
      }
    });
  }
  sim.run();
}

void own_rings(Cta& c, const std::vector<Unit>& units, int softmax) {
  run_cta<attn::RingPos<attn::K_SLOTS>, attn::RingPos<attn::V_SLOTS>>(c, units, {}, attn::K_SLOTS, 1, 2, softmax);
}
void one_ring(Cta& c, const std::vector<Unit>& units, int softmax) {
  Shared5 v;
  v.s = 1;
  run_cta<Shared5, Shared5>(c, units, v, 0, 2, 2, softmax);
}

// Copies: all alike, one that is late, a slow start, any of four times at random.
std::function<long(bool, int)> latencies(int mode) {
  if (mode < 4) return [=](bool, int) { return (long[]){300, 900, 1500, 4000}[mode]; };
  if (mode < 16) return [=](bool v, int t) { return !v && t == mode - 4 ? 4000L : 900L; };
  if (mode < 28) return [=](bool v, int t) { return v && t == 1000000 + mode - 16 ? 4000L : 900L; };
  if (mode < 32) return [=](bool v, int t) { return !v && t < mode - 27 ? 2000L : 900L; };
  return [=](bool v, int t) { unsigned h = (unsigned)(t * 2 + v) * 2654435761u + (unsigned)mode * 40503u; h ^= h >> 15; h *= 2246822519u; h ^= h >> 13; return (long[]){700, 900, 1100, 2000}[h & 3]; };
}
const int MODES = 72;

template <typename Run>
int all_units(Run run) {
  int runs = 0;
  static char text[128];
  for (int a : {1, 2, 3, 4, 5, 6, 8, 12})
    for (int b : {0, a, a + 1})
      for (int next = 0; next < 3; ++next)
        for (int mode = 0; mode < MODES; ++mode) {
          std::vector<Unit> units{{{a, b}}};
          if (next) units.push_back(next == 1 ? Unit{{3, 0}} : Unit{{2, 3}});
          snprintf(text, sizeof(text), "%d and %d key tiles, %zu units, copies %d", a, b, units.size(), mode);
          where = text;
          Cta c;
          c.latency = latencies(mode);
          run(c, units, mode % 3 == 0 ? 400 : 1800);
          if (c.abort) fault("a wait that ran out", 0, 0, 0);
          ++runs;
        }
  return runs;
}
"""


def run_model(tmp_path, main):
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(MODEL + main)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-Wno-unknown-pragmas", "-Wno-unused-function", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


def test_tiles_are_there_when_they_are_read_and_stay_until_they_have_been(tmp_path):
    """Units of one and two query tiles, one to twelve key tiles, alone and with another unit behind them, and any copy late."""
    run_model(tmp_path, """
int main() { all_units(own_rings); return wrong ? 1 : 0; }
""")


def test_nothing_is_given_back_behind_a_wait_that_gave_up(tmp_path):
    """Any one copy, of K or of V, that lands long after the waits' limit: the slots whose copies are on their way are not armed again, so
    that the drain behind the abort waits for every copy."""
    run_model(tmp_path, """
int main() {
  static char text[128];
  for (int b : {0, 1, 9})
    for (int late = 0; late < 28; ++late)
      for (int more = 0; more < 3; ++more) {              // the copies behind it: on time, as late, or a little late
        snprintf(text, sizeof(text), "late copy %d, second tile %d, more %d", late, b, more);
        where = text;
        Cta c;
        c.latency = [=](bool v, int t) {
          const int n = 2 * (v ? t - 1000000 : t) + v;
          return n == late ? NEVER : n > late && more == 1 ? NEVER + 37 * n : n > late && more == 2 ? LIMIT + 37 * n : 900;
        };
        own_rings(c, {{{9, b}}, {{5, 0}}}, 1800);         // ends when all events are over: the copies too
        if (!c.abort) fault("the late copy was not missed", 0, late, 0);
      }
  for (int late = 0; late < 28; ++late) {                 // and what the drain sees when it starts at once
    Cta c;
    where = "drain";
    c.latency = [=](bool v, int t) { return 2 * (v ? t - 1000000 : t) + v == late ? 3 * LIMIT : 900; };
    bool stopped = false;
    std::function<void()> watch = [&] {
      if (!c.abort) { c.sim.at(c.sim.now + 1000, watch); return; }
      if (!stopped) { stopped = true; c.sim.at(c.sim.now + 1000, watch); return; }       // every role has left
      c.sim.spawn([&] {
        auto drain = [&](int first, int n, int fills) {
          giveup::drain(fills, n, [&](int s, uint32_t parity) { c.sim.pass(20); return c.full[first + s].test(parity); });
        };
        drain(0, attn::K_SLOTS, c.fills[0]);
        drain(attn::K_SLOTS, attn::V_SLOTS, c.fills[1]);
        for (int s = 0; s < 5; ++s)
          if (c.slots[s].open) fault("drained beside a copy on its way", s, late, c.slots[s].open);
      });
    };
    c.sim.at(0, watch);
    own_rings(c, {{{9, 9}}, {{5, 0}}}, 1800);
  }
  return wrong ? 1 : 0;
}
""")


def test_the_model_sees_the_fault_of_one_ring_for_both(tmp_path):
    """With K and V in turns in a ring of five slots, units of one query tile go wrong where copies are late, and the others do not."""
    run_model(tmp_path, """
int main() {
  int lone = 0, pairs = 0;
  all_units([&](Cta& c, const std::vector<Unit>& units, int softmax) {
    const int before = wrong;
    one_ring(c, units, softmax);
    bool alone = false;
    for (const Unit& u : units) alone |= u.n[0] == 0 || u.n[1] == 0;
    (alone ? lone : pairs) += wrong > before || c.abort;
    c.abort = false;
  });
  printf("%d runs of lone tiles, %d of pairs\\n", lone, pairs);
  return lone > 0 && pairs == 0 ? 0 : 1;
}
""")


def test_a_softmax_warp_stores_as_one_and_behind_a_fence(tmp_path):
    """32 lanes that look at the barrier of the step before one after the other, while its phase ends at any time, and go on to an
    aligned store: they take one way to it, behind the phase's end and behind a fence that follows their last look.  The model sees it
    when the lanes do not vote, or do not fence."""
    run_model(tmp_path, """
enum { VOTES = 1, FENCES = 2 };
struct Meet { int here = 0; bool all = true; };
int faults(int with) {
  int bad = 0;
  for (int end = 1; end < 400; end += 3) {
    Sim sim;
    Bar pv;
    Meet votes[2];
    int waited = 0, stored = 0;
    sim.at(end, [&] { pv.arrive(); });
    for (int lane = 0; lane < 32; ++lane)
      sim.spawn([&, lane] {
        bool fenced = false;
        int round = 0;
        auto vote = [&](bool v) {
          if (!(with & VOTES)) return v;
          Meet& m = votes[round++];
          m.all &= v;
          for (++m.here; m.here < 32;) sim.pass(1);
          return m.all;
        };
        auto fence = [&] { fenced = (with & FENCES) != 0; };
        sim.pass(1 + lane);                     // the lanes' looks are not at one time
        bool done = attn::seen_by_all([&] { fenced = false; return pv.test(0); }, vote, fence);
        sim.pass(100);
        if (!done) {
          ++waited;
          done = attn::seen_by_all([&] { fenced = false; while (!pv.test(0)) sim.pass(1 + lane % 3); return true; }, vote, fence);
        }
        ++stored;
        bad += !done || !fenced || !pv.test(0);
      });
    sim.run();
    bad += stored != 32 || (waited != 0 && waited != 32);
  }
  return bad;
}
int main() {
  const int good = faults(VOTES | FENCES), lone = faults(FENCES), open = faults(VOTES);
  printf("%d faults, %d without the vote, %d without the fence\\n", good, lone, open);
  return good == 0 && lone > 0 && open > 0 ? 0 : 1;
}
""")
