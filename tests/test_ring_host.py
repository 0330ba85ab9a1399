"""The hand-over of the contraction's tile stages (csrc/ring.h), on the host: a producer and a
consumer thread run the header's rules against a model of the barriers (phases, pending
arrivals, bytes in flight) in which copies land late and any wait may give up, taking turns at
random.  Checked in every trial, whether or not a wait gave up: "full" is armed once a phase, no
copy starts while another fills its stage or its products read it, a stage is read only after its
copies have landed, none is in use once the producer has closed the ring, and none in flight
after the drain.  Two planted mistakes, a consumer that
gives stages back after a wait that gave up and a producer that does not drain, are found by
the same checks."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r'''
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <random>
#include <thread>
#include <vector>
#include "ring.h"

struct Bar {                       // mbarrier of arrival count 1
  int pending = 1, tx = 0;
  unsigned phase = 0;              // parity of the phase in progress
  void settle() { if (pending == 0 && tx == 0) { pending = 1; phase ^= 1; } }
  bool done(unsigned parity) const { return phase != (parity & 1); }
};

// One thread runs at a time; at each poll the turn passes to a random other role.
struct Model {
  std::mutex m;
  std::condition_variable cv;
  std::mt19937 rng;
  int turn = 0, alive = 2;
  bool over[2] = {false, false};
  int n;
  std::vector<Bar> full, empty;
  std::vector<int> copying, reading;
  bool abort_flag = false;
  const char* bad = nullptr;
  Model(int n, unsigned seed) : rng(seed), n(n), full(n), empty(n), copying(n, 0), reading(n, 0) {}
  void fault(const char* w) { if (!bad) bad = w; }
  void hardware() {                // at most one copy lands, one stage's products complete
    const int s = rng() % n;
    if (copying[s] && rng() % 4 == 0) {
      --copying[s];
      full[s].tx -= 1;
      full[s].settle();
    }
    const int q = rng() % n;
    if (reading[q] && rng() % 3 == 0) {
      --reading[q];
      if (empty[q].pending == 0) fault("empty arrived at twice in a phase");
      empty[q].pending -= 1;
      empty[q].settle();
    }
  }
  void step(int me) {              // let the others run
    std::unique_lock<std::mutex> l(m);
    hardware();
    if (!over[1 - me] && rng() % 2) {
      turn = 1 - me;
      cv.notify_all();
      cv.wait(l, [&] { return turn == me; });
    }
  }
  void begin(int me) {
    std::unique_lock<std::mutex> l(m);
    cv.wait(l, [&] { return turn == me; });
  }
  void end(int me) {
    std::unique_lock<std::mutex> l(m);
    over[me] = true;
    turn = 1 - me;
    cv.notify_all();
  }
  bool wait(int me, Bar& b, unsigned parity, int limit, bool look) {
    for (int i = 0; i < limit; ++i) {
      if (b.done(parity)) return true;
      if (look && abort_flag) return false;
      step(me);
    }
    abort_flag = true;
    return false;
  }
};

// plant: 0 none, 1 the consumer gives back and waits one poll after a wait that gave up, 2 no drain
static const char* trial(int n, int iters, int polls_p, int polls_c, unsigned seed, int plant) {
  Model w(n, seed);
  int filled = 0;
  std::thread prod([&] {
    w.begin(0);
    filled = prd::ring_produce(
        iters, n, [&](int s, unsigned par) { return w.wait(0, w.empty[s], par, polls_p, true); },
        [&](int s) {
          if (w.full[s].pending == 0) w.fault("full armed twice in a phase");
          w.full[s].pending -= 1;
          w.full[s].tx += 1;
          if (w.copying[s]) w.fault("copy into a stage that a copy is filling");
          if (w.reading[s]) w.fault("copy into a stage that is being read");
          w.copying[s] += 1;
          w.step(0);
        });
    // the ring's memory may be laid out anew
    if (filled == iters &&
        prd::ring_close(iters, n, [&](int s, unsigned par) { return w.wait(0, w.empty[s], par, polls_p, true); }))
      for (int s = 0; s < n; ++s)
        if (w.copying[s] || w.reading[s]) w.fault("ring closed with a stage in use");
    w.end(0);
  });
  std::thread cons([&] {
    w.begin(1);
    prd::RingPos pos;
    int limit = polls_c;
    for (int i = 0; i < iters; ++i)
      prd::ring_take(
          pos, n, limit,
          [&](int s, unsigned par, int& lim) {
            const bool ok = w.wait(1, w.full[s], par, lim, false);
            if (!ok && plant == 1) { lim = 1; w.abort_flag = true; return true; }
            return ok;
          },
          [&](int s, bool landed) {
            if (!landed) return;
            if (w.copying[s] && plant == 0) w.fault("stage used before its copies landed");
            w.reading[s] += 1;
            w.step(1);
          });
    w.end(1);
  });
  prod.join();
  cons.join();
  if (plant != 2)
    prd::ring_drain(filled, n, [&](int s, unsigned par) {
      for (int i = 0; i < 100000 && !w.full[s].done(par); ++i) w.hardware();
    });
  for (int s = 0; s < n; ++s)
    if (w.copying[s]) w.fault("copy in flight at the end");
  if (!w.abort_flag && filled != iters) w.fault("not all stages filled");
  return w.bad;
}

int main() {
  std::mt19937 rng(7);
  int found[3] = {0, 0, 0};
  for (int plant = 0; plant < 3; ++plant)
    for (int t = 0; t < 700; ++t) {
      const int n = 2 + rng() % 4, iters = 1 + rng() % 24;
      const int pp = rng() % 3 ? 4000 : 1 + rng() % 40, pc = rng() % 3 ? 1 + rng() % 40 : 4000;
      const char* bad = trial(n, iters, pp, pc, rng(), plant);
      if (bad && plant == 0) {
        std::printf("trial %d (n %d, iters %d, polls %d %d): %s\n", t, n, iters, pp, pc, bad);
        return 1;
      }
      found[plant] += bad != nullptr;
    }
  if (!found[1] || !found[2]) { std::printf("planted: %d %d\n", found[1], found[2]); return 2; }
  std::printf("ok\n");
  return 0;
}
'''


def test_ring_rules_hold_when_waits_give_up(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ is missing")
    src = tmp_path / "ring.cpp"
    exe = tmp_path / "ring"
    src.write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2505_20968_gb300", "csrc")
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", csrc, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)   # the deadlock watchdog
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
