"""Which cooperative grids may run side by side (csrc/coop_budget.h), on the
CPU: the rule is host code without CUDA, compiled here into a small program.

Grids of different streams that fit the device together must not wait for one
another (threads with handles of their own would take turns), and grids that
could run together must never need more SMs than there are (each could hold
some and wait for the rest forever).
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>
#include "coop_budget.h"
using mslice::CoopBudget;

static void need(bool ok, const char* what) {
  if (!ok) {
    std::printf("failed: %s\n", what);
    std::exit(1);
  }
}

int main() {
  const auto never = [](int) { return false; };
  std::vector<int> w;
  {  // grids that fit together do not wait; one that does not waits for what it takes over
    CoopBudget b(152);
    const int e1 = b.take(76, 1, never, w);
    need(w.empty(), "first grid");
    const int e2 = b.take(63, 2, never, w);
    need(w.empty(), "second grid beside the first");
    need(e1 != e2, "two events");
    b.take(63, 2, never, w);
    need(w == std::vector<int>{e2}, "a stream takes over its own units");
    b.take(20, 3, never, w);
    need(w == std::vector<int>{e1}, "13 free units and 7 of the oldest grid");
  }
  {  // the whole device: behind everything, and everything behind it
    CoopBudget b(152);
    const int e1 = b.take(10, 1, never, w), e2 = b.take(10, 2, never, w);
    const int all = b.take(304, 3, never, w);
    need(w.size() == 2 && w[0] != w[1] && (w[0] == e1 || w[0] == e2) && (w[1] == e1 || w[1] == e2), "waits for both");
    b.take(1, 1, never, w);
    need(w == std::vector<int>{all}, "behind the whole device");
    b.take(1, 2, [](int) { return true; }, w);
    need(w.empty(), "finished grids need no wait");
  }
  // Random streams of grids, run in random order as far as the waits and the
  // streams' own order allow: the grids running together fit the device.
  for (unsigned seed = 0; seed < 200; ++seed) {
    std::mt19937 rng(seed);
    const int units = 1 + (int)(rng() % 160), streams = 1 + (int)(rng() % 9), grids = 400;
    CoopBudget b(units);
    struct Grid {
      int blocks, stream;
      std::vector<int> behind;  // grids that have to end first
      int state = 0;            // 0 waiting, 1 running, 2 ended
    };
    std::vector<Grid> g;
    std::map<int, int> recorded;  // event -> the grid recorded last
    std::vector<int> last(streams, -1);
    size_t ended = 0;
    int running = 0;
    const auto step = [&] {  // one grid that may starts, or one that runs ends
      std::vector<int> can;
      for (size_t i = 0; i < g.size(); ++i) {
        bool ok = g[i].state == 0;
        for (int x : g[i].behind) ok = ok && g[x].state == 2;
        if (ok || g[i].state == 1) can.push_back((int)i);
      }
      need(!can.empty(), "nothing can go on");
      Grid& x = g[can[rng() % can.size()]];
      if (x.state == 0) {
        x.state = 1;
        running += std::min(x.blocks, units);
        need(running <= units, "running grids exceed the device");
      } else {
        x.state = 2;
        running -= std::min(x.blocks, units);
        ++ended;
      }
    };
    for (int i = 0; i < grids; ++i) {
      Grid x;
      x.stream = (int)(rng() % streams);
      x.blocks = rng() % 4 == 0 ? 2 * units : 1 + (int)(rng() % units);
      const int e = b.take(x.blocks, (uintptr_t)(x.stream + 1), [&](int ev) { return g[recorded[ev]].state == 2; }, w);
      for (int ev : w) x.behind.push_back(recorded[ev]);
      if (last[x.stream] >= 0) x.behind.push_back(last[x.stream]);
      recorded[e] = last[x.stream] = i;
      g.push_back(x);
      for (int k = (int)(rng() % 4); k > 0 && ended < g.size(); --k) step();
    }
    while (ended < g.size()) step();
    need(running == 0, "all ended");
  }
  std::printf("ok\n");
}
'''


def test_grids_that_may_run_together(tmp_path):
    src = tmp_path / "budget.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "budget"
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "paper_2608_03695_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
