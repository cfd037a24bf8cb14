"""The substitution's ring of copies (csrc/bte_window_plan.h), replayed on the host: every wait is for a copy
that has been issued, no copy is issued into a stage that is still to be read, every copy is issued once, and
every window that the plan accepts gets at least one stage within the shared memory of an SM."""
import os
import subprocess

from tests.conftest import ROOT

PROGRAM = r"""
#include <cstdio>
#include <set>
#include "bte_window_plan.h"
using namespace bte;

// 0, or the line of the first broken rule
static int replay(int np, int S) {
  std::set<int> issued, used;
  bool ok = true;
  auto issue = [&](int q) {
    if (q < 0) return;
    // copy q takes the stage of copy q - S, which must have been used; once each
    if (q >= 2 * np || !issued.insert(q).second || (q >= S && !used.count(q - S))) ok = false;
  };
  for (int q = 0; q < S && q < 2 * np; ++q) issue(q);
  if (!ok) return __LINE__;
  for (int q = 0; q < 2 * np; ++q) {
    // the barrier before the wait for a T: every thread is past copy q - 1
    if (q > 0 && q < np) used.insert(q - 1);
    issue(ring_before_wait(q, np, S));
    if (!ok) return __LINE__;
    if (!issued.count(q)) return __LINE__;  // the wait would never end
    if (q >= np - 1) used.insert(q);        // the barrier that ends a panel of U, or the forward pass
    issue(ring_after_use(q, np, S));
    if (!ok) return __LINE__;
  }
  return static_cast<int>(issued.size()) == 2 * np ? 0 : __LINE__;
}

int main() {
  int bad = 0;
  for (int S = 1; S <= 8; ++S)
    for (int np : {1, 2, 3, 4, 5, 7, 8, 9, 16, 17, 136, 327})
      if (int line = replay(np, S)) ++bad, std::printf("np %d, S %d: line %d\n", np, S, line);
  int one = 0;
  for (int nl = 1; nl <= 32; ++nl)
    for (int nr = 4; nr <= 880; ++nr) {
      const WindowPlan w = window_plan(nr, nl);
      if (!w.ok) continue;
      for (size_t ts : {4, 8})
        for (int nx : {3, 200}) {
          const WindowRing r = window_ring(w, ts, nx, 152);
          if (r.stages < 1 || r.stages > 8 || r.smem > 224 * 1024 || r.stage_bytes % 16) {
            if (++bad < 20) std::printf("nr %d, nl %d, %zu bytes, nx %d: %d stages, %zu bytes\n", nr, nl, ts, nx, r.stages, r.smem);
          }
          one += r.stages == 1;
        }
    }
  std::printf("%d broken, %d with one stage\n", bad, one);
  return bad || !one;
}
"""


def test_every_wait_of_the_ring_ends_and_every_window_has_a_stage(tmp_path):
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2502_16555_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", csrc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
