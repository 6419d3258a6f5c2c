"""The stage ring of the few-row GEMM (csrc/ring.h) against a model of its barriers, compiled for the host."""
import os
import subprocess

from conftest import ROOT

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "ring.h"

// Barrier "full" of every slot: number of its phases that have completed.
// A wait for `parity` returns while the current phase has the other parity.
struct Bars {
  std::vector<int> done;
  bool wait(int slot, uint32_t parity) const { return ((uint32_t)done[slot] & 1u) != parity; }
};

int main() {
  for (int n = 1; n <= 8; ++n)
    for (int uses = 0; uses <= 3 * n + 1; ++uses) {
      mlora::Ring at(n);
      for (int u = 0; u < uses; ++u) {
        if (at.slot != u % n || at.parity != (uint32_t)(u / n & 1)) return std::printf("place of use %d of %d\n", u, n), 1;
        at.next();
      }
      const int in_flight = uses < n ? uses : n;      // a slot is used again only after its loads have landed
      // every load has landed, or all but one: each wait returns, or exactly the one for that use does not
      for (int missing = -1; missing < in_flight; ++missing) {
        Bars b{std::vector<int>(n, 0)};
        for (int u = 0; u < uses; ++u) if (u != uses - 1 - missing || missing < 0) b.done[u % n]++;
        int visited = 0, blocked = 0, blocked_slot = -1;
        at.last_uses([&](int slot, uint32_t parity) {
          ++visited;
          if (!b.wait(slot, parity)) { ++blocked; blocked_slot = slot; }
        });
        if (visited != in_flight) return std::printf("ring %d, %d uses: %d visited\n", n, uses, visited), 1;
        if (blocked != (missing >= 0 ? 1 : 0)) return std::printf("ring %d, %d uses, %d missing: %d waits block\n", n, uses, missing, blocked), 1;
        if (missing >= 0 && blocked_slot != (uses - 1 - missing) % n) return std::printf("ring %d: wrong slot\n", n), 1;
      }
    }
  return 0;
}
"""


def test_a_role_that_gives_up_waits_for_the_loads_it_has_in_flight(tmp_path):
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2607_28848_b200", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
