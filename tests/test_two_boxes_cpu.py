"""Bookkeeping of the attention forward's A_ref loads (csrc/two_boxes.h, compiled for the host): whichever wait
gives up, every load that was issued has landed or is drained before the block ends. No GPU is needed."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34866_gb300", "csrc")

# The epilogue's use: two loads ahead, a tile of `per_tile` chunks whose remaining chunks are walked through after
# a wait that gave up, no load issued from there on.
PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "two_boxes.h"
int main() {
  for (int per_tile = 2; per_tile <= 4; per_tile += 2)
    for (int tiles = 1; tiles <= 3; ++tiles)
      for (int fail = 0; fail <= per_tile * tiles; ++fail) {  // the wait for load `fail` gives up (the last: none)
        const int total = per_tile * tiles;
        jab::TwoBoxes b;
        std::vector<int> waited(total, 0);
        int at = 0;  // loads waited for so far, in order
        auto issue = [&] { if (b.issued < total) ++b.issued; };
        auto wait = [&](int buf, unsigned parity) {
          if (at >= b.issued || buf != (at & 1) || parity != (unsigned)((at >> 1) & 1)) return printf("order\n"), false;
          if (at == fail) return false;
          ++waited[at++];
          return true;
        };
        issue();
        issue();
        bool have = true;
        for (int t = 0; t < tiles && have; ++t)
          for (int c = 0; c < per_tile; ++c) {
            if (have) have = b.take(wait);
            if (have) issue();
          }
        if (have != (fail >= total)) return printf("have %d %d %d\n", per_tile, tiles, fail), 1;
        b.drain([&](int buf, unsigned parity) {
          if (at >= b.issued || buf != (at & 1) || parity != (unsigned)((at >> 1) & 1)) printf("order\n");
          else ++waited[at++];
        });
        for (int n = 0; n < b.issued; ++n)
          if (waited[n] != 1) return printf("load %d of %d: %d waits, fail %d\n", n, b.issued, waited[n], fail), 1;
      }
  printf("ok\n");
}
"""


def test_every_issued_load_lands_or_is_drained(tmp_path):
    src, exe = tmp_path / "boxes.cpp", tmp_path / "boxes"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout
