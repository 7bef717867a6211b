"""The arrival counter of the grid barrier on the host: it keeps its order where it passes 2^32."""
import subprocess

from paper_2404_02521_gb300 import build

SOURCE = r"""
#include "grid_barrier.cuh"
#include <cstdio>
int main() {
  // every barrier of a group of `blocks`: no arrival but the last one reaches the target, and the last one does
  for (unsigned blocks : {1u, 2u, 152u, 304u, 1024u}) {
    unsigned seen = 0u - 40u * blocks - 7u, target = seen;
    for (int barrier = 0; barrier < 100; ++barrier) {
      target += blocks;
      for (unsigned b = 0; b < blocks; ++b) {
        if (bsp::grid_reached(seen, target)) { printf("early: blocks %u seen %u target %u\n", blocks, seen, target); return 1; }
        ++seen;
        // a block that looks late finds the next barrier's first arrivals there already
        if (b + 1 == blocks && !(bsp::grid_reached(seen, target) && bsp::grid_reached(seen + blocks - 1, target))) {
          printf("never: blocks %u seen %u target %u\n", blocks, seen, target);
          return 1;
        }
      }
    }
  }
  return 0;
}
"""


def test_arrivals_beyond_the_counters_range(tmp_path):
    src = tmp_path / "barrier.cu"
    src.write_text(SOURCE)
    exe = tmp_path / "barrier"
    r = subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, "-o", str(exe), str(src)], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
