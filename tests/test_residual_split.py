"""How the residual shares out its work (csrc/residual_split.h), compiled for the
host: no block that the launch starts late may find work."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_17636_gb300", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include "residual_split.h"

int main() {
  long bad = 0, wide = 0, small = 0;
  for (int sms : {108, 132, 148, 152, 160})
    for (int bpp = 1; bpp <= 4096; bpp *= 2)
      for (int planes : {3, 9, 17, 33, 65, 129, 257, 513, 64 * 33}) {
        const int grid = int(std::min(8l * sms, long(bpp) * planes));
        int reach = 0;   // blocks that find work with some smaller count
        for (int n = 1; n <= planes; ++n) {
          const ps::ResidualSplit s = ps::residual_split(n, bpp, grid, sms);
          const int busy = std::min(s.items, grid);
          (s.wide ? wide : small) += 1;
          // every cell has one item
          if (s.items != n * s.items_per_plane || s.items_per_plane * (s.wide ? 4 : 1) < bpp ||
              (s.items_per_plane - 1) * (s.wide ? 4 : 1) >= bpp) ++bad;
          // the retirement awaits busy + waiting blocks; the others may start
          // after it, with any smaller count
          if (s.waiting != 0 && s.waiting != grid - busy) ++bad;
          if (s.waiting == 0 && busy < grid && reach > busy) ++bad;
          reach = std::max(reach, busy);
        }
      }
  std::printf("%ld %ld %ld\n", bad, wide, small);
}
"""


def test_a_late_block_finds_no_item(tmp_path):
    """The retirement of the last arriving block lowers the count of active
    planes within the launch.  Whatever smaller count a block reads that
    neither had an item nor was awaited, no item may be its own."""
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    src = tmp_path / "split.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "split"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    bad, wide, small = (int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True,
                                                       check=True).stdout.split())
    assert wide > 1000 and small > 1000
    assert bad == 0
