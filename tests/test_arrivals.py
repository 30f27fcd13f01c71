"""The meetings of sa_small_kernel's blocks at the level ends (arrivals.h),
played on the host: no block passes a meeting before every block has arrived,
also where the arrival counter passes 2^32 (blocks x levels of a long
calibration)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_20713_gb300", "csrc")

PLAY = """
#include <cstdio>
#include <cstdlib>
#include "arrivals.h"
int main(int argc, char** argv) {
  const unsigned blocks = (unsigned)std::strtoul(argv[1], nullptr, 10);
  unsigned count = (unsigned)std::strtoul(argv[2], nullptr, 10), target = count;  // a meeting that has ended
  for (int meeting = 0; meeting < 4; ++meeting) {
    target += blocks;
    for (unsigned b = 0; b < blocks; ++b) {
      if (sabr::arrived(count, target)) return std::printf("passed with %u of %u\\n", b, blocks), 1;
      ++count;
    }
    if (!sabr::arrived(count, target)) return std::printf("did not pass\\n"), 1;
    // a block that is late to look sees the arrivals at the next meeting too
    if (!sabr::arrived(count + blocks - 1, target)) return std::printf("late look\\n"), 1;
  }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_meetings_across_the_end_of_the_counter(tmp_path):
    src = tmp_path / "play.cpp"
    src.write_text(PLAY)
    exe = str(tmp_path / "play")
    subprocess.run(["g++", "-O1", "-I", CSRC, str(src), "-o", exe], check=True)
    for blocks in (1, 2, 16, 64, 304, 608, 1216):
        for start in (0, 2**31 - blocks - 1, 2**31 - 1, 2**32 - 3 * blocks, 2**32 - 2 * blocks - 1, 2**32 - blocks,
                      2**32 - 1):
            r = subprocess.run([exe, str(blocks), str(start)], capture_output=True, text=True)
            assert r.returncode == 0, (blocks, start, r.stdout)
