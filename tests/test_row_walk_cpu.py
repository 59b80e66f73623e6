"""The row-OR's walk over the rows of a contraction, compiled for the host: at every
number of rows that the library accepts (below 2^31) each row belongs to one warp,
and the rows formed ahead of the loop never wrap around."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "row_walk.h"
int main() {
  const long long top = 2147483647ll;
  const long long rows[] = {1, 31, 4864, 155648, 155649, 1000003, top - 1300000, top - 155648, top - 1, top};
  const int warps[] = {1, 8, 16, 32, 4864, 9728};
  const int lanes[] = {1, 3, 8, 9, 31, 32};
  for (long long M : rows)
    for (int w : warps)
      for (int L : lanes) {
        if (M / w > 20000000) continue;  // (few warps at the top: the walk is the same)
        const pa::RowWalk walk(M, w, L);
        if (walk.batch < 1 || walk.batch > 32u / L || walk.step != walk.batch * (unsigned)w) return 1;
        long long seen = 0;
        for (int warp = 0; warp < w; warp += w > 64 ? w - 1 : 1) {
          uint32_t row = warp * walk.batch, ahead = row;
          long long row64 = row, ahead64 = ahead, turns = 0;
          for (int k = 0; k < 3; ++k) { ahead += walk.step; ahead64 += walk.step; }
          for (; row < walk.M; row += walk.step, row64 += walk.step) {
            if (row != row64 || ahead != ahead64 || ++turns > M) return 2;
            ahead += walk.step; ahead64 += walk.step;
            seen += (M - row64 < walk.batch ? M - row64 : walk.batch);
          }
          if (row64 < M || row != row64) return 3;
        }
        if (w <= 64 && seen != M) return 4;
      }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_walk_at_the_row_limit(tmp_path):
    src = tmp_path / "walk.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "walk"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_1609_00061_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
