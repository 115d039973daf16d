"""The closed forms the schedules are laid out with (csrc/lg_pattern.h) against the block predicate, counted block by
block: row and column starts, column lengths, the order of the columns in the kv tiles and where each tile's schedule
starts.  Every pattern with up to 24 blocks, sink / stride up to 8 and window / local run up to 9 blocks; compiled for
the host."""
import os
import shutil
import subprocess

import pytest

from paper_2410_01485_b200 import build

SOURCE = r"""
#define __forceinline__ inline
#include "lg_pattern.h"
#include <algorithm>
#include <cstdio>
#include <vector>
using namespace lg;
int main() {
  long bad = 0, n = 0;
  for (int nB = 1; nB <= 24; nB++)
    for (int mode = 0; mode < 3; mode++)
      for (int x = 0; x < (mode ? 9 : 1); x++)
        for (int y = 1; y < (mode ? 10 : 2); y++) {
          PatternDev p{};
          p.nB = nB; p.mode = mode; p.block = 64;
          if (mode == 1) { p.ns = x; p.nw = y; }
          if (mode == 2) { p.stride = x + 1; p.nl = y; }
          n++;
          std::vector<int> rows(nB + 1), cols(nB + 1), len(nB), order(nB);
          for (int q = 0; q < nB; q++)
            for (int k = 0; k < nB; k++)
              if (block_active(p, q, k)) { rows[q + 1]++; cols[k + 1]++; len[k]++; }
          for (int i = 0; i < nB; i++) { rows[i + 1] += rows[i]; cols[i + 1] += cols[i]; order[i] = i; }
          for (int i = 0; i <= nB; i++) bad += (row_start(p, i) != rows[i]) + (col_start(p, i) != cols[i]);
          for (int c = 0; c < nB; c++) {
            bad += col_len(p, c) != len[c];
            for (int q = c; q < c + len[c]; q++) bad += !block_active(p, q, c) + (col_pos(p, q, c) != cols[c] + q - c);
          }
          for (int R = 1; R <= 2; R++) {
            if (mode == 2 && R == 2)
              std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return len[a] > len[b]; });
            int sum = 0;
            for (int i = 0; i <= nB; i++) {
              bad += kv_start(p, R, i) != sum;
              if (i < nB) { bad += kv_col(p, R, i) != order[i]; sum += len[order[i]]; }
            }
          }
        }
  std::printf("%ld %ld\n", n, bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_closed_forms_match_the_predicate(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(cuda, "include"), str(src), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    patterns, bad = map(int, out.stdout.split())
    assert patterns == 24 * (1 + 2 * 81) and bad == 0 and out.returncode == 0
