"""Which form of the D = 64 forward a problem takes (fwd_two_ctas, csrc/lg_host.h): two CTAs on an SM only where the grid
keeps the pairs together.  The rule compiled for the host; no GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2410_01485_b200 import build

SOURCE = r"""
#define __forceinline__ inline
#include <cuda_runtime.h>
template <typename T> static cudaError_t cudaFuncSetAttribute(T* f, cudaFuncAttribute a, int v) { return ::cudaFuncSetAttribute((const void*)f, a, v); }
#include "lg_host.h"
#include <cstdio>
int main() {   // "B Hq L D block mode a b" a line (a, b = sink and window blocks, or stride and local blocks)
  int B, Hq, L, D, block, mode, a, b;
  while (std::scanf("%d %d %d %d %d %d %d %d", &B, &Hq, &L, &D, &block, &mode, &a, &b) == 8) {
    lg::Resolved r{};
    r.B = B; r.Hq = Hq; r.L = L; r.D = D; r.block = block; r.mode = r.pat.mode = mode;
    r.pat.nB = (L + block - 1) / block;
    r.pat.ns = r.pat.stride = a; r.pat.nw = r.pat.nl = b;
    r.n_stiles = (L + 255) / 256;
    r.nnz = lg::row_start(r.pat, r.pat.nB);
    std::printf("%d\n", lg::fwd_two_ctas(r));
  }
}
"""

CASES = [                                       # measured: the form that is faster
    ((1, 4, 3318, 64, 64, 0, 0, 0), 0),         # 52 CTAs
    ((1, 32, 8192, 64, 64, 0, 0, 0), 0),        # 1024 CTAs of 1 to 64 steps
    ((1, 64, 30000, 64, 64, 0, 0, 0), 1),       # 7552 CTAs
    ((1, 8, 3318, 64, 64, 1, 1, 16), 0),        # 104 CTAs
    ((3, 16, 6001, 64, 64, 1, 1, 16), 1),       # 1152 CTAs
    ((3, 16, 6001, 64, 128, 1, 1, 8), 1),
    ((1, 16, 8192, 64, 64, 1, 2, 49), 0),       # 512 CTAs of a window of 3136
    ((1, 32, 16384, 64, 64, 1, 1, 64), 1),      # 2048 CTAs of a window of 4096
    ((1, 4, 8192, 64, 64, 2, 16, 4), 0),        # 128 CTAs
    ((1, 16, 8192, 64, 64, 2, 16, 4), 1),       # 512 CTAs of short rows
    ((3, 16, 6001, 128, 64, 1, 1, 16), 0),      # D = 128: tensor memory is full with one
]


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_pairs_only_where_the_grid_fills_the_chip(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(cuda, "include"), str(src), "-o",
                    str(exe)], check=True)
    text = "".join(" ".join(map(str, c)) + "\n" for c, _ in CASES)
    got = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split()
    assert list(map(int, got)) == [want for _, want in CASES]
