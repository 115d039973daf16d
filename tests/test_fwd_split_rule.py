"""Which super-tiles the forward cuts along their keys (fwd_split, csrc/lg_pattern.h), compiled for the host: the tiles'
lengths against the block predicate, the limits that the workspace and the kernel rely on, and that the problems of
test_gpu_fwd_split.py are cut, the groups of its host-buffer step otherwise when on their own.  No GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2410_01485_b200 import build, synth

SOURCE = r"""
#define __forceinline__ inline
#include <cuda_runtime.h>
template <typename T> static cudaError_t cudaFuncSetAttribute(T* f, cudaFuncAttribute a, int v) { return ::cudaFuncSetAttribute((const void*)f, a, v); }
#include "lg_host.h"
#include <cstdio>
#include <cstdlib>
using namespace lg;
static PatternDev pattern(int L, int block, int mode, int a, int b) {
  PatternDev p{};
  p.nB = (L + block - 1) / block; p.block = block; p.mode = mode;
  if (mode == 1) { p.ns = a; p.nw = b; }
  if (mode == 2) { p.stride = a; p.nl = b; }
  return p;
}
int main() {
  std::srand(1);
  for (int i = 0; i < 100000; ++i) {   // a tile's steps
    const int block = std::rand() & 1 ? 64 : 128;
    const PatternDev p = pattern((1 + std::rand() % 60) * block, block, std::rand() % 3, 1 + std::rand() % 9, 1 + std::rand() % 12);
    const int n = 256 / block, r0 = std::rand() % p.nB;
    int blocks = 0;
    for (int kb = 0; kb < p.nB; ++kb) {
      bool on = false;
      for (int r = r0; r < r0 + n && r < p.nB; ++r) on |= block_active(p, r, kb);
      blocks += on;
    }
    if (fwd_tile_steps(p, r0, n) != (blocks * block + 127) / 128) { std::printf("steps\n"); return 1; }
  }
  for (int i = 0; i < 100000; ++i) {   // the limits
    const int block = std::rand() & 1 ? 64 : 128, L = 1 + std::rand() % 60000, heads = 1 + std::rand() % 128;
    const PatternDev p = pattern(L, block, std::rand() % 3, std::rand() % 20 + 1, std::rand() % 100 + 1);
    const int row0 = std::rand() % 4 == 0 ? std::rand() % p.nB : 0, tiles = (L - row0 * block + 255) / 256;
    const FwdSplit k = fwd_split(p, std::rand() & 1 ? 64 : 128, row0, tiles, heads);
    if (k.len == 0) continue;
    int longest = 0;
    for (int t = 0; t < tiles; ++t) { const int s = fwd_tile_steps(p, row0 + 256 / block * t, 256 / block); if (s > longest) longest = s; }
    if (k.n_cut < 1 || k.n_cut > tiles || k.places < 2 || k.places > kFwdMaxPieces || (longest + k.len - 1) / k.len > k.places ||
        heads * k.n_cut > kFwdMaxCutTiles || heads * k.n_cut * k.places > kFwdMaxPlaces) { std::printf("limits\n"); return 1; }
  }
  int heads, L, block, mode, a, b, D, row0;
  while (std::scanf("%d %d %d %d %d %d %d %d", &heads, &L, &D, &block, &mode, &a, &b, &row0) == 8) {
    Resolved r{};
    r.pat = pattern(L, block, mode, a, b);
    r.D = D; r.block = block; r.mode = mode; r.st_row0 = row0;
    r.n_stiles = (L - row0 * block + 255) / 256;
    r.nnz = row_start(r.pat, r.pat.nB);
    const FwdSplit k = fwd_split_of(r, heads);
    std::printf("%d %d %d\n", k.len, k.n_cut, k.places);
  }
}
"""


def _line(cfg, heads=None):
    a, b = {synth.MODE_FULL_CAUSAL: (0, 0), synth.MODE_SINK_WINDOW: (cfg.sink_tokens // cfg.block, cfg.window_tokens // cfg.block + bool(cfg.window_exact)),
            synth.MODE_STRIDED_LOCAL: (cfg.stride_blocks, cfg.local_blocks)}[cfg.mode]
    return (heads or cfg.B * cfg.Hq, cfg.L, cfg.D, cfg.block, cfg.mode, a, b, 0)


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs a host compiler")
    d = tmp_path_factory.mktemp("rule")
    (d / "t.cpp").write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(cuda, "include"), str(d / "t.cpp"), "-o", str(d / "t")],
                   check=True)

    def ask(lines):
        text = "".join(" ".join(map(str, x)) + "\n" for x in lines)
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True)
        assert out.returncode == 0, out.stdout
        return [tuple(map(int, x.split())) for x in out.stdout.splitlines()]
    return ask


def test_lengths_and_limits(rule):
    assert rule([]) == []


def test_gpu_cases_are_cut(rule):
    import test_gpu_fwd_split as gpu
    for c, k in zip(gpu.CASES, rule([_line(c, c.Hq) for c in gpu.CASES])):
        assert k[0] > 0, c.name
    assert rule([(4, 64 + 2048 + 300, 128, 64, 1, 1, 33, 33)])[0][0] > 0          # the chunk
    whole, group = rule([_line(gpu.GROUPS), _line(gpu.GROUPS, gpu.GROUPS.Hq // 4)])
    assert whole[0] > 0 and group[0] > 0 and whole != group


def test_more_gpu_cases_are_cut(rule):
    import test_gpu_fwd_cut as gpu
    chunks = [(B * Hq, sink + W + T, 128, 64, 1, sink // 64, W // 64 + 1, (sink + W) // 64) for B, Hq, _, sink, W, T, _ in gpu.CHUNKS]
    assert all(k[0] > 0 for k in rule([_line(gpu.FULL), _line(gpu.WINDOW)] + chunks))


def test_where_it_is_not_worth_it(rule):
    lines = [(64, 10007, 128, 128, 0, 0, 0, 0),      # 2560 CTAs: many rounds
             (2, 512, 64, 64, 1, 1, 2, 0),           # three steps a tile
             (16, 4096, 128, 64, 0, 0, 0, 0),        # 256 CTAs of 2 to 32 steps: the order alone fills the chip
             (16, 1500, 128, 64, 0, 0, 0, 0),        # 96 CTAs of up to 12 steps: 33.3 us, in pieces of 5 43.6 us
             (8, 3000, 128, 64, 1, 1, 32, 0),        # 96 CTAs of 18 steps: 43.8 us, in pieces of 8 52.0 us
             (48, 6001, 64, 64, 1, 1, 17, 0)]        # two CTAs on an SM
    assert all(k[0] == 0 for k in rule(lines))
