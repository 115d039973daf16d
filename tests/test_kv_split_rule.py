"""Host logic of the cut kv tiles (csrc/lg_pattern.h, lg_api.cu): which calls cut, alike for a problem and for its groups
of heads.  No GPU: sizes are what the library's size queries answer."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

from paper_2410_01485_b200 import binding, build
from tests.test_gpu_kv_split import CASES, DOC_GROUPS, GROUPS


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load_library()


@pytest.mark.parametrize("groups", [1, 2, 4])
@pytest.mark.parametrize("variant", ["two_pass", "keep_ds"])
def test_sequences_with_documents_are_cut_like_one_of_them(lib, groups, variant, monkeypatch):
    """With documents a batch runs sequence by sequence: whatever the number of head groups, a group's workspace holds
    two slices of the size one sequence takes in that group (its cut tiles' partial sums among them)."""
    monkeypatch.setenv("LG_BWD_VARIANT", variant)
    sizes = []
    for B in (1, 2):
        p = binding.attn_params(B, 16, 4, 6000, 64, 64, binding.MODE_SINK_WINDOW, sink_tokens=64, window_tokens=1024)
        p.doc_start = 256                          # only its presence is looked at: no call touches the array here
        sizes.append(lib.lg_sparse_attn_fwd_bwd_host_workspace_bytes(C.byref(p), groups))
    assert sizes[0] > 0 and sizes[1] == 2 * sizes[0]


SOURCE = r"""
#define __forceinline__ inline
#include "lg_pattern.h"
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>
using namespace lg;
static long allocations = 0;
void* operator new(std::size_t n) { ++allocations; return std::malloc(n); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
// stdin: "nB block mode a b G kv_heads n_ktiles" a line (a, b = sink and window blocks, or stride and local blocks);
// stdout: items of a piece (0: not cut), places, allocations of the rule, faults of its regions
int main() {
  PatternDev p{};
  int a, b, G, kv, nt;
  while (std::scanf("%d %d %d %d %d %d %d %d", &p.nB, &p.block, &p.mode, &a, &b, &G, &kv, &nt) == 8) {
    p.ns = p.nw = p.stride = p.nl = 0;
    if (p.mode == 1) { p.ns = a; p.nw = b; }
    if (p.mode == 2) { p.stride = a; p.nl = b; }
    const long before = allocations;
    const KvSplit k = kv_split(p, nt, G, row_start(p, p.nB), kv);
    const long spent = allocations - before;
    long bad = 0;
    const int R = 128 / p.block;
    if (p.nB <= 64)                                  // a tile's length: the query blocks that see one of its columns
      for (int t = 0; t < nt; ++t) {
        int n = 0;
        for (int q = 0; q < p.nB; ++q) {
          bool on = false;
          for (int x = R * t; x < R * t + R && x < p.nB; ++x) on |= block_active(p, q, kv_col(p, R, x));
          n += on;
        }
        bad += n != kv_tile_len(p, R, t);
      }
    if (k.len > 0) {                                 // every rank, longest tile first, has places for its pieces
      std::vector<int> len(nt);
      for (int t = 0; t < nt; ++t) len[t] = kv_tile_len(p, R, t);
      std::sort(len.begin(), len.end(), [](int x, int y) { return x > y; });
      int place = 0, i = 0, cut = 0;
      for (int y = 0; y < nt; ++y) {
        while (i + 1 < k.n_regions && y >= k.first_rank[i + 1]) ++i;
        if (y == k.first_rank[i]) bad += k.first_place[i] != place;
        const long pieces = (static_cast<long>(len[y]) * G + k.len - 1) / k.len;
        bad += pieces > k.segs[i] || k.segs[i] > kKvMaxSegs;
        place += k.segs[i];
        cut += k.segs[i] > 1;
        bad += (k.segs[i] > 1) != (y < k.n_ranks);
        if (y + 1 == k.n_ranks) bad += k.n_places != place;
      }
      bad += k.n_regions > kKvMaxRegions || k.first_rank[k.n_regions] != nt || k.first_place[k.n_regions] != place || cut != k.n_ranks;
    }
    std::printf("%d %d %ld %ld\n", k.len, k.len ? k.first_place[k.n_regions] : nt, spent, bad);
  }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """problems (nB, block, mode, a, b, G, kv heads, kv tiles) -> [(items of a piece, places, allocations, faults)]"""
    if shutil.which("g++") is None:
        pytest.skip("needs a host compiler")
    d = tmp_path_factory.mktemp("rule")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(cuda, "include"), str(src), "-o",
                    str(exe)], check=True)

    def run(problems):
        text = "".join(" ".join(map(str, x)) + "\n" for x in problems)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split()
        got = list(zip(*[iter(map(int, out))] * 4))
        assert len(got) == len(problems)
        return got

    return run


def _small_problems():
    for nB in (1, 2, 3, 7, 12, 16, 23, 24, 40, 64):
        for block in (64, 128):
            for mode, a, b in [(0, 0, 0)] + [(1, a, b) for a in (0, 1, 2, 3) for b in (1, 2, 5, 17)] + \
                              [(2, a, b) for a in (1, 2, 3, 5, 16) for b in (1, 2, 3, 4)]:
                for G, kv in ((1, 1), (1, 4), (3, 2), (8, 1), (8, 8), (16, 1)):
                    yield nB, block, mode, a, b, G, kv, -(-nB * block // 128)


def test_places_hold_every_tile_and_the_rule_allocates_nothing(rule):
    """kv_tile_len against the predicate; each launch rank has at least as many places as its tile has pieces; no memory
    is requested (nothing may be thrown through the C ABI)."""
    problems = list(_small_problems())
    got = rule(problems)
    assert sum(x[0] > 0 for x in got) > 500            # of 4440: the rule does cut
    assert all(x[2] == 0 for x in got)
    assert [p for p, x in zip(problems, got) if x[3]] == []


@pytest.mark.parametrize("mode, a, b, kv", [(1, 1, 2, 1), (1, 1, 1, 2), (2, 4000, 1, 1), (2, 30000, 2, 1)])
@pytest.mark.parametrize("block", [64, 128])
def test_places_stay_within_a_grid(rule, block, mode, a, b, kv):
    """The kv tiles (at most 65535) and the places of cut ones are a grid's y extent: no cut rather than a launch that fails."""
    problems = [(n * 128 // block, block, mode, a, b, 1, kv, n) for n in [60000, 64000] + list(range(65400, 65536))]
    got = rule(problems)
    assert got[0][0] > 0 and got[0][1] > 60000                         # cut well below the limit
    assert max(places for _, places, _, _ in got) <= 65535
    assert got[-1][0] == 0                                             # 65535 tiles leave no place to spare
    assert all(x[3] == 0 for x in got)


def _problem(cfg, kv_heads):
    a, b = [(0, 0), (cfg.sink_tokens // cfg.block, cfg.window_tokens // cfg.block + bool(cfg.window_exact)),
            (cfg.stride_blocks, cfg.local_blocks)][cfg.mode]
    return -(-cfg.L // cfg.block), cfg.block, cfg.mode, a, b, cfg.Hq // cfg.Hkv, kv_heads, -(-cfg.L // 128)


def test_the_gpu_tests_problems_are_cut(rule):
    """Those of the parity test, whether the whole batch counts or (with documents) a sequence of it; and where groups of
    heads are compared with the whole, a group by itself would be cut into other pieces."""
    for cfg in CASES:
        assert all(x[0] > 0 for x in rule([_problem(cfg, n * cfg.Hkv) for n in {1, cfg.B}])), cfg.name
    for cfg, groups in ((GROUPS, (2, 4)), (DOC_GROUPS, (2, 4))):
        whole, *parts = (x[0] for x in rule([_problem(cfg, cfg.Hkv // n) for n in (1, *groups)]))
        assert whole > 0 and all(0 < x != whole for x in parts), (cfg.name, whole, parts)


@pytest.mark.parametrize("groups", [1, 2, 4])
def test_groups_of_the_host_step_keep_ds_like_the_whole(lib, groups, monkeypatch):
    """Which backward runs is decided for the whole problem: its groups' results are bit-identical to it, and the limit
    on the dS buffer holds for what the groups' workspaces take together."""
    p = binding.attn_params(1, 16, 4, 8192, 128, 128, binding.MODE_SINK_WINDOW, sink_tokens=128, window_tokens=1024)
    ds = 16 * binding.lg_block_index_nnz(p) * 128 * 128 * 2
    monkeypatch.delenv("LG_BWD_VARIANT", raising=False)
    sizes = []
    for cap in (0.9 * ds, 1.1 * ds):                       # below the whole's buffer (and above any group's), and above it
        monkeypatch.setenv("LG_KEEP_DS_MAX_GB", "%.6f" % (cap / 1e9))
        assert lib.lg_sparse_attn_bwd_variant(C.byref(p)) == (0 if cap < ds else 2)
        sizes.append(lib.lg_sparse_attn_fwd_bwd_host_workspace_bytes(C.byref(p), groups))
    assert ds <= sizes[1] - sizes[0] < ds + (1 << 20)


@pytest.mark.parametrize("B", [1, 2])
def test_the_variant_reported_with_documents_is_the_one_that_runs(lib, B, monkeypatch):
    """Sequence by sequence: a sequence's own dS buffer decides, and the answer agrees with the workspace."""
    p = binding.attn_params(B, 16, 4, 8192, 128, 128, binding.MODE_SINK_WINDOW, sink_tokens=128, window_tokens=1024)
    p.doc_start = 256                                      # (only its presence is looked at)
    ds = 16 * binding.lg_block_index_nnz(p) * 128 * 128 * 2
    sizes = {}
    for variant in ("two_pass", "keep_ds"):
        monkeypatch.setenv("LG_BWD_VARIANT", variant)
        sizes[variant] = lib.lg_sparse_attn_workspace_bytes(C.byref(p), 1)
    assert B * ds <= sizes["keep_ds"] - sizes["two_pass"] < B * (ds + (1 << 20))
    monkeypatch.delenv("LG_BWD_VARIANT")
    for cap, want in ((0.9 * ds, "two_pass"), (1.1 * ds, "keep_ds")):
        monkeypatch.setenv("LG_KEEP_DS_MAX_GB", "%.6f" % (cap / 1e9))
        assert binding.bwd_variant_name(p) == want
        assert lib.lg_sparse_attn_workspace_bytes(C.byref(p), 1) == sizes[want]
