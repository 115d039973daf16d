"""A workspace that was large enough for a problem is large enough for a smaller one: forward-only attention workspaces over the
length and the head counts, chunk workspaces over the chunk and what lies before it.  No GPU."""
import ctypes as C

import pytest

from paper_2410_01485_b200 import binding, build, synth


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load_library()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("mode,kw", [(synth.MODE_FULL_CAUSAL, {}), (synth.MODE_SINK_WINDOW, dict(sink_tokens=64, window_tokens=2048)),
                                     (synth.MODE_STRIDED_LOCAL, dict(stride_blocks=8, local_blocks=4))], ids=["full", "window", "strided"])
def test_forward(lib, D, mode, kw):
    def size(heads, L):
        p = binding.attn_params(1, heads, heads, L, D, 64, mode, **kw)
        return lib.lg_sparse_attn_workspace_bytes(C.byref(p), 0)
    lengths = [500, 1300, 2000, 2048, 3318, 6000, 8000, 16384, 32768]
    for heads in (64, 8, 4, 2, 1):
        sizes = [size(heads, L) for L in lengths]
        assert 0 < sizes[0] and sizes == sorted(sizes)
        assert all(size(heads, L) == size(64, L) for L in lengths)           # the lists know nothing of the heads


@pytest.mark.parametrize("Hq,Hkv", [(64, 8), (32, 8), (8, 8), (4, 2)])
@pytest.mark.parametrize("B,block_tokens", [(1, 0), (2, 64)])
def test_chunks(lib, Hq, Hkv, B, block_tokens):
    p = binding.decode_params(B, Hq, Hkv, 128, 128, 4096, block_tokens=block_tokens)
    chunks = [1, 16, 64, 100, 256, 300, 512, 1000, 1500, 4096, 8192]
    before = [0, 100, 1000, 4000, 20000]
    table = [[lib.lg_chunk_prefill_workspace_bytes(C.byref(p), T, n) for T in chunks] for n in before]
    assert table[0][0] > 0
    assert all(row == sorted(row) for row in table) and all(list(col) == sorted(col) for col in zip(*table))
