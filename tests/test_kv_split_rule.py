"""Host logic of the cut kv tiles (csrc/lg_pattern.h, lg_api.cu): which calls cut, alike for a problem and for its groups
of heads.  No GPU: sizes are what the library's size queries answer."""
import ctypes as C

import pytest

from paper_2410_01485_b200 import binding, build


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
