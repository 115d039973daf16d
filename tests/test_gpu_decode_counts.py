"""Decode reads the token counts before the kernel ahead of it has finished, as a hint.  Here that kernel is one that lets its
successors start early (an append that itself waits for a forward), and writes other counts than the decode has seen by then."""
import pytest
import torch

from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,D,sink,W,bt", [
    (1, 8, 1, 128, 0, 4096, 0),
    (5, 16, 2, 64, 64, 960, 64),
    (300, 4, 2, 64, 0, 200, 0),            # more sequences than a block has threads
], ids=str)
def test_counts_written_by_an_overlapped_append(B, Hq, Hkv, D, sink, W, bt):
    from paper_2410_01485_b200 import binding as lg, build
    build.build()
    lg.load_library()
    p, cap = lg.decode_params(B, Hq, Hkv, D, sink, W, block_tokens=bt), sink + W
    g = torch.Generator(device="cuda").manual_seed(B)
    kc, vc = (torch.randn(B, Hkv, cap, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    q = torch.randn(B, Hq, D, generator=g, device="cuda").to(torch.bfloat16)
    ws = lg.decode_workspace(p)
    # the counts are rows of a cache of their own: an append of one row of 16 bf16 x 4 moves 16 int64
    rows = (B + 15) // 16
    pc = lg.decode_params(1, rows, rows, 64, 0, 1)
    cache, other = (torch.zeros(1, rows, 1, 64, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    n = cache.view(torch.int64).view(-1)[:B]
    steps = 12
    counts = torch.randint(-1, 2 * cap, (steps, rows * 16), generator=g, device="cuda")
    counts[3], counts[4], counts[5, ::2] = 0, cap, 1
    zero = torch.zeros(1, dtype=torch.int64, device="cuda")
    # something ahead of the append that takes a while on few SMs and lets its successors start: a forward of 16 CTAs
    # (with documents its tiles are not cut)
    docs = torch.zeros(1, 4096, dtype=torch.int32, device="cuda")
    pf = lg.attn_params(1, 1, 1, 4096, 64, 64, synth.MODE_FULL_CAUSAL, doc_start=docs)
    x = torch.randn(1, 1, 4096, 64, generator=g, device="cuda").to(torch.bfloat16)
    wf = lg.attn_workspace(pf, False)
    of, lf = torch.empty_like(x), torch.empty(1, 1, 4096, device="cuda")

    def run(wait):
        out = []
        for t in range(steps):
            lg.lg_sparse_attn_fwd(pf, x, x, x, o=of, lse=lf, workspace=wf)
            src = counts[t].view(torch.bfloat16).view(1, rows, 1, 64)
            lg.lg_kv_ring_append(pc, cache, other, src, src, zero)
            if wait:
                torch.cuda.synchronize()
            out.append(lg.lg_sparse_decode(p, q, kc, vc, n, workspace=ws))
            if wait:
                torch.cuda.synchronize()
        return out

    run(True)                                    # (everything loaded and compiled once)
    for (o, l), (o1, l1), c in zip(run(False), run(True), counts):
        assert torch.equal(o, o1) and torch.equal(l, l1)
        empty = c[:B] <= 0
        assert bool((l[empty] == -float("inf")).all()) and bool(torch.isfinite(l[~empty]).all())
