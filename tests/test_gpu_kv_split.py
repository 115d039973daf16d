"""The dK/dV pass with kv tiles cut into pieces (few kv heads, long tiles): both block sizes and head sizes, every
pattern, ragged lengths, grouped queries, documents (tiles shorter than planned), both backward variants; the host-buffer
step in head groups gives the same bits as the whole problem.  (test_kv_split_rule.py checks that these problems are cut,
and that the groups alone would be cut otherwise.)"""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import lg_oracle as O
from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu
TOL_G = 2e-2                       # the parity tests' bound on gradients below 4; half an ulp of bf16 more from there on


@pytest.fixture(scope="module")
def lg():
    from paper_2410_01485_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


CASES = [
    replace(synth.CFG1, name="sink_64_gqa8", L=1536, D=128, Hq=8, Hkv=1, block=64, sink_tokens=64, window_tokens=128),
    replace(synth.CFG1, name="sink_64_exact_ragged", L=2077, D=64, Hq=4, Hkv=2, block=64, sink_tokens=64, window_tokens=192, window_exact=True),
    replace(synth.CFG1, name="full_128_ragged", mode=synth.MODE_FULL_CAUSAL, L=1999, D=128, Hq=4, Hkv=1, block=128),
    replace(synth.CFG1, name="full_64_gqa3", mode=synth.MODE_FULL_CAUSAL, L=1100, D=64, Hq=3, Hkv=1, block=64, B=2),
    replace(synth.CFG1, name="strided_64", mode=synth.MODE_STRIDED_LOCAL, stride_blocks=4, local_blocks=2, L=1500, D=128, Hq=4, Hkv=1, block=64),
    replace(synth.CFG1, name="strided_128", mode=synth.MODE_STRIDED_LOCAL, stride_blocks=3, local_blocks=1, L=2304, D=64, Hq=4, Hkv=2, block=128),
]


def _check(got, ref, what):
    err = np.abs(synth.to_f64(got) - ref)
    assert (err <= TOL_G + np.where(np.abs(ref) >= 4, np.abs(ref) * 2.0 ** -8, 0)).all(), (what, err.max())


@pytest.mark.parametrize("variant", ["two_pass", "keep_ds"])
@pytest.mark.parametrize("docs", [False, True])
@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_split_tiles_parity(lg, cfg, docs, variant, monkeypatch):
    monkeypatch.setenv("LG_BWD_VARIANT", variant)
    ds = torch.stack([synth.make_doc_start(cfg.L, seed=5 + b, mean_len=500) for b in range(cfg.B)]).cuda() if docs else None
    p = lg.params_of(cfg, doc_start=ds)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=2, with_do=True)
    ws = lg.attn_workspace(p, True)
    o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
    grads = lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"], workspace=ws)
    again = lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"], workspace=ws)
    assert lg.lg_last_status(ws) == 0
    assert all(torch.equal(x, y) for x, y in zip(grads, again))         # the pieces are added in a fixed order
    for b in range(cfg.B):
        pat = O.Pattern.of(cfg)
        if docs:
            pat = replace(pat, doc_start=ds[b].cpu().numpy())
        q, k, v, do = (synth.to_f64(inp[x][b]) for x in ("q", "k", "v", "do"))
        refs = O.attn_backward(q, k, v, do, pat, 1.0 / np.sqrt(cfg.D), rows_per_slab=cfg.block)[:3]
        for x, ref, what in zip(grads, refs, ("dQ", "dK", "dV")):
            _check(x[b], ref, what)


GROUPS = replace(synth.CFG1, name="groups", mode=synth.MODE_FULL_CAUSAL, L=4096, D=64, Hq=8, Hkv=4, block=64)
DOC_GROUPS = replace(synth.CFG1, name="doc_groups", B=2, L=6000, D=64, Hq=16, Hkv=4, block=64, sink_tokens=64, window_tokens=1024)


def test_head_groups_of_the_host_step_split_like_the_whole(lg):
    cfg = GROUPS
    p = lg.params_of(cfg)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=12, with_do=True)
    o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"])
    ref = dict(zip(("o", "lse", "dq", "dk", "dv"), (o, lse) + lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"])))
    host = {k: v.cpu().pin_memory() for k, v in inp.items()}
    for groups in (4, 2):
        out = {n: torch.zeros(t.shape, dtype=t.dtype).pin_memory() for n, t in ref.items()}
        lg.sparse_attn_fwd_bwd_host(lg.params_of(cfg), host, out, head_groups=groups)
        torch.cuda.synchronize()
        for name, t in ref.items():
            assert torch.equal(out[name], t.cpu()), (groups, name)


@pytest.mark.parametrize("groups", [4, 2])
def test_head_groups_with_documents_in_several_sequences(lg, groups):
    """Documents in a batch of two (run sequence by sequence), 16 / 4 heads: a whole sequence is cut into pieces of 48
    items, two or four kv heads on their own would be cut into 24 or 16."""
    cfg = DOC_GROUPS
    ds = torch.stack([synth.make_doc_start(cfg.L, seed=30 + b, mean_len=5000) for b in range(2)]).cuda()
    p = lg.params_of(cfg, doc_start=ds)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=14, with_do=True)
    o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"])
    ref = dict(zip(("o", "lse", "dq", "dk", "dv"), (o, lse) + lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"])))
    host = {k: v.cpu().pin_memory() for k, v in inp.items()}
    out = {n: torch.zeros(t.shape, dtype=t.dtype).pin_memory() for n, t in ref.items()}
    lg.sparse_attn_fwd_bwd_host(lg.params_of(cfg, doc_start=ds), host, out, head_groups=groups)
    torch.cuda.synchronize()
    for name, t in ref.items():
        assert torch.equal(out[name], t.cpu()), (groups, name)


def test_head_groups_run_the_backward_of_the_whole(lg, monkeypatch):
    """A limit on the dS buffer that the whole problem exceeds and a group of its heads does not.  (A strided pattern: its
    kv tiles hold comb columns first, so the variants sum dQ in different orders.)"""
    cfg = replace(GROUPS, mode=synth.MODE_STRIDED_LOCAL, stride_blocks=4, local_blocks=2)
    p = lg.params_of(cfg)
    ds = cfg.Hq * lg.lg_block_index_nnz(p) * cfg.block * cfg.block * 2
    monkeypatch.setenv("LG_KEEP_DS_MAX_GB", "%.6f" % (0.5 * ds / 1e9))
    assert lg.bwd_variant_name(p) == "two_pass"
    inp = synth.make_attn_inputs(cfg, "cuda", seed=15, with_do=True)
    o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"])
    ref = dict(zip(("o", "lse", "dq", "dk", "dv"), (o, lse) + lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"])))
    host = {k: v.cpu().pin_memory() for k, v in inp.items()}
    out = {n: torch.zeros(t.shape, dtype=t.dtype).pin_memory() for n, t in ref.items()}
    lg.sparse_attn_fwd_bwd_host(lg.params_of(cfg), host, out, head_groups=4)
    torch.cuda.synchronize()
    for name, t in ref.items():
        assert torch.equal(out[name], t.cpu()), name
