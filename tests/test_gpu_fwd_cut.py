"""Forwards whose super-tiles are cut, in workspaces and layouts other than their own: the last, short chunk of a prompt in the workspace of
its long ones, lists prepared for many heads, lists that two streams share, results written through strides, chunks of several
sequences with a block-aligned window, and the checked build.  (test_fwd_split_rule.py checks that these problems are cut.)"""
import importlib.util
from dataclasses import replace

import pytest
import torch

from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu
TOL_O, TOL_LSE = 1e-2, 1e-3        # the parity tests' bounds

FULL = replace(synth.CFG1, name="full", mode=synth.MODE_FULL_CAUSAL, L=1999, D=128, Hq=4, Hkv=2, block=64)
WINDOW = replace(synth.CFG1, name="window", L=2900, D=64, Hq=2, Hkv=1, block=128, sink_tokens=128, window_tokens=1536)
CHUNKS = [(1, 64, 8, 128, 4096, 100, 0), (2, 8, 2, 64, 2048, 200, 64)]       # B, Hq, Hkv, sink, window, T, block_tokens


@pytest.fixture(scope="module")
def lg():
    from paper_2410_01485_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("B,Hq,Hkv,sink,W,T,bt", CHUNKS, ids=str)
def test_short_chunk_in_the_workspace_of_long_ones(lg, B, Hq, Hkv, sink, W, T, bt):
    D, n = 128, 5000
    p = lg.decode_params(B, Hq, Hkv, D, sink, W, block_tokens=bt)
    g = torch.Generator(device="cuda").manual_seed(T)
    kc, vc = (torch.randn(B, Hkv, sink + W, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    k, v = (torch.randn(B, Hkv, T, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    q = torch.randn(B, Hq, T, D, generator=g, device="cuda").to(torch.bfloat16)
    ws = lg.chunk_prefill_workspace(p, 1500, 20000)
    o, lse = lg.lg_chunk_prefill(p, q, k, v, kc, vc, n, workspace=ws)
    assert lg.lg_last_status(ws) == 0
    count = torch.full((B,), n, dtype=torch.int64, device="cuda")
    for t in range(T):
        lg.lg_kv_ring_append(p, kc, vc, k[:, :, t:t + 1].contiguous(), v[:, :, t:t + 1].contiguous(), count + t)
        if t in (0, 63, 64, T - 1):
            od, ld = lg.lg_sparse_decode(p, q[:, :, t].contiguous(), kc, vc, count + t + 1)
            assert (od.float() - o[:, :, t].float()).abs().max() <= 2 * TOL_O     # both within TOL_O of the same value
            assert (ld - lse[:, :, t]).abs().max() <= 2 * TOL_LSE


def test_lists_prepared_for_many_heads(lg):
    many = replace(FULL, Hq=64, Hkv=64)
    ws = lg.attn_workspace(lg.params_of(many), False)
    lg.lg_sparse_attn_prepare(lg.params_of(many), ws, False)
    inp = synth.make_attn_inputs(FULL, "cuda", seed=4)
    p = lg.params_of(FULL)
    p.lists_prepared = 1
    got = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
    assert lg.lg_last_status(ws) == 0
    ref = lg.lg_sparse_attn_fwd(lg.params_of(FULL), inp["q"], inp["k"], inp["v"])
    assert all(torch.equal(x, y) for x, y in zip(got, ref))


def test_two_streams_share_prepared_lists(lg):
    """Prepared lists are read only: two layers' forwards may run side by side on one workspace."""
    p = lg.params_of(FULL)
    ws = lg.attn_workspace(p, False)
    inputs = [synth.make_attn_inputs(FULL, "cuda", seed=s) for s in (1, 2)]
    ref = [lg.lg_sparse_attn_fwd(p, i["q"], i["k"], i["v"]) for i in inputs]
    lg.lg_sparse_attn_prepare(p, ws, False)
    p.lists_prepared = 1
    out = [[(torch.empty_like(r[0]), torch.empty_like(r[1])) for _ in range(20)] for r in ref]
    streams = [torch.cuda.Stream() for _ in ref]
    torch.cuda.synchronize()
    for step in range(20):
        for s, i, o in zip(streams, inputs, out):
            with torch.cuda.stream(s):
                lg.lg_sparse_attn_fwd(p, i["q"], i["k"], i["v"], o=o[step][0], lse=o[step][1], workspace=ws)
    torch.cuda.synchronize()
    assert lg.lg_last_status(ws) == 0
    for r, outs in zip(ref, out):
        assert all(torch.equal(r[0], o) and torch.equal(r[1], lse) for o, lse in outs)


@pytest.mark.parametrize("cfg", [FULL, WINDOW], ids=lambda c: c.name)
def test_results_through_strides(lg, cfg):
    inp = synth.make_attn_inputs(cfg, "cuda", seed=5)
    o, lse = lg.lg_sparse_attn_fwd(lg.params_of(cfg), inp["q"], inp["k"], inp["v"])
    # [B, L, H, D] in memory, the rows apart
    room = torch.full((cfg.B, cfg.L, cfg.Hq, cfg.D + 8), 7.0, dtype=torch.bfloat16, device="cuda")
    view = room[..., :cfg.D].transpose(1, 2)
    q, k, v = (inp[x].transpose(1, 2).contiguous().transpose(1, 2) for x in ("q", "k", "v"))
    _, lse2 = lg.lg_sparse_attn_fwd(lg.params_of(cfg), q, k, v, o=view)
    assert torch.equal(view, o) and torch.equal(lse, lse2) and bool((room[..., cfg.D:] == 7.0).all())


@pytest.mark.parametrize("cfg", [FULL, WINDOW], ids=lambda c: c.name)
def test_checked_build(lg, cfg):
    from paper_2410_01485_b200 import build
    spec = importlib.util.spec_from_file_location("lg_binding_checked_cut", lg.__file__)
    checked = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(checked)
    checked.LIB_PATH = build.build(debug=True)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=6)
    out = []
    for b in (lg, checked):
        p = b.params_of(cfg)
        ws = b.attn_workspace(p, False)
        out.append(b.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws))
        assert b.lg_last_status(ws) == 0
    assert all(torch.equal(x, y) for x, y in zip(*out))


def test_captured(lg):
    """One kernel node, replayed on other inputs."""
    p = lg.params_of(FULL)
    ws = lg.attn_workspace(p, False)
    lg.lg_sparse_attn_prepare(p, ws, False)
    p.lists_prepared = 1
    inp, other = (synth.make_attn_inputs(FULL, "cuda", seed=s) for s in (7, 8))
    o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
    graph = torch.cuda.CUDAGraph()
    before = lg.kernel_launches()
    with torch.cuda.graph(graph):
        lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], o=o, lse=lse, workspace=ws)
    assert lg.kernel_launches() == before + 1
    for x in ("q", "k", "v"):
        inp[x].copy_(other[x])
    graph.replay()
    torch.cuda.synchronize()
    ref = lg.lg_sparse_attn_fwd(lg.params_of(FULL), other["q"], other["k"], other["v"])
    assert torch.equal(o, ref[0]) and torch.equal(lse, ref[1]) and lg.lg_last_status(ws) == 0
