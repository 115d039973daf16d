"""The forward with super-tiles cut along their keys (few heads, long rows): both block
and head sizes, every pattern, ragged lengths, pieces whose references differ widely;
chunks against a ring; repeated calls; a workspace prepared for other head counts; NaN; the
host-buffer step in head groups.  (test_fwd_split_rule.py checks that these problems are cut.)"""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import lg_oracle as O
from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu
TOL_O, TOL_LSE = 1e-2, 1e-3        # the parity tests' bounds


@pytest.fixture(scope="module")
def lg():
    from paper_2410_01485_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


CASES = [
    replace(synth.CFG1, name="full_64", mode=synth.MODE_FULL_CAUSAL, L=1999, D=128, Hq=4, Hkv=2, block=64),
    replace(synth.CFG1, name="full_128", mode=synth.MODE_FULL_CAUSAL, L=2048, D=64, Hq=2, Hkv=1, block=128, B=2),
    replace(synth.CFG1, name="window_64", L=3001, D=64, Hq=2, Hkv=2, block=64, sink_tokens=128, window_tokens=1344, window_exact=True),
    replace(synth.CFG1, name="window_128", L=2900, D=128, Hq=2, Hkv=1, block=128, sink_tokens=0, window_tokens=1536),
    replace(synth.CFG1, name="comb_64", mode=synth.MODE_STRIDED_LOCAL, stride_blocks=2, local_blocks=9, L=3500, D=128, Hq=2, Hkv=2, block=64),
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_cut_tiles_parity(lg, cfg):
    p = lg.params_of(cfg)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=3)
    for i, at in enumerate((40, 700, 1500)):               # the pieces' references differ widely
        inp["k"][:, :, at] = inp["q"][:, ::cfg.Hq // cfg.Hkv, at + 100] * (0.5 + 0.5 * i)
    ws = lg.attn_workspace(p, False)
    o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
    lg.lg_sparse_attn_prepare(p, ws, False)
    for _ in range(3):                                     # the pieces are added in a fixed order
        o2, lse2 = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
        assert torch.equal(o, o2) and torch.equal(lse, lse2)
    assert lg.lg_last_status(ws) == 0
    scale = 1.0 / np.sqrt(cfg.D)
    for b in range(cfg.B):
        pat = O.Pattern.of(cfg)
        q, k, v = (synth.to_f64(inp[x][b]) for x in ("q", "k", "v"))
        Oo, LSE = O.attn_forward(q, k, v, pat, scale)
        Av, _ = O.attn_forward(q, k, np.abs(v), pat, scale)
        # (rows that a few keys carry: the roundings of the result and of the probabilities, 2^-8 each)
        err = np.abs(synth.to_f64(o[b]) - Oo)
        assert (err <= 2.0 ** -8 * (np.abs(Oo) + Av) + 1e-3).all(), err.max()
        assert np.abs(synth.to_f64(lse[b]) - LSE).max() <= TOL_LSE


def test_one_workspace_serves_both_directions_and_other_head_counts(lg):
    """Lists prepared for 8 heads with a backward; forward + backward of 4 and of 8 heads on them, in turn."""
    cfg = replace(synth.CFG1, name="both", mode=synth.MODE_FULL_CAUSAL, L=1999, D=128, Hq=8, Hkv=8, block=64)
    few = replace(cfg, Hq=4, Hkv=4)
    ws = max((lg.attn_workspace(lg.params_of(c), True) for c in (cfg, few)), key=lambda t: t.numel())
    lg.lg_sparse_attn_prepare(lg.params_of(cfg), ws, True)
    for _ in range(2):
        for c in (few, cfg):
            inp = synth.make_attn_inputs(c, "cuda", seed=6, with_do=True)
            p = lg.params_of(c)
            p.lists_prepared = 1
            o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
            got = (o, lse) + lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"], workspace=ws)
            assert lg.lg_last_status(ws) == 0
            p = lg.params_of(c)
            o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"])
            ref = (o, lse) + lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"])
            assert all(torch.equal(x, y) for x, y in zip(got, ref))


def test_nan_in_a_query_stays_in_its_row(lg):
    cfg = CASES[0]
    p = lg.params_of(cfg)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=8)
    ref, _ = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"])
    inp["q"][0, 1, 1500, 3] = float("nan")
    o, _ = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"])
    assert bool(torch.isnan(o[0, 1, 1500]).all())
    o[0, 1, 1500] = ref[0, 1, 1500]
    assert torch.equal(o, ref)


GROUPS = replace(synth.CFG1, name="groups", mode=synth.MODE_FULL_CAUSAL, L=2500, D=128, Hq=8, Hkv=4, block=64)


@pytest.mark.parametrize("D", [64, 128])
def test_head_groups_of_the_host_step_cut_like_the_whole(lg, D):
    """8 / 4 heads are cut otherwise than 2 / 1 of them alone would be."""
    cfg = replace(GROUPS, D=D)
    p = lg.params_of(cfg)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=12, with_do=True)
    o, lse = lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"])
    host = {k: v.cpu().pin_memory() for k, v in inp.items()}
    ref = dict(zip(("o", "lse", "dq", "dk", "dv"), (o, lse) + lg.lg_sparse_attn_bwd(p, inp["q"], inp["k"], inp["v"], o, lse, inp["do"])))
    out = {n: torch.zeros(t.shape, dtype=t.dtype).pin_memory() for n, t in ref.items()}
    lg.sparse_attn_fwd_bwd_host(lg.params_of(cfg), host, out, head_groups=4)
    torch.cuda.synchronize()
    for name, t in ref.items():
        assert torch.equal(out[name], t.cpu()), name


def test_chunk_whose_tiles_are_cut(lg):
    """One sequence, 300 tokens against a full ring: two super-tiles of 4 heads, cut; decoded token by token for comparison."""
    B, Hq, Hkv, D, sink, W, T, n = 1, 4, 2, 128, 64, 2048, 300, 5000
    p = lg.decode_params(B, Hq, Hkv, D, sink, W)
    g = torch.Generator(device="cuda").manual_seed(8)
    kc, vc = (torch.randn(B, Hkv, sink + W, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    k, v = (torch.randn(B, Hkv, T, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    q = torch.randn(B, Hq, T, D, generator=g, device="cuda").to(torch.bfloat16)
    o, lse = lg.lg_chunk_prefill(p, q, k, v, kc, vc, n)
    for t in range(T):
        lg.lg_kv_ring_append(p, kc, vc, k[:, :, t:t + 1].contiguous(), v[:, :, t:t + 1].contiguous(), torch.tensor([n + t], device="cuda"))
        if t in (0, 1, 63, 64, 100, 255, 256, 299):
            od, ld = lg.lg_sparse_decode(p, q[:, :, t].contiguous(), kc, vc, torch.tensor([n + t + 1], device="cuda"))
            assert (od.float() - o[:, :, t].float()).abs().max() <= 2 * TOL_O     # both within TOL_O of the same value
            assert (ld - lse[:, :, t]).abs().max() <= 2 * TOL_LSE
