"""The forward at D = 64 (two CTAs per SM, halves worked 32 columns at a time): scores whose maximum moves late, in
either 32-column chunk of a half, lengths around the tiles' edges, masks whose bounds fall inside a chunk."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import lg_oracle as O
from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu
TOL_LSE = 1e-3                     # the parity tests' bound


@pytest.fixture(scope="module")
def lg():
    from paper_2410_01485_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("L", [1, 63, 257, 1000])
@pytest.mark.parametrize("block,exact", [(64, False), (64, True), (128, False)])
def test_rising_scores_and_ragged_lengths(lg, L, block, exact):
    cfg = replace(synth.CFG1, name="d64", L=L, D=64, Hq=4, Hkv=2, block=block, sink_tokens=block, window_tokens=2 * block,
                  window_exact=exact)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=L)
    k = inp["k"]
    # keys 20, 52 (the two chunks of a half), 300 and 900 answer every query with scores far above all earlier ones, so
    # that the running reference moves by more than 2^8 in one half, several times
    for i, at in enumerate((20, 52, 300, 900)):
        if at < L:
            k[:, :, at] = inp["q"][:, ::2, min(L - 1, at + 40)] * (1.5 + i)
    ws = lg.attn_workspace(lg.params_of(cfg), False)
    o, lse = lg.lg_sparse_attn_fwd(lg.params_of(cfg), inp["q"], k, inp["v"], workspace=ws)
    assert lg.lg_last_status(ws) == 0
    Oo, LSE = O.attn_forward(synth.to_f64(inp["q"][0]), synth.to_f64(k[0]), synth.to_f64(inp["v"][0]), O.Pattern.of(cfg), 1.0 / 8)
    # A few keys carry these rows, so the roundings do not average out: the result's own (at most 2^-8 |O|) and those of
    # the probabilities before the second product (at most 2^-8 each, together 2^-8 sum p |v|); 1e-3 for the fp32 sums.
    Av, _ = O.attn_forward(synth.to_f64(inp["q"][0]), synth.to_f64(k[0]), np.abs(synth.to_f64(inp["v"][0])), O.Pattern.of(cfg), 1.0 / 8)
    err = np.abs(synth.to_f64(o[0]) - Oo)
    assert (err <= 2.0 ** -8 * (np.abs(Oo) + Av) + 1e-3).all(), err.max()
    assert np.abs(synth.to_f64(lse[0]) - LSE).max() <= TOL_LSE


@pytest.mark.parametrize("L", [1, 63, 257, 1000])
@pytest.mark.parametrize("block,exact", [(64, False), (64, True), (128, False)])
def test_both_forms_give_the_same_bits(lg, L, block, exact):
    """A batch of eight runs two CTAs on an SM, one of its sequences has an SM per CTA (fwd_two_ctas, csrc/lg_host.h):
    groups of a problem's heads or sequences must come out as in the whole."""
    cfg = replace(synth.CFG1, name="forms", B=8, L=L, D=64, Hq=32, Hkv=8, block=block, sink_tokens=block, window_tokens=2 * block,
                  window_exact=exact)
    inp = synth.make_attn_inputs(cfg, "cuda", seed=L)
    k = inp["k"]
    for i, at in enumerate((20, 52, 300, 900)):
        if at < L:
            k[:, :, at] = inp["q"][:, ::4, min(L - 1, at + 40)] * (1.5 + i)
    o, lse = lg.lg_sparse_attn_fwd(lg.params_of(cfg), inp["q"], k, inp["v"])
    one = replace(cfg, B=1)
    for b in range(cfg.B):
        ob, lb = lg.lg_sparse_attn_fwd(lg.params_of(one), *(t[b:b + 1] for t in (inp["q"], k, inp["v"])))
        assert torch.equal(ob[0], o[b]) and torch.equal(lb[0], lse[b])
