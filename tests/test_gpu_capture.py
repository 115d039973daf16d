"""Calls captured into a CUDA graph (their kernels are launched overlapped) and calls on two streams at once: the same bits as
plain calls, also on a replay with other inputs in the same buffers."""
from dataclasses import replace

import pytest
import torch

from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lg():
    from paper_2410_01485_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


CASES = [
    replace(synth.CFG1, name="tiny"),
    replace(synth.CFG1, name="d128_ragged_gqa", L=777, D=128, Hq=8, Hkv=2),
    replace(synth.CFG1, name="d64_pairs_cut", L=3001, D=64, Hq=16, Hkv=2, sink_tokens=64, window_tokens=128),
    replace(synth.CFG1, name="strided", mode=synth.MODE_STRIDED_LOCAL, stride_blocks=4, local_blocks=2, L=1500, D=128, Hq=4, Hkv=1),
]


class Step:
    """A training step on fixed buffers; with documents its lists are built in the step."""

    def __init__(self, lg, cfg, docs=False, prepared=True):
        self.lg, self.rebuild = lg, docs
        self.ds = synth.make_doc_start(cfg.L, seed=3, mean_len=400)[None].cuda() if docs else None
        self.p = lg.params_of(cfg, doc_start=self.ds)
        self.inp = {k: torch.empty_like(v) for k, v in synth.make_attn_inputs(cfg, "cuda", seed=0, with_do=True).items()}
        self.ws = lg.attn_workspace(self.p, True)
        if prepared and not docs:
            lg.lg_sparse_attn_prepare(self.p, self.ws, True)
        i = self.inp
        self.o, self.lse = torch.empty_like(i["q"]), torch.empty(i["q"].shape[:3], device="cuda")
        self.grads = [torch.empty_like(i[x]) for x in "qkv"]

    def load(self, cfg, seed):
        for k, v in synth.make_attn_inputs(cfg, "cuda", seed=seed, with_do=True).items():
            self.inp[k].copy_(v)

    def __call__(self):
        i, lg = self.inp, self.lg
        if self.rebuild:
            lg.lg_sparse_attn_prepare(self.p, self.ws, True)
        lg.lg_sparse_attn_fwd(self.p, i["q"], i["k"], i["v"], o=self.o, lse=self.lse, workspace=self.ws)
        lg.lg_sparse_attn_bwd(self.p, i["q"], i["k"], i["v"], self.o, self.lse, i["do"], *self.grads, workspace=self.ws)

    def results(self):
        return [t.clone() for t in (self.o, self.lse, *self.grads)]


@pytest.mark.parametrize("docs, prepared", [(False, True), (False, False), (True, True)])
@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_captured_training_step(lg, cfg, docs, prepared):
    step = Step(lg, cfg, docs, prepared)
    want = {}
    for seed in (1, 2):
        step.load(cfg, seed)
        step()
        want[seed] = step.results()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        step()
        step()
    for seed in (2, 1, 2):
        step.load(cfg, seed)
        for t in (step.o, step.lse, *step.grads):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want[seed], step.results())), seed
    assert lg.lg_last_status(step.ws) == 0


def test_captured_serving_steps(lg):
    """A chunk against the ring, then append + decode, in one graph."""
    B, Hq, Hkv, D, sink, W, T, n = 2, 8, 2, 128, 64, 256, 100, 500
    p = lg.decode_params(B, Hq, Hkv, D, sink, W)
    g = torch.Generator(device="cuda").manual_seed(0)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    kc0, vc0 = r(B, Hkv, sink + W, D), r(B, Hkv, sink + W, D)
    kc, vc = kc0.clone(), vc0.clone()
    q, k, v, qd = r(B, Hq, T, D), r(B, Hkv, T, D), r(B, Hkv, T, D), r(B, Hq, D)
    before, after = (torch.full((B,), x, dtype=torch.int64, device="cuda") for x in (n, n + T))
    oc, lc = torch.empty_like(q), torch.empty(B, Hq, T, device="cuda")
    od, ld = torch.empty_like(qd), torch.empty(B, Hq, device="cuda")
    wc, wd = lg.chunk_prefill_workspace(p, T, n), lg.decode_workspace(p)

    def steps():
        lg.lg_chunk_prefill(p, q, k, v, kc, vc, n, o=oc, lse=lc, workspace=wc)
        lg.lg_kv_ring_append(p, kc, vc, k, v, before)
        lg.lg_sparse_decode(p, qd, kc, vc, after, o=od, lse=ld, workspace=wd)

    steps()
    want = [t.clone() for t in (oc, lc, kc, vc, od, ld)]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        steps()
    for _ in range(2):
        kc.copy_(kc0); vc.copy_(vc0)
        for t in (oc, lc, od, ld):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, (oc, lc, kc, vc, od, ld)))
    assert lg.lg_last_status(wc) == 0


def test_two_streams_at_once(lg):
    """Two steps with buffers and workspaces of their own, interleaved on two streams."""
    a, b = Step(lg, CASES[0]), Step(lg, CASES[2])
    a.load(CASES[0], 1); b.load(CASES[2], 2)
    a(); b()
    want = a.results(), b.results()
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        with torch.cuda.stream(sa):
            a(); a()
        with torch.cuda.stream(sb):
            b()
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(want[0], a.results()))
    assert all(torch.equal(x, y) for x, y in zip(want[1], b.results()))
