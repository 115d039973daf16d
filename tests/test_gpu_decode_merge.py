"""The merge of a decode unit's records: any number of records a unit, records of CTAs whose slice is empty, head
groups that are not full, back-to-back append + decode steps (launched overlapped)."""
import numpy as np
import pytest
import torch

from oracle import lg_oracle as O
from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu
TOL_O, TOL_LSE = 1e-2, 1e-3        # the decode tests' bounds


@pytest.fixture(scope="module")
def lg():
    from paper_2410_01485_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("B,Hq,Hkv,D,cap,ns", [
    (1, 8, 1, 128, 512, [512]),            # 2 CTAs, 2 records
    (1, 5, 1, 128, 2304, [2304]),          # 9 records: one more than a batch of loads; 5 of 8 heads
    (1, 12, 1, 64, 4096, [4001]),          # two head groups, the second half full
    (1, 2, 2, 128, 8192, [8192]),          # 32 records a unit
    (1, 8, 1, 64, 40000, [39999]),         # more records than a warp has lanes, several times
    (1, 8, 1, 128, 8192, [5]),             # one tile for 32 CTAs: every slice but one is empty
    (3, 8, 2, 128, 1024, [1024, 0, 17]),   # a sequence without tokens, units of very different lengths
], ids=str)
def test_merge_of_records(lg, B, Hq, Hkv, D, cap, ns):
    p = lg.decode_params(B, Hq, Hkv, D, 0, cap)
    g = torch.Generator(device="cuda").manual_seed(cap + Hq)
    kc, vc = (torch.randn(B, Hkv, cap, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    q = torch.randn(B, Hq, D, generator=g, device="cuda").to(torch.bfloat16)
    n = torch.tensor(ns, dtype=torch.int64, device="cuda")
    ws = lg.decode_workspace(p)
    o, lse = lg.lg_sparse_decode(p, q, kc, vc, n, workspace=ws)
    o2, lse2 = lg.lg_sparse_decode(p, q, kc, vc, n, workspace=ws)      # the counters are re-armed, the order is fixed
    assert torch.equal(o, o2) and torch.equal(lse, lse2)
    for b in range(B):
        oo, ll = O.decode(synth.to_f64(q[b]), synth.to_f64(kc[b, :, :max(ns[b], 1)]), synth.to_f64(vc[b, :, :max(ns[b], 1)]), ns[b], 0, cap,
                          1.0 / np.sqrt(D))
        assert np.abs(synth.to_f64(o[b]) - oo).max() <= TOL_O
        if ns[b]:
            assert np.abs(synth.to_f64(lse[b]) - ll).max() <= TOL_LSE
        else:
            assert bool((lse[b] == -float("inf")).all())


def test_overlapped_append_and_decode_steps(lg):
    """Fifty append + decode steps queued without a wait give what the same steps give one by one."""
    B, Hq, Hkv, D, sink, W = 2, 8, 2, 128, 64, 448
    p = lg.decode_params(B, Hq, Hkv, D, sink, W)
    g = torch.Generator(device="cuda").manual_seed(3)
    k, v = (torch.randn(50, B, Hkv, 1, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    q = torch.randn(50, B, Hq, D, generator=g, device="cuda").to(torch.bfloat16)
    before = torch.tensor([500, 40], dtype=torch.int64, device="cuda") + torch.arange(50, device="cuda")[:, None]
    after = before + 1

    def steps(wait):
        kc, vc = (torch.full((B, Hkv, sink + W, D), 0.25, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        ws, out = lg.decode_workspace(p), []
        for t in range(50):
            lg.lg_kv_ring_append(p, kc, vc, k[t], v[t], before[t])
            out.append(lg.lg_sparse_decode(p, q[t], kc, vc, after[t], workspace=ws))
            if wait:
                torch.cuda.synchronize()
        return out, kc, vc

    (a, ka, va), (b, kb, vb) = steps(False), steps(True)
    assert torch.equal(ka, kb) and torch.equal(va, vb)
    assert all(torch.equal(x, y) for s, t in zip(a, b) for x, y in zip(s, t))
