"""Decode steps whose counts are written by an ordinary kernel just ahead (other lengths, empty and negative ones among them) give what the
same steps give one by one, also for batches of more sequences than a block has threads.  (That kernel does not let the decode
start early; counts that change behind the decode's early look at them are in test_gpu_decode_counts.py.)"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lg():
    from paper_2410_01485_b200 import binding, build
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("B,Hq,Hkv,D,sink,W,bt", [
    (1, 8, 1, 128, 0, 4096, 0),
    (5, 16, 2, 64, 64, 960, 64),
    (300, 4, 2, 64, 0, 200, 0),
], ids=str)
def test_counts_of_the_kernel_before(lg, B, Hq, Hkv, D, sink, W, bt):
    p = lg.decode_params(B, Hq, Hkv, D, sink, W, block_tokens=bt)
    g = torch.Generator(device="cuda").manual_seed(B)
    kc, vc = (torch.randn(B, Hkv, sink + W, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    q = torch.randn(B, Hq, D, generator=g, device="cuda").to(torch.bfloat16)
    cap = sink + W
    counts = torch.randint(-1, 2 * cap, (20, B), generator=g, device="cuda")
    counts[3] = 0
    counts[4] = cap
    counts[5, ::2] = 1
    n = torch.zeros(B, dtype=torch.int64, device="cuda")
    ws = lg.decode_workspace(p)

    def steps(wait):
        out = []
        for t in range(20):
            torch.add(counts[t], 0, out=n)         # a kernel on the same stream, just ahead
            out.append(lg.lg_sparse_decode(p, q, kc, vc, n, workspace=ws))
            out.append(lg.lg_sparse_decode(p, q, kc, vc, n, workspace=ws))
            if wait:
                torch.cuda.synchronize()
        return out

    for (o, l), (o1, l1) in zip(steps(False), steps(True)):
        assert torch.equal(o, o1) and torch.equal(l, l1)
    out = steps(True)
    for t in range(20):
        empty = counts[t] <= 0
        assert bool((out[2 * t][1][empty] == -float("inf")).all()) and bool(torch.isfinite(out[2 * t][1][~empty]).all())
