"""The two forms of the ring append on both sides of the lines between them: calls as long as the ring and one token longer, calls of
as many blocks as the early form takes and one more."""
import pytest
import torch

pytestmark = pytest.mark.gpu
B = 3
LONGEST_EARLY = 4 * 148 * 8 * 256 // (B * 8)     # tokens of one head of 64 that fill the early form's blocks


@pytest.mark.parametrize("Hkv,D,sink,window,T", [
    (2, 128, 64, 448, 448),
    (2, 64, 64, 448, 449),
    (1, 64, 0, 64, LONGEST_EARLY),
    (1, 64, 0, 64, LONGEST_EARLY + 1),
    (1, 128, 192, 320, LONGEST_EARLY),
    (1, 128, 0, LONGEST_EARLY, LONGEST_EARLY),
], ids=str)
def test_append_equals_the_last_writer_of_each_slot(Hkv, D, sink, window, T):
    from paper_2410_01485_b200 import binding as lg, build
    build.build()
    lg.load_library()
    before = [0, 100, -1]
    p = lg.decode_params(B, Hkv, Hkv, D, sink, window)
    g = torch.Generator(device="cuda").manual_seed(T)
    k, v = (torch.randn(B, Hkv, T, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    kc, vc = (torch.full((B, Hkv, sink + window, D), x, dtype=torch.bfloat16, device="cuda") for x in (-1.0, -2.0))
    kr, vr = kc.clone(), vc.clone()
    lg.lg_kv_ring_append(p, kc, vc, k, v, torch.tensor(before, dtype=torch.int64, device="cuda"))
    for b, n in enumerate(before):
        if n < 0:
            continue
        j = torch.arange(n, n + T, device="cuda")
        j = j[(j < sink) | (j >= n + T - window)]           # the last token of each slot
        slot = torch.where(j < sink, j, sink + (j - sink) % window)
        kr[b][:, slot], vr[b][:, slot] = k[b][:, j - n], v[b][:, j - n]
    assert torch.equal(kc, kr) and torch.equal(vc, vr)
