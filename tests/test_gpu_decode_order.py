"""The order in which the decode sums the products of a score: steps of 16 along the head dimension, one after the other."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("window", [64, 4096])
def test_scores_are_summed_along_the_head_dimension(D, window):
    from paper_2410_01485_b200 import binding as lg, build
    build.build()
    lg.load_library()
    p = lg.decode_params(1, 1, 1, D, 0, window, scale=1.0)
    q, k = (torch.zeros(1, 1, n, D, dtype=torch.bfloat16, device="cuda") for n in (1, window))
    q[0, 0, 0, [0, 16, 32]] = torch.tensor([2.0 ** 14, 1.0, 2.0 ** 14], dtype=torch.bfloat16, device="cuda")
    k[..., [0, 16, 32]] = torch.tensor([2.0 ** 14, 1.0, -2.0 ** 14], dtype=torch.bfloat16, device="cuda")
    _, lse = lg.lg_sparse_decode(p, q[:, :, 0].contiguous(), k, k, torch.ones(1, dtype=torch.int64, device="cuda"))
    # 2^28 + 1 is 2^28 in fp32, so the second product is lost before the third takes the first away; any other order keeps it
    assert lse.item() == 0.0
