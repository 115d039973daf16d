"""Memory that was a workspace before may hold the header's magic between words that were written over since (a list that ended
there): a call that starts on it reports nothing, and errors that a kernel left unread are still kept."""
import pytest
import torch

from paper_2410_01485_b200 import synth

pytestmark = pytest.mark.gpu
TIMEOUT = -5


@pytest.mark.parametrize("word,latched", [(0x278, 0), (0, 0x278), (0x3f803f80, 0), (0, 0x41004100), (0, 0)], ids=hex)
def test_stale_words(word, latched):
    from paper_2410_01485_b200 import binding as lg, build
    build.build()
    p = lg.params_of(synth.CFG1)
    ws = lg.attn_workspace(p, False)
    inp = synth.make_attn_inputs(synth.CFG1, "cuda", seed=1)
    lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)         # leaves the magic
    ws[:8].view(torch.int32).copy_(torch.tensor([word, latched], dtype=torch.int32))
    lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
    assert lg.lg_last_status(ws) == 0
    lg.lg_selftest_wait_timeout(ws)
    for _ in range(2):
        lg.lg_sparse_attn_fwd(p, inp["q"], inp["k"], inp["v"], workspace=ws)
    assert lg.lg_last_status(ws) == TIMEOUT and lg.lg_last_status(ws) == 0
