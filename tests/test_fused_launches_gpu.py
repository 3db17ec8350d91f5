"""The fused entry's inference rows and panel rows in one launch."""
import pytest
import torch

from paper_2512_23087_b200 import binding, inputs

import test_fused_gpu as fused

pytestmark = pytest.mark.gpu
W = inputs.WORKLOADS["c4_fused_lmhead"]


def _call(b, rho=1e-2, **kw):
    r = binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, rho, b.upstream, infer_logits=b.infer, **kw)
    torch.cuda.synchronize()
    assert r.workspace[:4].view(torch.int32).item() == 0
    return r


# inference rows in granules and, from an odd vocabulary, in pieces; one partial wave and several
@pytest.mark.parametrize("T,V", [(129, 4100), (300, 6016), (300, 6001), (700, 9001)])
def test_rows_of_both_policies_in_one_launch(T, V):
    """Several panels have a launch for the inference rows: every result of a token is the same, bit for bit."""
    b = inputs.make_fused(W, seed=V, device=fused.DEV, T=T, H=64, V=V)
    b.ids[0], b.ids[1] = -1, V
    one, several = _call(b), _call(b, panel_rows=128)
    for x, y in ((one.train, several.train), (one.infer, several.infer)):
        for n in ("max", "lse", "lse_safe", "logp", "logp_mp", "comp_mp", "count", "log_cov"):
            assert torch.equal(getattr(x, n).view(torch.int32), getattr(y, n).view(torch.int32)), n
    assert torch.equal(one.log_ratio.view(torch.int32), several.log_ratio.view(torch.int32))
    assert torch.equal(one.flags, several.flags)
