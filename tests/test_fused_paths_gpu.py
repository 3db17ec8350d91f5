"""Paths of the fused entry that depend on sizes and alignment: inference rows off the 32-byte grid, the panel's rows with
one or two partial sums a thread, the default panel and the workspace that it fits."""
import ctypes
import dataclasses

import pytest
import torch

from paper_2512_23087_b200 import binding, inputs

import parity
import test_fused_gpu as fused

pytestmark = pytest.mark.gpu
DEV = fused.DEV
W = inputs.WORKLOADS["c4_fused_lmhead"]


# few rows are taken in pieces of 4 bytes, more in pieces of 16; rows of less than a piece, of one, and of several strips of
# 512 elements with an end of their own
@pytest.mark.parametrize("pad,offset", [(0, 1), (1, 0), (3, 5), (8, 8)])
@pytest.mark.parametrize("T,V", [(24, 3), (24, 5), (24, 1025), (24, 9001), (600, 9), (600, 517), (600, 4099)])
@pytest.mark.parametrize("checks", [False, True], ids=["", "bounds"])
def test_inference_rows_that_start_anywhere(T, V, pad, offset, checks):
    b = inputs.make_fused(W, seed=V, device=DEV, T=T, H=64, V=V)
    b.ids[0], b.ids[1] = -1, V
    ld = V + pad
    buf = torch.full((offset + T * ld + 64,), 3.0e4, dtype=torch.bfloat16, device=DEV)
    infer = buf[offset:offset + T * ld].view(T, ld)[:, :V]
    infer.copy_(4 * b.infer)   # some of the tokens below the threshold
    for rho in (1e-2, 0.0):
        def run():
            r = binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, rho, b.upstream, infer_logits=infer)
            torch.cuda.synchronize()
            return r
        if checks:
            with binding.bounds_checking_library():
                r = run()
                assert binding.dvp_debug_bounds_status() == 0, "an index was out of range"
        else:
            r = run()
        ids = b.ids.clone()
        ids[1] = -1   # the oracle's name for a row without a token
        want = parity.run_oracle(infer.contiguous(), None, ids, rho)
        parity.check_side(r.infer, want.train, infer, V, "infer", {})
        assert r.flags[0].item() & binding.DVP_FLAG_NO_ID and r.flags[1].item() & binding.DVP_FLAG_BAD_ID


@pytest.mark.parametrize("T,H,V", [(591, 64, 4099), (592, 64, 4099), (600, 64, 4096), (700, 64, 1003), (600, 64, 7)])
def test_panel_rows(T, H, V):
    batch, res, want, rerun = fused._run_fused(T, H, V, 1e-2, seed=T + V)
    fused._check_fused(batch, 1e-2, res, want, V, rerun=rerun)


# several K ranges for d_hidden; several panels; a whole number of tiles
@pytest.mark.parametrize("T,H,V,panel", [(200, 100, 3000, 0), (300, 33, 2051, 128), (64, 260, 4096, 0)])
def test_hidden_sizes_that_are_no_multiple_of_8(T, H, V, panel):
    """W is transposed for d_hidden then.  The strides are multiples of 8, and what lies between the rows is neither read nor
    written."""
    rho, ld = 1e-2, (H + 7) // 8 * 8
    b = inputs.make_fused(W, seed=V, device=DEV, T=T, H=H, V=V)

    def padded(rows, fill, like=None):
        m = torch.full((rows, ld), fill, dtype=torch.float32 if like is None else like.dtype, device=DEV)
        if like is not None:
            m[:, :H] = like
        return m
    hidden, w = padded(T, 3.0e4, b.hidden), padded(V, 3.0e4, b.w_vocab)
    b = dataclasses.replace(b, hidden=hidden[:, :H], w_vocab=w[:, :H])

    def rerun(upstream):
        d_hidden, d_w = padded(T, 7.0), padded(V, 7.0)
        a, res = binding._fused_args(b.hidden, b.w_vocab, b.ids, rho, upstream, b.infer, d_w[:, :H], False, panel, None, True)
        res.d_hidden, a.d_hidden, a.ld_dh = d_hidden[:, :H], d_hidden.data_ptr(), ld
        workspace = torch.empty(binding.dvp_workspace_bytes(binding.DVP_ENTRY_FUSED_LMHEAD, a), dtype=torch.uint8, device=DEV)
        a.workspace, a.workspace_bytes = workspace.data_ptr(), workspace.numel()
        assert binding.load_library().dvp_fused_lmhead_forward_backward(ctypes.byref(a)) == binding.DVP_OK
        torch.cuda.synchronize()
        assert workspace[:4].view(torch.int32).item() == 0
        assert (d_hidden[:, H:] == 7).all() and (d_w[:, H:] == 7).all()
        return res
    res = rerun(b.upstream)
    want, _ = fused._oracle_with_the_devices_set(b, rho, res)
    fused._check_fused(b, rho, res, want, V, rerun=rerun)


def test_default_panel_and_its_workspace():
    """A small vocabulary has panels of more than 4096 tokens by default; a workspace for 4096 is still enough."""
    T, H, V = 4300, 64, 1000
    b = inputs.make_fused(W, seed=1, device=DEV, T=T, H=H, V=V)

    def call(**kw):
        r = binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, 1e-3, b.upstream, infer_logits=b.infer, **kw)
        torch.cuda.synchronize()
        assert r.workspace[:4].view(torch.int32).item() == 0
        return r
    one, two = call(), call(panel_rows=4096)
    assert one.workspace.numel() > two.workspace.numel()
    small = call(workspace=torch.empty_like(two.workspace))
    assert torch.equal(small.d_w, two.d_w) and torch.equal(small.d_hidden, two.d_hidden)
    for n in ("lse", "logp_mp", "count", "log_cov"):
        assert torch.equal(getattr(one.train, n), getattr(two.train, n)), n
    # two sums of 2176 and 2124 products instead of 4096 and 204: a rounding for every 16 of them
    for x, y in ((one.d_w, two.d_w), (one.d_hidden, two.d_hidden)):
        assert ((x - y).norm(dim=1) <= 1e-5 * y.norm(dim=1).max()).all()
    with pytest.raises(binding.DvpError) as e:
        call(workspace=torch.empty(two.workspace.numel() - 256, dtype=torch.uint8, device=DEV))
    assert e.value.status == binding.DVP_ERR_WORKSPACE


# two sums of 34 slices, the last one of 12 tokens; two full ones; three; several panels of two
@pytest.mark.parametrize("T,panel", [(4300, 0), (8192, 0), (9000, 0), (20000, 8192)])
def test_long_sums_of_d_w(T, panel):
    """Terms of one sign, where an accumulator of the tensor core loses the more the more of them it takes: the default's
    error is that of panels of 4096."""
    H, V = 64, 1000
    b = inputs.make_fused(W, seed=T, device=DEV, T=T, H=H, V=V)
    b.hidden.copy_(b.hidden.abs()), b.upstream.copy_(b.upstream.abs() + 0.5), b.ids.zero_()
    z = b.hidden.double() @ b.w_vocab.double().t()
    want = -(torch.softmax(z, 1) * b.upstream.double()[:, None]).t() @ b.hidden.double()   # but for row 0

    def call(rows):
        r = binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, 0.0, b.upstream, panel_rows=rows)
        torch.cuda.synchronize()
        assert r.workspace[:4].view(torch.int32).item() == 0
        return r.d_w[1:]
    got, short = call(panel), call(4096)
    error, least = ((x.double() - want[1:]).norm().item() for x in (got, short))
    assert least <= 3e-5 * want[1:].norm().item()
    # n terms of about one size lose n^2 / 2 units: no sum is longer than 4096, and none than the others, so that theirs lose
    # no more than panels of 4096; 2 % for what is left of the terms' sizes
    assert error <= least * 1.02
    if T == 8192:
        assert torch.equal(got, short)
