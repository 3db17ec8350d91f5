"""Rows that start anywhere: odd vocabularies with their rows back to back, bases off the 32-byte grid,
and gradient matrices that lie differently than their logits.  The row kernels cut each row at its own
32-byte boundaries; the elements in front of the first and behind the last whole piece, and the pieces
themselves, must all be taken exactly once, and nothing outside the rows may be written."""
import contextlib
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2512_23087_b200 import binding, inputs

import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
W = inputs.WORKLOADS


def _place(x, ld, offset):
    """The same rows with stride `ld`, starting `offset` elements into a fresh buffer; outside them a huge logit."""
    T, V = x.shape
    buf = torch.full((offset + T * ld + 64,), 3.0e4, dtype=x.dtype, device=x.device)
    view = buf[offset:offset + T * ld].view(T, ld)[:, :V]
    view.copy_(x)
    return view


# V: below one piece, around one and two pieces, an odd middle size, several sweeps of a block;
# (ld - V, offset of the logits, offset of the gradient): alike, and alike only in some or no rows
@pytest.mark.parametrize("pad,offset,grad_pad,grad_offset", [(0, 0, 0, 0), (3, 5, 3, 5), (1, 8, 0, 3), (16, 1, 8, 0)])
@pytest.mark.parametrize("V", [5, 31, 47, 2999, 50021])
@pytest.mark.parametrize("dtype,grad_dtype", [("bf16", torch.bfloat16), ("f16", torch.float32), ("f32", torch.float32),
                                              ("f32", torch.bfloat16)])
@pytest.mark.parametrize("checks", [False, True], ids=["", "bounds"])
def test_rows_that_start_anywhere(dtype, grad_dtype, V, pad, offset, grad_pad, grad_offset, checks):
    T = 13
    w = dataclasses.replace(W["c0_small_f32"], dtype=dtype, head_boost=5.0)
    b = inputs.make_rows(w, seed=V + pad, device=DEV, T=T, V=V)
    train, infer = _place(b.train, V + pad, offset), _place(b.infer, V + pad + 2, offset + 1)
    b = dataclasses.replace(b, train=train, infer=infer)
    ld = V + grad_pad
    buf = torch.full((grad_offset + T * ld + 64,), 7.0, dtype=grad_dtype, device=DEV)
    grad = buf[grad_offset:grad_offset + T * ld].view(T, ld)[:, :V]

    def run(rho):
        res = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, upstream=b.upstream, grad_train=grad,
                                  want_mask=True)
        torch.cuda.synchronize()
        return res

    for rho in (1e-3, 0.0):
        buf.fill_(7.0)
        if checks:
            with binding.bounds_checking_library():
                res = run(rho)
                assert binding.dvp_debug_bounds_status() == 0, "an index was out of range"
        else:
            res = run(rho)
        parity.check_forward(res, b, rho, V, True)
        outside = torch.ones_like(buf, dtype=torch.bool)
        outside[grad_offset:grad_offset + T * ld].view(T, ld)[:, :V] = False
        assert (buf[outside] == 7.0).all(), "written outside the gradient's rows"


# few and long rows are shared by several blocks each
@pytest.mark.parametrize("pad,offset,grad_pad,grad_offset", [(0, 0, 0, 0), (3, 5, 3, 5), (1, 8, 0, 3), (16, 1, 8, 0)])
@pytest.mark.parametrize("T,V", [(13, 5), (13, 31), (13, 47), (13, 2999), (600, 4097), (3, 50021)])
@pytest.mark.parametrize("dtype,grad_dtype", [("bf16", torch.bfloat16), ("f16", torch.float32), ("f32", torch.float32),
                                              ("f32", torch.bfloat16)])
@pytest.mark.parametrize("checks", [False, True], ids=["", "bounds"])
def test_backward_rows_that_start_anywhere(dtype, grad_dtype, T, V, pad, offset, grad_pad, grad_offset, checks):
    w = dataclasses.replace(W["c0_small_f32"], dtype=dtype, head_boost=5.0)
    b = inputs.make_rows(w, seed=V + pad, device=DEV, T=T, V=V)
    b = dataclasses.replace(b, train=_place(b.train, V + pad, offset))
    ld = V + grad_pad
    for rho in (1e-3, 0.0):
        buf = torch.full((grad_offset + T * ld + 64,), 7.0, dtype=grad_dtype, device=DEV)
        grad = buf[grad_offset:grad_offset + T * ld].view(T, ld)[:, :V]
        saved = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer)
        with binding.bounds_checking_library() if checks else contextlib.nullcontext():
            binding.dvp_backward(b.train, b.ids, rho, b.upstream, saved, grad_train=grad)
            torch.cuda.synchronize()
            assert not checks or binding.dvp_debug_bounds_status() == 0, "an index was out of range"
        want = parity.run_oracle(b.train, b.infer, b.ids, rho, b.upstream)
        parity.check_grad(grad, want.grad, {})
        outside = torch.ones_like(buf, dtype=torch.bool)
        outside[grad_offset:grad_offset + T * ld].view(T, ld)[:, :V] = False
        assert (buf[outside] == 7.0).all(), "written outside the gradient's rows"


# the same with a finite mask (pruned sampled tokens have a gradient too), and with the entry of the sampled token formed from
# lse_safe
@pytest.mark.parametrize("pad,offset,grad_pad,grad_offset", [(3, 5, 3, 5), (1, 8, 0, 3)])
@pytest.mark.parametrize("T,V", [(13, 47), (600, 4097), (3, 50021)])
@pytest.mark.parametrize("dtype,grad_dtype", [("bf16", torch.bfloat16), ("f16", torch.float32), ("f32", torch.float32)])
@pytest.mark.parametrize("how", ["finite mask", "no comp"])
def test_backward_options_at_any_alignment(dtype, grad_dtype, T, V, pad, offset, grad_pad, grad_offset, how):
    w = dataclasses.replace(W["c0_small_f32"], dtype=dtype, head_boost=5.0)
    b = inputs.make_rows(w, seed=V + pad, device=DEV, T=T, V=V)
    b.ids[::4] = b.train[::4].float().argmin(1)   # pruned tokens
    b = dataclasses.replace(b, train=_place(b.train, V + pad, offset))
    kw = {"mask_value": -50.0} if how == "finite mask" else {}
    rho, ld = 1e-2, V + grad_pad
    buf = torch.full((grad_offset + T * ld + 64,), 7.0, dtype=grad_dtype, device=DEV)
    grad = buf[grad_offset:grad_offset + T * ld].view(T, ld)[:, :V]
    saved = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, **kw)
    binding.dvp_backward(b.train, b.ids, rho, b.upstream, saved, grad_train=grad, use_comp=how != "no comp", **kw)
    torch.cuda.synchronize()
    ids, up = b.ids.cpu().numpy(), b.upstream.cpu().numpy().astype(np.float64)
    if how == "finite mask":
        want = oracle.dvp_rows_listing(b.train.cpu().double().numpy(), ids, rho, -50.0, dtype=parity.ORACLE_DTYPE[b.train.dtype],
                                       upstream=up, threshold_in_storage_type=False)[1]
        got = grad
    else:
        want = parity.run_oracle(b.train, b.infer, b.ids, rho, b.upstream).grad
        # 1 - exp(z_a - lse_safe): one float32 rounding of lse_safe and the stored value's own
        at = torch.arange(T, device=DEV)
        own, at_own = grad[at, b.ids].cpu().double().numpy(), want[np.arange(T), ids]
        bound = 2e-6 * np.abs(up) * (1 + saved.train.lse_safe.abs().cpu().double().numpy())
        assert (np.abs(own - at_own) <= bound + parity.UNIT_ROUNDOFF[grad_dtype] * np.abs(at_own)).all()
        got = grad.clone()
        got[at, b.ids], want[np.arange(T), ids] = 0.0, 0.0
    parity.check_grad(got, want, {})
    outside = torch.ones_like(buf, dtype=torch.bool)
    outside[grad_offset:grad_offset + T * ld].view(T, ld)[:, :V] = False
    assert (buf[outside] == 7.0).all(), "written outside the gradient's rows"


@pytest.mark.parametrize("grad_pad", [0, 1])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("T,V", [(64, 50021), (2000, 4096)])
def test_backward_entries_have_one_arithmetic(T, V, dtype, grad_pad):
    """Entries of 16 bits are those of float32, rounded: forming them costs no digit."""
    w = dataclasses.replace(W["c2_bf16_fwdbwd"], dtype="bf16" if dtype == torch.bfloat16 else "f16")
    b = inputs.make_rows(w, seed=V, device=DEV, T=T, V=V)
    saved = binding.dvp_forward(b.train, b.ids, 0.0, infer_logits=b.infer)
    exact = binding.dvp_backward(b.train, b.ids, 0.0, b.upstream, saved, grad_dtype=torch.float32)
    buf = torch.empty(T, V + grad_pad, dtype=dtype, device=DEV)
    got = binding.dvp_backward(b.train, b.ids, 0.0, b.upstream, saved, grad_train=buf[:, :V])
    torch.cuda.synchronize()
    assert torch.equal(got, exact.to(dtype))


@pytest.mark.parametrize("cluster", [2, 4])
@pytest.mark.parametrize("V,grad_pad", [(151935, 0), (70001, 1)])
def test_clusters_share_rows_that_start_anywhere(V, grad_pad, cluster):
    b = inputs.make_rows(W["c2_bf16_fwdbwd"], seed=V, device=DEV, T=5, V=V)
    grad = torch.empty(5, V + grad_pad, dtype=torch.bfloat16, device=DEV)[:, :V]
    res = binding.dvp_forward(b.train, b.ids, 1e-4, infer_logits=b.infer, upstream=b.upstream, grad_train=grad,
                              want_mask=True, launch_hint=256 | (cluster << 24))
    torch.cuda.synchronize()
    parity.check_forward(res, b, 1e-4, V, True)
