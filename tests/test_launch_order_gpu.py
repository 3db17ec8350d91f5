"""Launches of a call may begin before their predecessor ends, and the fused entry's work beside one another.  Inputs that the
stream has not written yet when the call is made, calls that share a workspace, and captured calls must give bit for
bit what a call on finished inputs gives."""
import ctypes
import dataclasses

import pytest
import torch

from paper_2512_23087_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
W = inputs.WORKLOADS
SIDE = ("max", "lse", "lse_safe", "logp", "logp_mp", "comp_mp", "count", "log_cov")


def _results(r, more):
    return {**{f"{s}.{n}": getattr(getattr(r, s), n) for s in ("train", "infer") for n in SIDE},
            **{n: getattr(r, n) for n in ("log_ratio", "flags") + more}}


def _same(got, want):
    for n, x in want.items():
        assert torch.equal(torch.nan_to_num(got[n].float(), nan=9e9), torch.nan_to_num(x.float(), nan=9e9)), n


def _rows_call(b, weighted):
    kw = dict(weight_kind=binding.DVP_WEIGHT_TRUNCATE, weight_hi=1.01) if weighted else {}
    r = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, upstream=b.upstream, **kw)
    return _results(r, ("grad_train", "weight") if weighted else ("grad_train",))


def _fused_call(b, workspace=None):
    r = binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, 1e-3, b.upstream, infer_logits=b.infer,
                                                  panel_rows=128, workspace=workspace)
    return _results(r, ("d_hidden", "d_w")), r


def _refill(b, other, names):
    for n in names:
        getattr(b, n).copy_(getattr(other, n))


ROWS = ("train", "infer", "ids", "upstream")
FUSED = ("hidden", "w_vocab", "infer", "ids", "upstream")


@pytest.mark.parametrize("weighted", [False, True])
# both policies' rows in one launch; three launches (with weights two); two launches that fit the chip; one launch
@pytest.mark.parametrize("T,V", [(6, 151936), (900, 20000), (250, 20000), (50, 3001)])
def test_rows_behind_a_long_kernel(T, V, weighted):
    first, second = (inputs.make_rows(W["c2_bf16_fwdbwd"], seed=s, device=DEV, T=T, V=V) for s in (1, 2))
    want = _rows_call(second, weighted)
    torch.cuda.synchronize()
    torch.cuda._sleep(20_000_000)   # some ten milliseconds; the inputs arrive behind it
    _refill(first, second, ROWS)
    got = _rows_call(first, weighted)
    first.train.zero_(), first.infer.zero_(), first.ids.zero_()   # and are gone right after
    torch.cuda.synchronize()
    _same(got, want)


@pytest.mark.parametrize("T,H,V", [(300, 256, 6000), (130, 128, 4099)])
def test_fused_calls_share_a_workspace(T, H, V):
    """Several panels a call; two problems in turn through one workspace, inputs behind a long kernel, no synchronisation."""
    a, b, buf = (inputs.make_fused(W["c4_fused_lmhead"], seed=s, device=DEV, T=T, H=H, V=V) for s in (1, 2, 3))
    want_a, r = _fused_call(a)
    torch.cuda.synchronize()
    want_b, _ = _fused_call(b)
    torch.cuda.synchronize()
    workspace = torch.empty_like(r.workspace)
    torch.cuda._sleep(20_000_000)
    got = []
    for x in (a, b, a, b):
        _refill(buf, x, FUSED)
        got.append(_fused_call(buf, workspace)[0])
    torch.cuda.synchronize()
    assert workspace[:4].view(torch.int32).item() == 0
    for g, w in zip(got, (want_a, want_b, want_a, want_b)):
        _same(g, w)


# both policies' rows in one launch, in two (with and without the training rows first), and in three
@pytest.mark.parametrize("T,weighted", [(40, True), (40, False), (250, True), (250, False), (400, False)])
def test_captured_calls(T, weighted):
    a, b = (inputs.make_rows(W["c2_bf16_fwdbwd"], seed=s, device=DEV, T=T, V=20000) for s in (1, 2))
    fa, fb = (inputs.make_fused(W["c4_fused_lmhead"], seed=s, device=DEV, T=140, H=128, V=4000) for s in (1, 2))
    wants = []
    for x, f in ((a, fa), (b, fb)):
        wants.append((_rows_call(x, weighted), _fused_call(f)[0]))
        torch.cuda.synchronize()
    x, f = (inputs.make_rows(W["c2_bf16_fwdbwd"], seed=3, device=DEV, T=T, V=20000),
            inputs.make_fused(W["c4_fused_lmhead"], seed=3, device=DEV, T=140, H=128, V=4000))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):   # once outside the capture
        _rows_call(x, weighted), _fused_call(f)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        rows, (fused, keep) = _rows_call(x, weighted), _fused_call(f)
    for (rw, fw), (xr, xf) in zip(wants, ((a, fa), (b, fb))):
        _refill(x, xr, ROWS), _refill(f, xf, FUSED)
        graph.replay()
        torch.cuda.synchronize()
        _same(rows, rw), _same(fused, fw)


@pytest.mark.parametrize("V", [100, 2000, 20000])
def test_an_error_of_the_caller_is_left_alone(V):
    """A call that succeeds says nothing about errors that the caller has yet to read, and clears none."""
    b = inputs.make_rows(W["c2_bf16_fwdbwd"], seed=1, device=DEV, T=4, V=V)
    _rows_call(b, False)
    torch.cuda.synchronize()
    runtime = ctypes.CDLL("libcudart.so.12")   # the one that torch and the library have loaded
    assert runtime.cudaGetLastError() == 0
    invalid_device = runtime.cudaSetDevice(1000)
    assert invalid_device != 0 and runtime.cudaPeekAtLastError() == invalid_device
    _rows_call(b, False)
    assert runtime.cudaGetLastError() == invalid_device
    assert runtime.cudaGetLastError() == 0
    torch.cuda.synchronize()


# one launch; the training rows first and the inference rows waiting for them; three launches
@pytest.mark.parametrize("T", [40, 250, 400])
def test_log_ratio_of_odd_rows_in_every_order(T):
    """Rows that are not finite have no meaning, but a token that the flags call a member is not given the ratio of a pruned
    one, whichever launch forms it: with the gradient as without it."""
    V = 20000
    b = inputs.make_rows(dataclasses.replace(W["c2_bf16_fwdbwd"], dtype="f16"), seed=4, device=DEV, T=T, V=V)
    a = b.ids[:6].long()
    inf = float("inf")
    b.train[0, a[0]] = inf                        # overflowed logits of sampled tokens
    b.infer[1, a[1]] = inf
    b.train[2, a[2]] = b.infer[2, a[2]] = inf
    b.train[3, a[3]] = b.infer[3, a[3]] = -inf    # with rho = 0 every token is safe
    b.train[4] = -inf
    b.train[5, a[5]] = -inf
    for rho in (1e-3, 0.0):
        with_grad = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, upstream=b.upstream)
        without = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer)
        torch.cuda.synchronize()
        assert torch.equal(with_grad.flags, without.flags)
        x, y = with_grad.log_ratio, without.log_ratio
        odd = ~torch.isfinite(y)
        assert torch.equal(odd, ~torch.isfinite(x)) and odd[:6].sum() >= 4
        assert torch.equal(torch.nan_to_num(x[odd], nan=9e9), torch.nan_to_num(y[odd], nan=9e9))
        assert ((x - y)[~odd].abs() <= 1e-5).all()   # sums over other partial sums


@pytest.mark.parametrize("T", [4, 40, 250, 400])
def test_masks_of_the_inference_rows_before_the_gradient_takes_their_place(T):
    b = inputs.make_rows(W["c2_bf16_fwdbwd"], seed=5, device=DEV, T=T, V=20000)
    want = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, upstream=b.upstream, want_mask=True)
    torch.cuda.synchronize()
    got = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, upstream=b.upstream, grad_train=b.infer,
                              want_mask=True)
    torch.cuda.synchronize()
    assert torch.equal(got.infer.mask, want.infer.mask) and torch.equal(got.train.mask, want.train.mask)
    assert torch.equal(got.infer.count, want.infer.count) and torch.equal(got.flags, want.flags)
