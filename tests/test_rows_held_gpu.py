"""Small calls, whose rows are held in registers: at the lines of the rule that takes them, at the edges of a thread's, a
block's and a cluster's share of a row, and on rows that are not ordinary, against the oracle and the row kernel."""
import contextlib
import dataclasses

import pytest
import torch

from paper_2512_23087_b200 import binding, inputs

import oracle
import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
W = inputs.WORKLOADS
SIDE = ("max", "lse", "lse_safe", "logp", "logp_mp", "comp_mp", "count", "log_cov")
ROW_KERNEL = 256   # a launch hint leaves the call to the row kernel


def _batch(dtype, T, V, seed=3, ld=None):
    w = dataclasses.replace(W["c2_bf16_fwdbwd"], dtype=dtype)
    return inputs.make_rows(w, seed=seed, device=DEV, T=T, V=V, ld=ld)


def _call(b, rho, **kw):
    res = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, upstream=b.upstream, **kw)
    torch.cuda.synchronize()
    return res


# granules of 16 (8) elements: less than one, 64 threads of four and one more, 512 of four and one more (two blocks), the
# longest row of eight blocks and one beyond it; 512 tokens and one more
SIZES = [("bf16", 3, 1), ("f16", 5, 15), ("f32", 2, 9), ("bf16", 7, 4096), ("bf16", 7, 4097 + 15), ("f16", 4, 32768),
         ("bf16", 4, 32769), ("f32", 4, 16384), ("f32", 3, 16393), ("bf16", 1, 262144), ("bf16", 2, 262145), ("f32", 2, 100003),
         ("bf16", 512, 515), ("bf16", 513, 515), ("f32", 500, 1001),
         # five granules a thread: two blocks of them, one block full and one granule beyond it, where the chip is full
         ("bf16", 16, 151936), ("f32", 148, 20480), ("f32", 148, 20488), ("f16", 148, 40960), ("bf16", 1, 327680)]


@pytest.mark.parametrize("checks", [False, True], ids=["", "bounds"])
@pytest.mark.parametrize("dtype,T,V", SIZES)
def test_edges(dtype, T, V, checks):
    b = _batch(dtype, T, V)
    b.ids[0] = V - 1
    if T > 2:
        b.ids[1] = -1
    with binding.bounds_checking_library() if checks else contextlib.nullcontext():
        for rho in (1e-4, 0.0):
            res = _call(b, rho, want_mask=True)
            if checks:
                assert binding.dvp_debug_bounds_status() == 0, "an index was out of range"
            parity.check_forward(res, b, rho, V, True)


# one block a row with three granules a thread, with two, and the next rows, which have several without a gradient or with one
@pytest.mark.parametrize("dtype,T,V", [("bf16", 6, 24576), ("bf16", 6, 24577), ("f16", 40, 8209), ("f32", 6, 12288), ("f32", 6, 12289),
                                       ("bf16", 6, 16384), ("bf16", 6, 16385), ("f32", 40, 8192), ("f32", 6, 8193)])
def test_one_policy(dtype, T, V):
    b = _batch(dtype, T, V)
    for rho in (1e-4, 0.0):
        res = binding.dvp_forward(b.train, b.ids, rho, upstream=b.upstream)
        alone = binding.dvp_forward(b.train, b.ids, rho)
        torch.cuda.synchronize()
        want = parity.run_oracle(b.train, None, b.ids, rho, upstream=b.upstream)
        for r in (res, alone):
            parity.check_side(r.train, want.train, b.train, V, "train", {})
        parity.check_grad(res.grad_train, want.grad, {})


# one, two, four and eight blocks a row
@pytest.mark.parametrize("dtype,T,V", [("bf16", 148, 30001), ("f32", 300, 2003), ("f16", 50, 50021), ("f32", 50, 20003),
                                       ("bf16", 9, 30001), ("bf16", 25, 100001), ("f16", 5, 50021), ("f32", 3, 60000)])
@pytest.mark.parametrize("pad", [0, 3, 16])
def test_weights_and_gradient_rows_that_lie_differently(dtype, T, V, pad):
    b = _batch(dtype, T, V, ld=V + 5)
    grad = torch.full((T, V + pad), 7.0, dtype=b.train.dtype, device=DEV)
    weight = (oracle.WEIGHT_TRUNCATE, 0.0, 1.01)
    res = _call(b, 1e-3, grad_train=grad[:, :V], weight_kind=weight[0], weight_lo=weight[1], weight_hi=weight[2])
    parity.check_weighted(res, b, 1e-3, V, weight)
    assert (grad[:, V:] == 7).all()


@pytest.mark.parametrize("mask_value", [None, -50.0])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
def test_rows_that_are_not_ordinary(dtype, mask_value):
    """As the row kernel has them: what is infinite or no number with it is so here, the rest is equal up to the order of the
    sums (32-bit sums of 9,001 terms, and 16-bit entries that round the other way)."""
    V = 9001
    b = _batch(dtype, 9, V)
    low = torch.finfo(b.train.dtype).min
    for z in (b.train, b.infer):
        z[0] = float("-inf")
        z[1] = low
        z[2, 17] = float("inf")
        z[3, 4000] = float("nan")
        z[4, 1:] = float("-inf")
        z[5, :8999] = low
        z[6] = 2.5
    b.infer[7] = float("-inf")
    for rho in (1e-3, 0.0):
        got, want = (_call(b, rho, mask_value=mask_value, launch_hint=h) for h in (0, ROW_KERNEL))
        assert torch.equal(got.flags, want.flags)
        pairs = [(n, getattr(getattr(got, s), n), getattr(getattr(want, s), n)) for s in ("train", "infer") for n in SIDE]
        pairs += [("log_ratio", got.log_ratio, want.log_ratio), ("gradient", got.grad_train, want.grad_train)]
        for n, x, y in pairs:
            x, y = x.double(), y.double()
            if rho == 0.0:   # +inf - inf is no threshold: the count then is that of a kernel's own pieces
                x[2], y[2] = 0.0, 0.0
            assert torch.equal(torch.isnan(x), torch.isnan(y)) and torch.equal(torch.isinf(x), torch.isinf(y)), n
            x, y = (torch.nan_to_num(v, nan=0.0, posinf=1.0, neginf=-1.0) for v in (x, y))
            unit = {"f32": 1e-6, "bf16": 2.0 ** -7, "f16": 2.0 ** -10}[dtype] if n == "gradient" else 1e-6
            assert ((x - y).abs() <= unit * y.abs() + 2e-6).all(), n


# eight blocks a row (two-byte logits); five granules a thread; float32; rows of less than a block's threads
@pytest.mark.parametrize("dtype,V", [("bf16", 151936), ("bf16", 327680), ("f16", 50021), ("f32", 163840), ("f32", 30001),
                                     ("bf16", 2051)])
def test_full_sum_keeps_small_terms(dtype, V):
    """One token at 0 and all others at -17, where e^-17 = 0.69 * 2^-24 is lost when it is added to 1 by itself.  The sum that
    holds the 1 is rounded by half a unit, 2^-24, with each of the at most 8 pairs of its granule, 5 granules, the other half
    of the pair, the row's end, 5 exchanges in the warp, 4 slots a lane, 5 exchanges of those, the sampled token, and a few
    times in the logarithm."""
    train = torch.full((6, V), -17.0, dtype=inputs.torch_dtype(dtype), device=DEV)
    for t, k in enumerate((3, 40, 700, 1023, 2047, 2050)):
        train[t, k] = 0.0
    ids = torch.tensor([3, V - 1, 5, 1023, -1, 2050], device=DEV)
    bound = (8 + 5 + 1 + 1 + 5 + 4 + 5 + 1 + 4) * 2.0 ** -24
    z = train.double()
    lse = torch.logsumexp(z, 1)
    logp = z.gather(1, ids.clamp(min=0)[:, None])[:, 0] - lse
    one, two = (binding.dvp_forward(train, ids, 1e-3, **kw) for kw in ({}, dict(infer_logits=train.clone())))
    torch.cuda.synchronize()
    for side in (one.train, two.train, two.infer):
        assert (side.lse.double() - lse).abs().max().item() <= bound
        assert (side.log_cov.double() + lse).abs().max().item() <= bound   # the safe set is the one token: ln Z = -lse
        assert ((side.logp.double() - logp).abs() <= bound + 2.0 ** -24 * logp.abs())[ids >= 0].all()


# four blocks a row; one, of 512 threads, 128, 512, 256 and 64
@pytest.mark.parametrize("dtype,T,V", [("bf16", 6, 30000), ("bf16", 148, 32000), ("f16", 300, 8000), ("f32", 148, 16000),
                                       ("bf16", 148, 5003), ("f32", 500, 1001)])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("one_matrix", [False, True])
def test_place_of_the_inference_rows(dtype, T, V, weighted, one_matrix):
    """The gradient over the inference rows, which are read before: every result is that of a call with a gradient of its
    own.  The inference rows come from memory, the training rows from L2 where they are others."""
    b = _batch(dtype, T, V)
    if one_matrix:
        b.infer.copy_(b.train)
    kw = dict(weight_kind=binding.DVP_WEIGHT_TRUNCATE, weight_hi=1.01) if weighted else {}
    want = _call(b, 1e-3, **kw)
    infer, other = b.infer.clone(), torch.empty(1 << 26, device=DEV)
    for _ in range(3):
        infer.copy_(b.infer)
        other.zero_()   # twice L2
        train = infer if one_matrix else b.train.copy_(b.train.clone())
        got = binding.dvp_forward(train, b.ids, 1e-3, infer_logits=infer, upstream=b.upstream, grad_train=infer, **kw)
        torch.cuda.synchronize()
        assert torch.equal(got.grad_train, want.grad_train) and torch.equal(got.flags, want.flags)
        pairs = [(n, getattr(getattr(got, s), n), getattr(getattr(want, s), n)) for s in ("train", "infer") for n in SIDE]
        pairs += [("log_ratio", got.log_ratio, want.log_ratio)] + ([("weight", got.weight, want.weight)] if weighted else [])
        for n, x, y in pairs:
            assert torch.equal(x.view(torch.int32), y.view(torch.int32)), n
