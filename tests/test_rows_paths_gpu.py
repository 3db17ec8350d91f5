"""Paths of the row kernel that depend on sizes and on which outputs are asked for: a guess of the maximum that is far off,
rows split over several blocks, and the places through which ln pi^mp_infer(a) passes between the two launches."""
import copy
import ctypes
import dataclasses

import pytest
import torch

from paper_2512_23087_b200 import binding, inputs

import oracle
import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
W = inputs.WORKLOADS


def _check(batch, rho, V, **kw):
    res = binding.dvp_forward(batch.train, batch.ids, rho, infer_logits=batch.infer, upstream=batch.upstream,
                              want_mask=True, **kw)
    torch.cuda.synchronize()
    parity.check_forward(res, batch, rho, V, True)
    return res


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("threads", [64, 256])
def test_maximum_far_above_every_guess(dtype, threads):
    """One token 200 above all others: e^200 overflows in the units of any earlier guess.  It sits in the first step, in a
    later one, in the last piece, outside the pieces, or is (next to) the sampled token."""
    V, places = 40003, [0, 70, 17000, 25001, 39990, 40002]
    w = dataclasses.replace(W["c0_small_f32"], dtype=dtype, head_boost=0.0)
    b = inputs.make_rows(w, seed=5, device=DEV, T=2 * len(places), V=V)
    for i, k in enumerate(places):
        for t in (2 * i, 2 * i + 1):
            b.train[t, k] = 200.0
            b.infer[t, k] = 201.0
        b.ids[2 * i] = 12345
        b.ids[2 * i + 1] = min(k + 1, V - 1)
    for rho in (1e-3, 0.0):
        _check(b, rho, V, launch_hint=threads)


@pytest.mark.parametrize("dtype,T,V", [("bf16", 3, 151936), ("bf16", 150, 30001), ("f32", 2, 262144), ("f16", 40, 70000),
                                       ("f32", 600, 515), ("bf16", 1, 12289), ("bf16", 1, 12287)])
def test_default_shapes(dtype, T, V):
    """Few rows take several blocks each, many short ones small blocks; sizes on both sides of the rules' lines."""
    w = dataclasses.replace(W["c2_bf16_fwdbwd"], dtype=dtype)
    b = inputs.make_rows(w, seed=V, device=DEV, T=T, V=V)
    _check(b, 1e-4, V)


@pytest.mark.parametrize("parts", [2, 4, 8])
@pytest.mark.parametrize("V", [151936, 50021])
def test_rows_split_over_blocks_with_weights(V, parts):
    b = inputs.make_rows(W["c2_bf16_fwdbwd"], seed=parts, device=DEV, T=9, V=V)
    weight = (oracle.WEIGHT_TRUNCATE, 0.0, 1.01)
    res = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, upstream=b.upstream,
                              weight_kind=weight[0], weight_lo=weight[1], weight_hi=weight[2],
                              launch_hint=256 | (parts << 24))
    torch.cuda.synchronize()
    parity.check_weighted(res, b, 1e-3, V, weight)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("V", [1, 2, 5003])
@pytest.mark.parametrize("kept", [(), ("log_ratio",), ("flags",), ("weight",), ("log_ratio", "flags"), ("logp_mp_i",)])
def test_outputs_left_out(kept, V, weighted):
    """Any output may be missing; what is asked for is bit for bit what the full call gives."""
    w = W["c2_bf16_fwdbwd"]
    b = inputs.make_rows(dataclasses.replace(w, head_boost=2.0, head_max=1), seed=V, device=DEV, T=37, V=V)
    b.ids[3], b.ids[4] = -1, V
    kw = dict(weight_kind=binding.DVP_WEIGHT_TRUNCATE, weight_hi=1.01) if weighted else {}
    full = binding.dvp_forward(b.train, b.ids, 1e-2, infer_logits=b.infer, upstream=b.upstream, **kw)
    a = binding.ForwardArgs()
    a.struct_size, a.logits_dtype, a.grad_dtype = ctypes.sizeof(binding.ForwardArgs), binding.DVP_BF16, binding.DVP_BF16
    a.T, a.V, a.rho = 37, V, 1e-2
    a.ld_train = a.ld_infer = a.ld_grad = V
    grad = torch.full((37, V), 7.0, dtype=torch.bfloat16, device=DEV)
    a.train_logits, a.infer_logits, a.ids = b.train.data_ptr(), b.infer.data_ptr(), b.ids.data_ptr()
    a.upstream, a.grad_train = b.upstream.data_ptr(), grad.data_ptr()
    out = {n: torch.empty(37, dtype=torch.uint8 if n == "flags" else torch.float32, device=DEV) for n in kept}
    if "log_ratio" in out:
        a.log_ratio = out["log_ratio"].data_ptr()
    if "flags" in out:
        a.flags = out["flags"].data_ptr()
    if "weight" in out and weighted:
        a.weight_out = out["weight"].data_ptr()
    if "logp_mp_i" in out:
        a.infer.logp_mp = out["logp_mp_i"].data_ptr()
    if weighted:
        a.weight_kind, a.weight_hi = binding.DVP_WEIGHT_TRUNCATE, 1.01
    a.stream = torch.cuda.current_stream().cuda_stream
    assert binding.load_library().dvp_forward(ctypes.byref(a)) == binding.DVP_OK
    torch.cuda.synchronize()
    same = lambda x, y: torch.equal(torch.nan_to_num(x.float(), nan=9e9), torch.nan_to_num(y.float(), nan=9e9))
    assert same(grad, full.grad_train)
    if "log_ratio" in out:
        assert same(out["log_ratio"], full.log_ratio)
    if "flags" in out:
        assert same(out["flags"], full.flags)
    if "weight" in out and weighted:
        assert same(out["weight"], full.weight)
    if "logp_mp_i" in out:
        assert same(out["logp_mp_i"], full.infer.logp_mp)


@pytest.mark.parametrize("T,V,dtype", [(1, 5003, "bf16"), (148, 5003, "bf16"), (149, 5003, "bf16"), (592, 5003, "bf16"),
                                       (1300, 5003, "bf16"), (5, 151936, "bf16"), (37, 151936, "f16"), (74, 4096, "f32"),
                                       (75, 4096, "f32"), (9, 262143, "f32"),
                                       # rows longer than registers hold, in one launch and in two
                                       (18, 330001, "bf16"), (19, 330001, "bf16"), (9, 170001, "f32"), (10, 170001, "f32")])
def test_launches_of_a_call(T, V, dtype):
    """Both policies' rows in one launch, in two with either first, and in three, on both sides of the rules' lines.  Without
    some of the outputs, or with the gradient over the inference rows, the order is another one and the results the same."""
    w = dataclasses.replace(W["c2_bf16_fwdbwd"], dtype=dtype, head_boost=2.0, head_max=1)
    b = inputs.make_rows(w, seed=T, device=DEV, T=T, V=V)
    full = _check(b, 1e-2, V)
    again = binding.dvp_forward(b.train, b.ids, 1e-2, infer_logits=b.infer, upstream=b.upstream)
    over = b.infer.clone()
    placed = binding.dvp_forward(b.train, b.ids, 1e-2, infer_logits=over, upstream=b.upstream, grad_train=over)
    some, a = {"log_ratio": torch.empty(T, device=DEV), "flags": torch.empty(T, dtype=torch.uint8, device=DEV)}, binding.ForwardArgs()
    grad = torch.empty_like(b.train)
    code = binding._DTYPES[b.train.dtype]
    a.struct_size, a.logits_dtype, a.grad_dtype = ctypes.sizeof(binding.ForwardArgs), code, code
    a.T, a.V, a.rho = T, V, 1e-2
    a.ld_train = a.ld_infer = a.ld_grad = V
    a.train_logits, a.infer_logits, a.ids = b.train.data_ptr(), b.infer.data_ptr(), b.ids.data_ptr()
    a.upstream, a.grad_train = b.upstream.data_ptr(), grad.data_ptr()
    a.log_ratio, a.flags = some["log_ratio"].data_ptr(), some["flags"].data_ptr()
    a.stream = torch.cuda.current_stream().cuda_stream
    assert binding.load_library().dvp_forward(ctypes.byref(a)) == binding.DVP_OK
    torch.cuda.synchronize()
    for got in (again.grad_train, placed.grad_train, grad):
        assert torch.equal(got, full.grad_train)
    for n, x in some.items():
        assert all(torch.equal(y, getattr(full, n)) for y in (getattr(again, n), getattr(placed, n), x)), n
    for n in ("lse", "logp_mp", "log_cov", "count"):
        assert all(torch.equal(getattr(r.infer, n), getattr(full.infer, n)) for r in (again, placed)), n


# the last call in one launch and the first in two; the last whose rows are held in registers and the next
@pytest.mark.parametrize("T", [296, 297, 256, 257])
@pytest.mark.parametrize("dtype,V", [("bf16", 3001), ("f16", 2048), ("f32", 1500)])
def test_launches_without_a_gradient(T, dtype, V):
    b = inputs.make_rows(dataclasses.replace(W["c2_bf16_fwdbwd"], dtype=dtype), seed=T, device=DEV, T=T, V=V)
    res = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, want_mask=True)
    torch.cuda.synchronize()
    parity.check_forward(res, b, 1e-3, V, False)


@pytest.mark.parametrize("dtype,V,hint", [("bf16", 151936, 64), ("bf16", 151936, 256), ("bf16", 151936, 256 | (2 << 24)),
                                          ("f16", 50021, 64), ("f32", 262144, 512), ("f32", 40003, 64)])
def test_full_sum_keeps_small_terms(dtype, V, hint):
    """One token at 0 and all others at -17, where e^-17 = 0.69 * 2^-24 is lost when it is added to 1 by itself.  Each
    step's terms (two granules a thread) are added up first: one rounding of the sum a step, log2(512) when the threads' sums
    meet, and a few in the logarithm."""
    elem = 4 if dtype == "f32" else 2
    dt = inputs.torch_dtype(dtype)
    train = torch.full((6, V), -17.0, dtype=dt, device=DEV)
    for t, k in enumerate((3, 40, 700, 1023, 2047, 2050)):
        train[t, k] = 0.0
    ids = torch.tensor([3, V - 1, 5, 1023, -1, 2050], device=DEV)
    res = binding.dvp_forward(train, ids, 1e-3, launch_hint=hint)
    torch.cuda.synchronize()
    z = train.double()
    lse = torch.logsumexp(z, 1)
    threads, parts = hint & 0xffff, max(1, hint >> 24)
    steps = -(-V * elem // (64 * threads * parts))
    bound = (steps + 9 + 4) * 2.0 ** -24
    assert (res.train.lse.double() - lse).abs().max().item() <= bound
    assert (res.train.log_cov.double() + lse).abs().max().item() <= bound   # the safe set is the one token: ln Z = -lse
    has = ids >= 0
    logp = z[has].gather(1, ids[has, None])[:, 0] - lse[has]
    assert ((res.train.logp[has].double() - logp).abs() <= bound + 2.0 ** -24 * logp.abs()).all()


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("place", ["train", "infer"])
@pytest.mark.parametrize("T,V", [(5, 151936), (700, 20000), (37, 5003)])
def test_gradient_in_place_of_logits(T, V, place, weighted):
    """The gradient may take the place of either matrix, also where ln pi^mp_infer(a) has no output to pass through."""
    b = inputs.make_rows(W["c2_bf16_fwdbwd"], seed=T, device=DEV, T=T, V=V)
    kw = dict(weight_kind=binding.DVP_WEIGHT_TRUNCATE, weight_hi=1.01) if weighted else {}
    full = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, upstream=b.upstream, **kw)
    train, infer = b.train.clone(), b.infer.clone()
    grad = train if place == "train" else infer
    res = binding.dvp_forward(train, b.ids, 1e-3, infer_logits=infer, upstream=b.upstream, grad_train=grad, **kw)
    torch.cuda.synchronize()
    assert torch.equal(grad, full.grad_train) and torch.equal(res.log_ratio, full.log_ratio)
    assert torch.equal(res.train.lse, full.train.lse) and torch.equal(res.infer.lse, full.infer.lse)
    train.copy_(b.train), infer.copy_(b.infer)
    a = binding.ForwardArgs()
    a.struct_size, a.logits_dtype, a.grad_dtype = ctypes.sizeof(binding.ForwardArgs), binding.DVP_BF16, binding.DVP_BF16
    a.T, a.V, a.rho = T, V, 1e-3
    a.ld_train = a.ld_infer = a.ld_grad = V
    a.train_logits, a.infer_logits, a.ids = train.data_ptr(), infer.data_ptr(), b.ids.data_ptr()
    a.upstream, a.grad_train = b.upstream.data_ptr(), grad.data_ptr()
    if weighted:
        a.weight_kind, a.weight_hi = binding.DVP_WEIGHT_TRUNCATE, 1.01
    a.stream = torch.cuda.current_stream().cuda_stream
    assert binding.load_library().dvp_forward(ctypes.byref(a)) == binding.DVP_OK
    torch.cuda.synchronize()
    if weighted:   # one kernel for both rows, sums in another order: one rounding of bfloat16 apart at most
        d = (grad.float() - full.grad_train.float()).abs()
        assert (d <= 2.0 ** -7 * full.grad_train.float().abs() + 1e-30).all()
    else:
        assert torch.equal(grad, full.grad_train)


def test_out_names_the_tensors_it_holds():
    """A copy of a result owns its buffers, and a tensor put into a result takes the next call's values."""
    b, other = (inputs.make_rows(W["c2_bf16_fwdbwd"], seed=s, device=DEV, T=20, V=5003) for s in (1, 2))
    first = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, want_mask=True)
    kept = copy.deepcopy(first)
    want = binding.dvp_forward(other.train, other.ids, 1e-3, infer_logits=other.infer, want_mask=True)
    reused = copy.deepcopy(first)
    old, reused.infer.lse = reused.infer.lse, torch.zeros_like(reused.infer.lse)
    binding.dvp_forward(other.train, other.ids, 1e-3, infer_logits=other.infer, out=reused)
    torch.cuda.synchronize()
    for side in ("train", "infer"):
        for n in ("max", "lse", "lse_safe", "logp", "logp_mp", "comp_mp", "count", "log_cov", "mask"):
            assert torch.equal(getattr(getattr(reused, side), n), getattr(getattr(want, side), n)), n
            assert torch.equal(getattr(getattr(first, side), n), getattr(getattr(kept, side), n)), n
    assert torch.equal(reused.flags, want.flags) and torch.equal(reused.log_ratio, want.log_ratio)
    assert torch.equal(old, kept.infer.lse)


def test_numbers_beyond_their_c_type_are_the_library_s_to_refuse():
    b = inputs.make_rows(W["c2_bf16_fwdbwd"], seed=1, device=DEV, T=4, V=512)
    saved = binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer)
    f = inputs.make_fused(W["c4_fused_lmhead"], seed=1, device=DEV, T=4, H=64, V=512)
    for call in (lambda: binding.dvp_forward(b.train, b.ids, 1e-3, launch_hint=-1),
                 lambda: binding.dvp_forward(b.train, b.ids, 1e-3, infer_logits=b.infer, upstream=b.upstream, weight_kind=-1),
                 lambda: binding.dvp_backward(b.train, b.ids, 1e-3, b.upstream, saved, launch_hint=-1),
                 lambda: binding.dvp_fused_lmhead_forward_backward(f.hidden, f.w_vocab, f.ids, 1e-3, f.upstream,
                                                                   panel_rows=2 ** 31 + 128)):
        with pytest.raises(binding.DvpError) as e:
            call()
        assert e.value.status == binding.DVP_ERR_INVALID_ARG
    with pytest.raises(TypeError):
        binding.dvp_forward(b.train, b.ids, 1e-3, launch_hint=256.0)


@pytest.mark.parametrize("hint", [0, 64, 256, 256 | (2 << 24), 512 | (8 << 24)])
@pytest.mark.parametrize("V", [1, 31, 33, 1023, 1025, 32767, 70001])
def test_mask_words(V, hint):
    """Ends of words, of a warp's 32 words, and rows whose blocks share the mask; rho = 0 keeps everything."""
    b = inputs.make_rows(W["c2_bf16_fwdbwd"], seed=V, device=DEV, T=3, V=V)
    for rho in (1e-3, 0.0):
        res = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, want_mask=True, launch_hint=hint)
        torch.cuda.synchronize()
        for side, z in ((res.train, b.train), (res.infer, b.infer)):
            z = z.double().cpu()
            keep = z >= z.max(1, keepdim=True).values + (torch.log(torch.tensor(rho, dtype=torch.float64)) if rho else -float("inf"))
            assert (parity.unpack_mask(side.mask, V) == keep.numpy()).all()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("hint", [64, 256, 256 | (2 << 24), 256 | (4 << 24), 256 | (8 << 24)])
def test_maxima_that_climb(dtype, hint):
    """Maxima that rise by more than e^60 several times in a row, so that what was added up before them overflows, or nearly
    so: in one exchange's steps, in neighbouring ones, in the last steps, in the last element; sampled tokens elsewhere,
    at one of them, or none.  With several blocks a row each sees its own part of the climb."""
    V = 70001
    w = dataclasses.replace(W["c0_small_f32"], dtype=dtype, head_boost=0.0)
    b = inputs.make_rows(w, seed=11, device=DEV, T=8, V=V)
    places = [[40, 17000, 35000, 52000, 70000], [5000, 5001, 5040, 9000, 69990], [66000, 67000, 68000, 69000, 70000],
              [70000, 60000, 40000, 20000, 3], [30000, 30001, 30002, 30003, 30004], [16383, 16384, 32767, 32768, 65535],
              [0, 1024, 2048, 4096, 8192], [12000, 24000, 36000, 48000, 60000]]
    for t, ks in enumerate(places):
        for i, k in enumerate(ks):
            b.train[t, k] = 62.0 * (i + 1) + t
            b.infer[t, k] = 62.5 * (i + 1) + t
    b.ids[:] = torch.tensor([1, 5040, 70000, -1, 30003, 16384, -1, 60001], device=DEV)
    for rho in (1e-3, 0.0):
        _check(b, rho, V, launch_hint=hint)


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
def test_float32_gradient_entries(dtype):
    """Rows of two tokens that count, the sampled one and one exactly 1 above it: the other's entry is -g / (1 + e^-1), whose
    only errors are e^-1's, the sum's and the quotient's, a unit of 2^-24 each at most.  It is made of differences of
    logits that are exact here, so it is the same in every row, wherever the maximum lies."""
    T, V = 4096, 800
    g = torch.Generator(device=DEV).manual_seed(3)
    m = (torch.randint(64, 8192, (T, 1), generator=g, device=DEV).float() / 256).to(torch.bfloat16).float().clamp(min=4.0)
    m = torch.where(m >= 16, m.round(), (m * 16).round() / 16)   # m and m - 1 are exact in every type
    z = torch.full((T, V), -40.0, device=DEV)
    ids = torch.randint(0, V // 2, (T,), generator=g, device=DEV)
    other = V // 2 + torch.randint(0, V // 2, (T,), generator=g, device=DEV)
    z.scatter_(1, ids[:, None], m - 1)
    z.scatter_(1, other[:, None], m)
    z = z.to(inputs.torch_dtype(dtype))
    up = torch.ones(T, device=DEV)
    res = binding.dvp_forward(z, ids, 1e-3, upstream=up, grad_dtype=torch.float32)
    torch.cuda.synchronize()
    want = -1 / (1 + torch.exp(torch.tensor(-1.0, dtype=torch.float64)))
    got = res.grad_train.gather(1, other[:, None])
    assert (got.double() / want.item() - 1).abs().max().item() <= 3 * 2.0 ** -24
    assert (got == got[0]).all()
