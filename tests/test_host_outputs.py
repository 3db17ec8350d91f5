"""The helper that lays a call's outputs over one allocation: types, lengths, alignment, no overlap."""
import pytest
import torch

from paper_2512_23087_b200 import binding, build


@pytest.mark.parametrize("inference_mode", [False, True])
@pytest.mark.parametrize("T", [0, 1, 3, 4, 5, 257])
def test_outputs_lie_side_by_side(T, inference_mode):
    build.build_host()
    binding.load_library()
    with torch.inference_mode(inference_mode):
        like = torch.empty(2, 3, dtype=torch.bfloat16)
        tensors, address, stride = binding._host.outputs(like, T, 3, 2)
        assert [t.dtype for t in tensors] == [torch.float32] * 3 + [torch.int32] * 2 + [torch.uint8]
        assert stride % 16 == 0 and stride >= 4 * T
        for i, t in enumerate(tensors):
            assert t.shape == (T,) and t.is_contiguous() and t.device == like.device and not t.requires_grad
            if T:
                assert t.data_ptr() == address + i * stride
            t.fill_(i + 1)
        for i, t in enumerate(tensors):
            assert (t == i + 1).all()


def test_outputs_refuses_other_arguments():
    binding.load_library()
    with pytest.raises(TypeError):
        binding._host.outputs(1, 2, 3, 4)


@pytest.mark.parametrize("T", [-1, -8, 2 ** 60])
def test_outputs_refuses_lengths_no_vector_has(T):
    binding.load_library()
    with pytest.raises(RuntimeError, match="elements"):
        binding._host.outputs(torch.empty(1), T, 3, 2)


@pytest.mark.gpu
def test_out_of_memory_keeps_its_type():
    binding.load_library()
    with pytest.raises(torch.OutOfMemoryError):   # 2^44 bytes: the allocator refuses
        binding._host.outputs(torch.empty(1, device="cuda:0"), 2 ** 40, 3, 0)
    assert binding._host.outputs(torch.empty(1, device="cuda:0"), 5, 3, 0)[2] == 32


def test_forward_refuses_what_it_is_not_made_for():
    """Before anything is launched, with the types of error that Python code gives."""
    x, ids = torch.zeros(3, 5), torch.zeros(3, dtype=torch.int64)
    for error, call in ((ValueError, lambda: binding.dvp_forward(x, ids, 0.1)),
                        (ValueError, lambda: binding.dvp_forward(x[0], ids, 0.1)),
                        (TypeError, lambda: binding.dvp_forward(None, ids, 0.1)),
                        (TypeError, lambda: binding.dvp_forward(x, ids, 0.1, launch_hint=2.0)),
                        (ValueError, lambda: binding.dvp_forward(x, ids, "a"))):
        with pytest.raises(error):
            call()
    with pytest.raises(TypeError):
        binding._host.forward(1, 2)


@pytest.mark.gpu
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("infer", [False, True])
def test_forward_gives_what_the_packed_call_gives(infer, weighted):
    """A call that also wants the masks goes through Python; all else must be the same, refusals too."""
    if weighted and not infer:
        return
    g = torch.Generator(device="cuda:0").manual_seed(1)
    z = torch.randn(7, 1003, generator=g, device="cuda:0") * 4
    zi = z + 0.1 * torch.randn(7, 1003, generator=g, device="cuda:0") if infer else None
    ids = torch.randint(0, 1003, (7,), generator=g, device="cuda:0", dtype=torch.int32)
    up = torch.randn(7, generator=g, device="cuda:0")
    kw = dict(infer_logits=zi, upstream=up, grad_dtype=torch.bfloat16, mask_value=-50.0)
    if weighted:
        kw.update(weight_kind=binding.DVP_WEIGHT_TRUNCATE, weight_hi=1.01)
    stream = torch.cuda.Stream()
    a, b = binding.dvp_forward(z, ids, 1e-2, **kw), binding.dvp_forward(z, ids, 1e-2, want_mask=True, **kw)
    torch.cuda.synchronize()
    c = binding.dvp_forward(z, ids, 1e-2, stream=stream, grad_train=torch.empty_like(a.grad_train), **{**kw, "grad_dtype": None})
    torch.cuda.synchronize()
    assert set(vars(a)) == set(vars(b)) and (a.infer is None) == (not infer) and a.train.mask is None
    for r in (a, c):
        for n in vars(b):
            x, y = getattr(r, n), getattr(b, n)
            if n in ("train", "infer") and y is not None:
                assert list(vars(x)) == list(vars(y))
                assert all(torch.equal(getattr(x, m), getattr(y, m)) for m in vars(y) if m != "mask"), n
            elif y is None:
                assert x is None
            else:
                assert x.dtype == y.dtype and x.shape == y.shape and torch.equal(x, y), n
    for error, bad in ((ValueError, dict(infer_logits=z[:, :5])), (TypeError, dict(upstream=up.double())),
                       (binding.DvpError, dict(weight_kind=binding.DVP_WEIGHT_RATIO, infer_logits=None)),
                       (KeyError, dict(grad_train=torch.empty(7, 1003, device="cuda:0", dtype=torch.float64)))):
        with pytest.raises(error):
            binding.dvp_forward(z, ids, 1e-2, **{**kw, **bad})
    with pytest.raises(TypeError):
        binding.dvp_forward(z, ids.float(), 1e-2)
    with pytest.raises(KeyError):
        binding.dvp_forward(z.double(), ids, 1e-2)


def test_helper_is_rebuilt_for_another_torch(monkeypatch, tmp_path):
    """A helper built against another torch (or interpreter) lays tensors over the wrong layout: it is neither kept by the
    build nor used by the binding."""
    monkeypatch.setattr(build, "HOST", str(tmp_path / "_host.so"))
    monkeypatch.setattr(build.subprocess, "run", _fake_compiler(tmp_path))
    build.build_host()
    first = (tmp_path / "count").read_text()
    build.build_host()
    assert (tmp_path / "count").read_text() == first == "1"
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    build.build_host()
    assert (tmp_path / "count").read_text() == "2"
    build.build_host(force=True)
    assert (tmp_path / "count").read_text() == "3"
    monkeypatch.setattr(binding, "_lib", None)
    with pytest.raises(RuntimeError, match="built for another"):
        binding.load_library()


def _fake_compiler(tmp_path):
    """Stands in for g++: writes the text that the helper would carry, and counts."""
    def run(cmd, **kw):
        n = tmp_path / "count"
        n.write_text(str(int(n.read_text()) + 1 if n.exists() else 1))
        define = next(c for c in cmd if c.startswith("-DDVP_HOST_TARGET="))
        with open(cmd[cmd.index("-o") + 1], "wb") as f:
            f.write(b"[built for " + define.split("=", 1)[1].strip('"').encode() + b"]")
        return build.subprocess.CompletedProcess(cmd, 0, "", "")
    return run
