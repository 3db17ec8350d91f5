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
