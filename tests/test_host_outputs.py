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
