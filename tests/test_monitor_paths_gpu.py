"""The monitoring kernel on rows that start anywhere, and on rows with one value far above all others."""
import pytest
import torch

from paper_2512_23087_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(train, infer):
    r = binding.dvp_monitor(train, infer)
    torch.cuda.synchronize()
    a, q = torch.log_softmax(train.double(), 1), torch.log_softmax(infer.double(), 1)
    for got, want in ((r.kl_infer_train, (q.exp() * (q - a)).sum(1)), (r.kl_train_infer, (a.exp() * (a - q)).sum(1)),
                      (r.entropy_train, -(a.exp() * a).sum(1)), (r.entropy_infer, -(q.exp() * q).sum(1))):
        # float32 sums of terms of the logits' magnitude (at most 201)
        assert (got.double() - want).abs().max().item() <= 2e-5 + 201 * 2.0 ** -20


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("V,pad_t,pad_i,off", [(5, 0, 0, 0), (31, 0, 0, 1), (1003, 0, 0, 3), (4099, 1, 1, 0),
                                               (4099, 0, 2, 0), (50021, 0, 0, 0)])
def test_rows_that_start_anywhere(V, pad_t, pad_i, off, dtype):
    g = torch.Generator(device=DEV).manual_seed(V)
    T = 7
    z = torch.randn(T, V, generator=g, device=DEV) * 2
    place = lambda x, ld: torch.full((off + T * ld,), 3e4, device=DEV, dtype=dtype)[off:].view(T, ld)[:, :V].copy_(x)
    _check(place(z, V + pad_t), place(z + 0.1 * torch.randn(T, V, generator=g, device=DEV), V + pad_i))


@pytest.mark.parametrize("T,V", [(5, 24575), (5, 24576), (3, 49151), (3, 49169), (2, 98303), (2, 98305), (297, 24576),
                                 (149, 49152), (74, 98305)])
@pytest.mark.parametrize("off", [0, 5])
def test_rows_shared_by_several_blocks(T, V, off):
    """Rows of 1,536, 3,072 and 6,144 pieces take two, four and eight blocks while as many fit the chip at once."""
    g = torch.Generator(device=DEV).manual_seed(V)
    z = torch.randn(T, V, generator=g, device=DEV) * 2
    place = lambda x: torch.full((off + T * V,), 3e4, device=DEV, dtype=torch.bfloat16)[off:].view(T, V).copy_(x)
    _check(place(z), place(z + 0.1 * torch.randn(T, V, generator=g, device=DEV)))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_one_value_far_above_the_others(dtype):
    g = torch.Generator(device=DEV).manual_seed(1)
    z = torch.randn(4, 40003, generator=g, device=DEV)
    for t, k in enumerate((0, 20000, 39999, 40002)):
        z[t, k] = 200.0
    zi = z.clone()
    zi[1, 5] = 201.0
    _check(z.to(dtype), zi.to(dtype))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("pad", [0, 1])
def test_rows_of_mostly_fill(pad, dtype):
    """Filtered logits hold the lowest value of their type, which times log2(e) is no float32; a thread may meet it first."""
    V = 40000
    g = torch.Generator(device=DEV).manual_seed(2)
    z = torch.full((4, V), torch.finfo(dtype).min, dtype=torch.float64, device=DEV).to(dtype)
    zi = torch.full((4, V + pad), torch.finfo(dtype).min, dtype=torch.float64, device=DEV).to(dtype)[:, :V]
    for t, (lo, hi) in enumerate([(V // 2, V), (V - 5, V), (0, 9), (V // 3, V // 3 + 1000)]):
        x = 2 * torch.randn(hi - lo, generator=g, device=DEV)
        z[t, lo:hi] = x.to(dtype)
        zi[t, lo:hi] = (x + 0.1 * torch.randn(hi - lo, generator=g, device=DEV)).to(dtype)
    _check(z, zi)


@pytest.mark.parametrize("V,dtype,steps", [(15000, torch.float16, 8), (16000, torch.bfloat16, 8), (6000, torch.float32, 6)])
def test_sums_keep_small_terms_in_short_rows(V, dtype, steps):
    """One token at 0 and all others at -17, where e^-17 = 0.69 * 2^-24 is lost when it is added to 1 by itself.  Each
    step's terms are added up first: one rounding of the sum a step, one a pair of logits in the step of the maximum itself
    (16 or 8), six where the 64 threads' sums meet, and a few in the logarithms."""
    z = torch.full((1300, V), -17.0, dtype=dtype, device=DEV)   # fewer rows take more threads each
    for t, k in enumerate((0, 33, 70)):
        z[t::3, k] = 0.0
    r = binding.dvp_monitor(z, z)
    torch.cuda.synchronize()
    a = torch.log_softmax(z.double(), 1)
    err = (r.entropy_train.double() + (a.exp() * a).sum(1)).abs().max().item()
    assert err <= (steps + 32 // z.element_size() + 6 + 4) * 2.0 ** -24
