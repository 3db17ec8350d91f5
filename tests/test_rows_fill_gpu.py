"""Rows in which most logits hold the lowest value of their type (or -inf), as top-k and grammar filters leave them: such a
value times log2(e) is no float32, and a block that shares a row may see nothing else."""
import pytest
import torch

from paper_2512_23087_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _filled(V, dtype, fill, seed):
    """Six rows with logits in one window each (first part, middle, end, a few tokens), the rest `fill`; ids inside the window,
    outside of it, or none."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    z = torch.full((6, V), fill, dtype=torch.float64, device=DEV).to(dtype)
    windows = [(0, V // 9), (V // 2, V // 2 + V // 7), (V - V // 9, V), (V // 3, V // 3 + 5), (V - 3, V), (V // 2, V // 2 + 1)]
    for t, (lo, hi) in enumerate(windows):
        z[t, lo:hi] = (3 * torch.randn(hi - lo, generator=g, device=DEV)).to(dtype)
    return z, windows


@pytest.mark.parametrize("who", ["inside", "masked", "none"])
@pytest.mark.parametrize("hint", [0, 64, 256, 256 | (2 << 24), 256 | (4 << 24), 256 | (8 << 24)])
@pytest.mark.parametrize("dtype,fill", [(torch.bfloat16, "lowest"), (torch.bfloat16, "-inf"), (torch.float32, "lowest"),
                                        (torch.float32, "-inf"), (torch.float16, "lowest"), (torch.float16, "-inf")])
def test_rows_of_mostly_fill(dtype, fill, hint, who):
    V = 70001
    z, windows = _filled(V, dtype, torch.finfo(dtype).min if fill == "lowest" else -float("inf"), seed=hint % 1000)
    ids = torch.tensor([{"inside": lo, "masked": hi % V if hi < V else 0, "none": -1}[who] for lo, hi in windows], device=DEV)
    rho = 1e-3
    r = binding.dvp_forward(z, ids, rho, infer_logits=z, launch_hint=hint)
    torch.cuda.synchronize()
    d = z.double()
    m = d.max(1).values
    lse = torch.logsumexp(d, 1)
    keep = d >= (m + torch.log(torch.tensor(rho, dtype=torch.float64)))[:, None]
    lse_safe = torch.logsumexp(torch.where(keep, d, torch.full_like(d, -float("inf"))), 1)
    # float32 sums of at most 70001 terms and one rounding of the value itself
    near = lambda got, want: (got.double() - want).abs().le(4e-6 + 2.0 ** -23 * want.abs()).logical_or(got.double() == want)
    for side in (r.train, r.infer):
        assert torch.equal(side.max.double(), m) and torch.equal(side.count.long(), keep.sum(1))
        assert near(side.lse, lse).all() and near(side.lse_safe, lse_safe).all()
        assert near(side.log_cov, lse_safe - lse).all()
        if who == "none":
            assert side.logp.isnan().all() and side.logp_mp.isnan().all()
        else:
            a = d.gather(1, ids[:, None])[:, 0]
            assert near(side.logp, (a - lse).clamp(min=-3.4028235e38) if fill == "lowest" else a - lse).all()
            inside = keep.gather(1, ids[:, None])[:, 0]
            assert near(side.logp_mp[inside], (a - lse_safe)[inside]).all() and (side.logp_mp[~inside] == -float("inf")).all()


@pytest.mark.parametrize("hint", [0x11 << 16, 256 | (3 << 16), 256 | (4 << 16)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_kernels_by_hint_on_rows_of_mostly_fill(dtype, hint):
    V = 70016
    z, windows = _filled(V, dtype, torch.finfo(dtype).min, seed=1)
    ids = torch.tensor([lo for lo, _ in windows], device=DEV)
    r = binding.dvp_forward(z, ids, 1e-3, infer_logits=z, launch_hint=hint)
    torch.cuda.synchronize()
    lse = torch.logsumexp(z.double(), 1)
    assert ((r.train.lse.double() - lse).abs() <= 4e-6 + 2.0 ** -23 * lse.abs()).all()   # as above
    assert torch.equal(r.train.lse, r.infer.lse) and torch.isfinite(r.train.log_cov).all()
