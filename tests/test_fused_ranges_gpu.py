"""d_hidden of few tokens: its few output tiles are computed as several ranges of the vocabulary, whose partial results
are summed in order; and tokens that share a sampled id, whose rows of d_w are added in token order."""
import pytest
import torch

from paper_2512_23087_b200 import binding, inputs

import test_fused_gpu as fused

pytestmark = pytest.mark.gpu


# one tile with as many ranges as fit; H that ends inside a vector and inside a tile; V below H (no room for ranges);
# two rows of tiles, the last of one token
@pytest.mark.parametrize("T,H,V", [(24, 128, 9001), (33, 520, 8200), (16, 1032, 1000), (257, 264, 6000)])
def test_ranges_of_the_vocabulary(T, H, V):
    batch, res, want, rerun = fused._run_fused(T, H, V, 1e-3, seed=T)
    fused._check_fused(batch, 1e-3, res, want, V, rerun=rerun)
    again = rerun(batch.upstream)
    assert torch.equal(again.d_hidden, res.d_hidden) and torch.equal(again.d_w, res.d_w)


@pytest.mark.parametrize("n_ids", [1, 5])
def test_many_tokens_of_one_id(n_ids):
    w = inputs.WORKLOADS["c4_fused_lmhead"]
    b = inputs.make_fused(w, seed=9, device=fused.DEV, T=300, H=256, V=2000)
    b.ids.copy_(torch.arange(300, device=fused.DEV) % n_ids * 7)
    r = [binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, 0.0, b.upstream, infer_logits=b.infer)
         for _ in range(2)]
    torch.cuda.synchronize()
    z = b.hidden.double() @ b.w_vocab.double().t()
    g = -torch.softmax(z, 1) * b.upstream.double()[:, None]
    g.scatter_add_(1, b.ids[:, None], b.upstream.double()[:, None])
    want = g.t() @ b.hidden.double()
    # float16 gradient panel: 2^-11 a term at most, tokens of one row add up
    assert ((r[0].d_w.double() - want).norm(dim=1) <= 1e-3 * want.norm(dim=1) + 1e-6 * want.norm(dim=1).max()).all()
    assert torch.equal(r[0].d_w, r[1].d_w)


# products with a short k store exchanged pieces of four neighbouring rows (up to 8 slices of 64): ends inside the four
# rows, the warp's 32 and the block's 128, columns that end inside a group of 32, and either side of the line
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("k", [8, 512, 520])
@pytest.mark.parametrize("m,n", [(1, 8), (3, 40), (35, 32), (130, 264), (513, 304)])
def test_stores_of_short_products(m, n, k, accumulate):
    g = torch.Generator(device=fused.DEV).manual_seed(m + n + k)
    a = torch.randn(m, k, generator=g, device=fused.DEV).to(torch.bfloat16)
    b = torch.randn(n, k, generator=g, device=fused.DEV).to(torch.bfloat16)
    buf = torch.full((m + 4, n + 8), 3.0, device=fused.DEV)
    out, status = binding.dvp_gemm_tn(a, b, alpha=0.5, out=buf[:m, :n], accumulate=accumulate)
    torch.cuda.synchronize()
    assert status.item() == 0
    ref = 0.5 * (a.double() @ b.double().t()) + (3.0 if accumulate else 0.0)
    # one rounding of the running sum per 16-wide step of k, one of the scaled value, one of the addition
    bound = 2.0 ** -24 * (k / 16 + 2) * (a.double().abs() @ b.double().abs().t() + 3.0)
    assert ((out.double() - ref).abs() <= bound).all()
    assert (buf[m:] == 3.0).all() and (buf[:, n:] == 3.0).all()


@pytest.mark.parametrize("V", [32768, 32775])
def test_inference_rows_of_mostly_fill(V):
    """Filtered inference logits hold the lowest bfloat16, which times log2(e) is no float32; a thread may meet it first."""
    w = inputs.WORKLOADS["c4_fused_lmhead"]
    b = inputs.make_fused(w, seed=3, device=fused.DEV, T=24, H=128, V=V)
    b.infer[:, :V // 2] = torch.finfo(torch.bfloat16).min
    b.infer[1, :V - 3] = torch.finfo(torch.bfloat16).min
    b.ids.copy_(torch.arange(24, device=fused.DEV) + V - 26)
    r = binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, 1e-4, b.upstream, infer_logits=b.infer)
    torch.cuda.synchronize()
    lse = torch.logsumexp(b.infer.double(), 1)
    logp = b.infer.double().gather(1, b.ids[:, None])[:, 0] - lse
    # float32 sums of at most 32775 terms and one rounding of the value itself
    assert (r.infer.lse.double() - lse).abs().max().item() <= 4e-6
    ok = logp > -1e30
    assert ok.sum() >= 23 and (r.infer.logp.double() - logp)[ok].abs().max().item() <= 6e-6
    assert torch.isfinite(r.d_hidden).all() and torch.isfinite(r.d_w).all()
