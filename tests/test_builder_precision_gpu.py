"""The builder's fp32 factors against the eigenvectors of the same keys' covariance in 64 bits, where the keys' mean or their
scale makes the products lose bits."""

import pytest
import torch

from paper_2607_09052_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mean", ["none", "all", "some"])
@pytest.mark.parametrize("L", [16, 32, 64, 128])
@pytest.mark.parametrize("D,sub,rank", [(128, 85, 4), (128, 33, 8), (64, 24, 4), (128, 0, 4)])
def test_factors_do_not_lose_the_bits_of_the_mean(D, sub, rank, L, mean):
    """A mean of 30 spreads per element, in all dimensions or in a few, drops out of the centred keys: the residual of every
    factor, |Sigma x - |x|^2 x| over lambda_0 |x|, is that of rounding alone.  The centred Gram matrix, its tridiagonal form and
    the factors are each formed in fp32: 24 units of 2^-24 allow for their sums and products (a projection that keeps the
    mean in its sums shows 2e-6 and more here)."""
    from paper_2607_09052_b200 import binding as B
    wl = synth.Workload("mean", 2, 4, 2, D, 24 * L, L, 16, rank=rank, topk=2, window=L, summary_dtype="fp32", sub_dim=sub,
                        key_model="iid", shuffle_pages=True, seed=7)
    inp = synth.generate(wl, "cuda")
    keys = inp["k_pages"].float()
    if mean == "all":
        keys += 30.0
    elif mean == "some":
        keys[..., 3:12:4] += torch.tensor([30.0, -45.0, 20.0], device="cuda")
    inp["k_pages"] = keys.to(torch.bfloat16)
    cfg = B.make_config(wl)
    summ = B.SummaryBuffers(cfg, "cuda", inp.get("u_q"))
    ws = B.alloc_workspace(cfg, "cuda")
    B.cobs_build_summaries(cfg, B.make_kv(inp), 0, wl.max_blocks, summ, ws)
    assert B.cobs_read_status(ws) == 0
    _, xi, _ = B.summary_views(cfg, summ)
    K = inp["k_pages"][inp["page_table"].long()].permute(0, 2, 1, 3, 4).reshape(2, 2, -1, L, D).double()
    K = K - K.mean(3, keepdim=True)
    if sub:
        K = torch.einsum("bhnld,hds->bhnls", K, inp["u_q"].double())
    sigma = K.transpose(-1, -2) @ K / L
    lam0 = torch.linalg.eigvalsh(sigma)[..., -1]
    x = xi.double()
    n2 = (x * x).sum(-1)
    resid = (x @ sigma - n2[..., None] * x).norm(dim=-1) / (lam0[..., None] * n2.sqrt())
    assert float(resid.max()) <= 24 * 2.0 ** -24, float(resid.max())
