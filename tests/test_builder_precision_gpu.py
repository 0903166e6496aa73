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


def degenerate_keys(kind, n, L, D, gen):
    """n blocks of L keys [n, L, D] with fewer directions than factors, or with eigenvalues that coincide."""
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    if kind == "equal":                                  # two equal eigenvalues, everything else zero: exact in bf16
        t = torch.arange(L, device="cuda") % 4
        k = torch.zeros((n, L, D), device="cuda")
        k[:, :, 5] = 2.0 * ((t == 0).float() - (t == 1).float())
        k[:, :, D - 3] = 2.0 * ((t == 2).float() - (t == 3).float())
        return k
    if kind == "constant":
        return rnd(n, 1, D).expand(n, L, D)
    if kind == "zero":
        return torch.zeros((n, L, D), device="cuda")
    if kind == "three":                                  # three distinct keys
        return rnd(n, 3, D)[:, torch.arange(L, device="cuda") % 3]
    return rnd(n, L, 2) @ rnd(n, 2, D)                   # two directions and the rounding of their products


@pytest.mark.parametrize("kind", ["equal", "constant", "zero", "three", "two"])
@pytest.mark.parametrize("L,D,sub,rank,n", [(16, 64, 0, 4, 70), (32, 128, 0, 8, 40), (64, 128, 0, 4, 40), (64, 128, 0, 4, 5), (128, 64, 0, 3, 40),
                                            (64, 128, 85, 4, 40), (128, 128, 85, 8, 9), (16, 128, 33, 16, 40)])
def test_blocks_of_fewer_directions_than_factors(L, D, sub, rank, n, kind):
    """Every block of the call degenerate, fewer of them than the careful kernel's CTAs have threads and more: the rank-r matrix
    within the errors of an eigenvalue, zeros where there is no direction.  Blocks with two equal eigenvalues are those that
    the one-warp kernel declines: it has marked them all (in the workspace's score area), and the careful kernel has done them."""
    from paper_2607_09052_b200 import binding as B
    wl = synth.Workload("degenerate", 4, 8, 2, D, n * L, L, 16, rank=rank, topk=2, window=L, summary_dtype="fp32", sub_dim=sub,
                        key_model="iid", shuffle_pages=True, seed=7)
    inp = synth.generate(wl, "cuda")
    gen = torch.Generator(device="cuda").manual_seed(3)
    keys = degenerate_keys(kind, 4 * 2 * n, L, D, gen).bfloat16().view(4, 2, n * L // 16, 16, D)
    inp["k_pages"][inp["page_table"].long().view(-1)] = keys.transpose(1, 2).reshape(-1, 2, 16, D)
    cfg = B.make_config(wl)
    summ = B.SummaryBuffers(cfg, "cuda", inp.get("u_q"))
    summ.xi.fill_(255)
    ws = B.alloc_workspace(cfg, "cuda")
    B.cobs_build_summaries(cfg, B.make_kv(inp), 0, wl.max_blocks, summ, ws)
    assert B.cobs_read_status(ws) == 0
    marks_at = (256 + 6 * 65535 * 4 + 255) // 256 * 256          # behind the status block and the counters
    marks = ws[marks_at:marks_at + 4 * 8 * n].view(torch.int32)
    if kind == "equal" and not sub:
        assert int(marks.sum()) == 8 * n
    elif kind in ("constant", "zero", "three"):
        assert int(marks.sum()) == 0
    _, xi, _ = B.summary_views(cfg, summ)
    K = keys.view(4, 2, n, L, D).double()
    K = K - K.mean(3, keepdim=True)
    if sub:
        K = torch.einsum("bhnld,hds->bhnls", K, inp["u_q"].double())
    lam, v = torch.linalg.eigh(K.transpose(-1, -2) @ K / L)
    x = xi.double()
    if kind in ("constant", "zero"):
        assert torch.all(xi == 0)
        return
    # at most the eigenvalues' own error for each direction that is left out, and for those that are not: 2^-20 of the largest
    top = (v[..., -rank:] * lam[..., None, -rank:]) @ v[..., -rank:].transpose(-1, -2)
    err = torch.linalg.matrix_norm(x.transpose(-1, -2) @ x - top, ord=2) / lam[..., -1]
    assert float(err.max()) <= 4 * 2.0 ** -20, float(err.max())
    prod = (x @ x.transpose(-1, -2)).abs() / lam[..., -1, None, None]
    assert float(torch.triu(prod, 1).max()) <= 2.0 ** -17


@pytest.mark.parametrize("kind", ["flat", "decay", "spike", "ten", "pairs"])
@pytest.mark.parametrize("L,D,sub,rank,n", [(128, 128, 0, 1, 48), (128, 128, 0, 8, 48), (128, 64, 0, 5, 48), (128, 128, 85, 4, 48),
                                            (64, 128, 0, 8, 48), (64, 64, 24, 4, 48), (64, 128, 0, 5, 160), (64, 128, 0, 8, 301),
                                            (64, 64, 0, 1, 443), (64, 128, 85, 4, 301)])
def test_leading_directions_of_hard_spectra(L, D, sub, rank, n, kind):
    """A flat spectrum, a steep one, one direction that outweighs all others, fewer directions than the solver iterates with, and
    pairs of nearly equal eigenvalues: every factor an eigenvector to the rounding of its sums (the bound of the test above, twice
    where the largest eigenvalue is a hundred times the next), none of the leading ones left out.  4 n blocks: fewer than
    are resident at a time, and more."""
    from paper_2607_09052_b200 import binding as B
    wl = synth.Workload("hard", 2, 2, 2, D, n * L, L, 16, rank=rank, topk=2, window=L, summary_dtype="fp32", sub_dim=sub,
                        key_model="iid", shuffle_pages=True, seed=11)
    inp = synth.generate(wl, "cuda")
    keys = inp["k_pages"].float()
    j = torch.arange(D, device="cuda")
    if kind == "decay":
        keys *= 0.8 ** j
    elif kind == "spike":
        keys[..., 3] *= 10.0
    elif kind == "ten":
        keys *= j < 10
    elif kind == "pairs":
        keys *= 0.7 ** (j // 2)
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
    lam = torch.linalg.eigvalsh(sigma).flip(-1)[..., :rank]
    x = xi.double()
    n2 = (x * x).sum(-1)
    resid = (x @ sigma - n2[..., None] * x).norm(dim=-1) / (lam[..., :1] * n2.sqrt())
    bound = (48 if kind == "spike" else 24) * 2.0 ** -24
    assert float(resid.max()) <= bound, float(resid.max())
    assert float(((n2 - lam).abs() / lam[..., :1]).max()) <= bound


@pytest.mark.parametrize("L,D,sub,rank,n,dtype", [(64, 128, 0, 8, 300, "fp32"), (64, 128, 0, 4, 230, "fp4"), (64, 64, 24, 4, 300, "fp32"), (64, 64, 0, 12, 40, "fp32"),
                                                  (128, 128, 0, 8, 150, "fp32"), (128, 64, 0, 4, 130, "fp4"), (128, 128, 85, 4, 120, "fp32"),
                                                  (32, 64, 0, 4, 300, "fp32"), (16, 64, 0, 4, 300, "bf16")])
def test_a_block_has_the_same_bits_in_every_call(L, D, sub, rank, n, dtype):
    """All 8 n blocks in one call, and again in calls of one block of every sequence and KV head, of a few, and of half of them: a
    block's summary is a function of its keys.  (A decode loop builds the blocks of all sequences again whenever one fills.)"""
    from paper_2607_09052_b200 import binding as B
    wl = synth.Workload("bits", 2, 4, 4, D, n * L, L, 16, rank=rank, topk=2, window=L, summary_dtype=dtype, sub_dim=sub,
                        key_model="iid", shuffle_pages=True, seed=17)
    inp = synth.generate(wl, "cuda")
    inp["k_pages"][::3, ..., 7] *= 20.0                   # some blocks with a channel that outweighs the others
    cfg = B.make_config(wl)
    ws = B.alloc_workspace(cfg, "cuda")
    whole, parts = B.SummaryBuffers(cfg, "cuda", inp.get("u_q")), B.SummaryBuffers(cfg, "cuda", inp.get("u_q"))
    kv = B.make_kv(inp)
    B.cobs_build_summaries(cfg, kv, 0, n, whole, ws)
    cuts = sorted({0, 1, 2, 5, 12, 25, n // 2, n})
    for first, last in zip(cuts, cuts[1:]):
        B.cobs_build_summaries(cfg, kv, first, last, parts, ws)
    assert B.cobs_read_status(ws) == 0
    for one, other in zip(B.summary_views(cfg, whole), B.summary_views(cfg, parts)):
        if one is not None:
            assert torch.equal(one.contiguous().view(torch.uint8), other.contiguous().view(torch.uint8))
