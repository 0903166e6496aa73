"""Block scores against the same estimates in 64 bits."""

import math

import pytest
import torch

from paper_2607_09052_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,rank,sub", [("bf16", 4, 0), ("fp32", 8, 0), ("fp32", 4, 85), ("exact", 1, 0)])
def test_scores_carry_the_rounding_of_the_estimates_and_no_more(dtype, rank, sub):
    """Estimates e lie between 2 and 8 here (ln L = 4.2), where half a unit in the last place is 2.4e-7 and its root mean square
    1.4e-7; a score is a mean over four heads of exponentials, each with the rounding of its own e and that of the sum and
    the exponential (a few times 2^-24): 1.7e-7 over all blocks.  One more rounded term per head of the size of e, such as
    a log-sum-exp, is common to all blocks of a unit and shows as 2.3e-7 or more."""
    from paper_2607_09052_b200 import binding as B
    total, n = 0.0, 0
    for seed in range(6):
        wl = synth.Workload("prec", 2, 16, 4, 128, 256 * 64, 64, 16, rank=rank, topk=8, window=200, sub_dim=sub,
                            summary_dtype="bf16" if dtype == "exact" else dtype, key_model="iid", shuffle_pages=True, seed=seed)
        inp = synth.generate(wl, "cuda")
        cfg = B.make_config(wl)
        kv = B.make_kv(inp)
        summ = B.SummaryBuffers(cfg, "cuda", inp.get("u_q"))
        ws = B.alloc_workspace(cfg, "cuda")
        sel, cnt = torch.zeros((2, 4, 8), dtype=torch.int32, device="cuda"), torch.zeros((2, 4), dtype=torch.int32, device="cuda")
        scores = torch.zeros((2, 4, wl.max_blocks), device="cuda")
        q = inp["q"].double().view(2, 4, 4, 128) / math.sqrt(128)
        if dtype == "exact":
            B.cobs_exact_select(cfg, inp["q"], kv, sel, cnt, scores, ws)
            K = inp["k_pages"][inp["page_table"].long()].permute(0, 2, 1, 3, 4).reshape(2, 4, -1, 64, 128).double()
            e = torch.logsumexp(torch.einsum("bhnld,bhgd->bhgnl", K, q), -1)
        else:
            B.cobs_build_summaries(cfg, kv, 0, wl.max_blocks, summ, ws)
            B.cobs_score_select(cfg, inp["q"], summ, inp["seq_lens"], sel, cnt, scores, ws)
            mean, xi, _ = B.summary_views(cfg, summ)
            qt = torch.einsum("bhgd,hds->bhgs", q, inp["u_q"].double()) if sub else q
            e = math.log(64) + torch.einsum("bhnd,bhgd->bhgn", mean.double(), q) + \
                0.5 * (torch.einsum("bhnrs,bhgs->bhgnr", xi.double(), qt) ** 2).sum(-1)
        assert B.cobs_read_status(ws) == 0
        want = torch.softmax(e, -1).sum(2)
        total += float((((scores.double() - want) / want) ** 2).sum())
        n += want.numel()
    assert math.sqrt(total / n) <= 1.7e-7, math.sqrt(total / n)
