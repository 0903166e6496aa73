"""Selection: ties in every layout of the top-k search, and units beyond the step kernel's capacity."""

import math

import pytest
import torch

from oracle import cobs_oracle as O
from paper_2607_09052_b200 import synth
from parity import SCORE_TOL, check_selection

pytestmark = pytest.mark.gpu


def _binding():
    from paper_2607_09052_b200 import binding
    return binding


def one_page_inputs(wl, n_pages=1, seed=0):
    """Inputs whose page tables name the same few pages over and over: a context of any length in a small pool."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    d, hkv = wl.head_dim, wl.n_kv_heads
    pages = torch.randn((2, n_pages, hkv, wl.page_size, d), generator=gen, device="cuda").bfloat16()
    return {"q": torch.randn((wl.batch, wl.n_q_heads, d), generator=gen, device="cuda").bfloat16(), "k_pages": pages[0], "v_pages": pages[1],
            "page_table": torch.randint(0, n_pages, (wl.batch, wl.max_pages_per_seq), generator=gen, device="cuda", dtype=torch.int32),
            "seq_lens": torch.tensor(wl.lens(), dtype=torch.int32, device="cuda")}


# Candidates per unit at the edges of the layouts: one warp with four and eight keys per lane (up to as many keys as the CTA has
# threads), two and eight keys per thread, any number; with eight warps per CTA (few units) and with four (more units than SMs,
# where more than 576 keys lie over the copy rings).
EDGES = [1, 48, 49, 127, 128, 129, 255, 256, 257, 511, 512, 513, 575, 576, 577, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 6001]


@pytest.mark.parametrize("copies", [1, 8])
@pytest.mark.parametrize("topk", [48, 128])
def test_exact_ties_at_the_edges_of_every_layout(topk, copies):
    """Blocks of two kinds, identical within a kind: every score is one of two values, and the selection is all of the better
    kind plus the lowest-index ones of the other, or the lowest-index ones of the better kind."""
    B = _binding()
    L, D, G, window = 16, 64, 4, 40
    n_cands = EDGES * copies
    lens = [n * L + window for n in n_cands]
    nb = (max(lens) + L - 1) // L
    wl = synth.Workload("ties", len(lens), G, 1, D, nb * L, L, 16, rank=2, topk=topk, window=window, summary_dtype="bf16", seq_lens=lens)
    inp = one_page_inputs(wl)
    gen = torch.Generator(device="cuda").manual_seed(5)
    v = torch.randn(D, generator=gen, device="cuda")
    inp["q"] = (v + 0.3 * torch.randn((len(lens), G, D), generator=gen, device="cuda")).bfloat16()
    cfg = B.make_config(wl)
    summ = B.SummaryBuffers(cfg, "cuda")
    ws = B.alloc_workspace(cfg, "cuda")
    mean_v, xi_v, _ = B.summary_views(cfg, summ)
    hot = torch.arange(nb, device="cuda") % 16 == 3
    mean_v[:, 0] = torch.where(hot[:, None], 0.5 * v, -0.5 * v).bfloat16()
    xi_v[:] = (0.2 * torch.randn((2, D), generator=gen, device="cuda")).bfloat16()
    sel, cnt = torch.full((len(lens), 1, topk), -7, dtype=torch.int32, device="cuda"), torch.full((len(lens), 1), -7, dtype=torch.int32, device="cuda")
    sel_f, cnt_f = sel.clone(), cnt.clone()
    out = torch.zeros((len(lens), G, D), device="cuda")
    B.cobs_score_select(cfg, inp["q"], summ, inp["seq_lens"], sel, cnt, None, ws)
    B.cobs_decode_step(cfg, inp["q"], B.make_kv(inp), summ, out, None, sel_f, cnt_f, ws)
    assert B.cobs_read_status(ws) == 0
    assert torch.equal(sel, sel_f) and torch.equal(cnt, cnt_f)
    hot_c = [b for b in range(nb) if b % 16 == 3]
    cold_c = [b for b in range(nb) if b % 16 != 3]
    for i, n in enumerate(n_cands):
        k = min(topk, n)
        h = [b for b in hot_c if b < n][:k]
        want = sorted(h + [b for b in cold_c if b < n][:k - len(h)])
        assert int(cnt[i, 0]) == k and sel[i, 0].tolist() == want + [-1] * (topk - k), n


def check_long_units(dtype, sub, n, rank=2, D=64, hkv=1, skew=False):
    """Units of n blocks: scores against the estimates in 64 bits, selection by the tie band, the step's selection equal to
    cobs_score_select's and its output to cobs_sparse_decode's."""
    B = _binding()
    L, G, topk = 16, 2, 33
    wl = synth.Workload("long", 1, G * hkv, hkv, D, n * L, L, 16, rank=rank, topk=topk, window=100, summary_dtype=dtype, sub_dim=sub, seq_lens=[n * L - 3])
    inp = one_page_inputs(wl, n_pages=4)
    gen = torch.Generator(device="cuda").manual_seed(9)
    u_q = torch.linalg.qr(torch.randn((hkv, D, sub), generator=gen, device="cuda"))[0].contiguous() if sub else None
    cfg = B.make_config(wl)
    kv = B.make_kv(inp)
    summ = B.SummaryBuffers(cfg, "cuda", u_q, skew=skew)
    ws = B.alloc_workspace(cfg, "cuda")
    mean_v, xi_v, scale_v = B.summary_views(cfg, summ)
    mean_v.copy_(6.4 / math.sqrt(D) * torch.randn(mean_v.shape, generator=gen, device="cuda"))
    ds = sub or D
    xi = 3.4 / math.sqrt(rank * D) * torch.randn((1, hkv, n, rank, ds), generator=gen, device="cuda")
    if dtype == "fp4":
        pad = B.cobs_padded_sub_dim(cfg)
        B.cobs_quantise_xi(cfg, xi.view(-1, ds), summ.xi, summ.scale)
        grid = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6], dtype=torch.float64, device="cuda")
        xi = grid[B.unpack_fp4_rows(xi_v.reshape(-1, pad // 2), pad).long()][:, :ds].view(1, hkv, n, rank, ds) * scale_v.double()[..., None]
    else:
        xi_v.copy_(xi)
        xi = xi_v.double()
    if skew:
        summ.skew.copy_(0.3 * torch.randn(summ.skew.shape, generator=gen, device="cuda"))
    sel, cnt = torch.full((1, hkv, topk), -7, dtype=torch.int32, device="cuda"), torch.zeros((1, hkv), dtype=torch.int32, device="cuda")
    sel_f, cnt_f = sel.clone(), cnt.clone()
    scores = torch.zeros((1, hkv, n), device="cuda")
    out_a, out_f = torch.zeros((2, 1, G * hkv, D), device="cuda")
    B.cobs_score_select(cfg, inp["q"], summ, inp["seq_lens"], sel, cnt, scores, ws)
    B.cobs_sparse_decode(cfg, inp["q"], kv, sel, cnt, out_a, None, ws)
    B.cobs_decode_step(cfg, inp["q"], kv, summ, out_f, None, sel_f, cnt_f, ws)
    assert B.cobs_read_status(ws) == 0
    n_sum = n - 1
    n_cand = O.window_start(n * L - 3, 100, L) // L
    for h in range(hkv):
        q = inp["q"].double()[0, h * G:(h + 1) * G] / math.sqrt(D)
        p = torch.einsum("nrs,gs->gnr", xi[0, h].double(), q @ u_q[h].double() if sub else q)
        e = math.log(L) + q @ mean_v.double()[0, h].T + 0.5 * (p ** 2).sum(-1)
        if skew:
            e = e + (summ.skew[0, h].double() * p ** 3).sum(-1) / 6
        want = torch.softmax(e[:, :n_sum], -1).sum(0)
        assert float(((scores[0, h, :n_sum].double() - want).abs() / want).max()) <= SCORE_TOL
        ok, msg, _ = check_selection(sel[0, h].tolist(), want.cpu().numpy(), n_cand, topk)
        assert ok, msg
    assert torch.equal(sel, sel_f) and torch.equal(cnt, cnt_f)
    assert float((out_f - out_a).abs().max() / out_a.abs().max()) <= 1e-5


@pytest.mark.parametrize("n", [24575, 24576, 24577, 30001])
@pytest.mark.parametrize("dtype,sub", [("fp4", 0), ("bf16", 0), ("fp32", 0), ("fp4", 33), ("bf16", 33), ("fp32", 33)])
def test_units_at_and_beyond_the_step_kernels_capacity(dtype, sub, n):
    """24 576 blocks per unit are what the step kernel holds the scores of; above, scoring and selection run in the generic
    kernels."""
    check_long_units(dtype, sub, n)


# one or two units with many elements to score row by row go to the generic kernels: both sides of each line
@pytest.mark.parametrize("dtype,sub,rank,D,hkv,skew,n", [
    ("fp32", 0, 8, 64, 1, False, 14563), ("fp32", 0, 8, 64, 1, False, 14564), ("fp32", 85, 16, 128, 1, False, 5637),
    ("fp32", 85, 16, 128, 1, False, 5638), ("fp32", 0, 16, 128, 2, False, 11564), ("fp32", 0, 16, 128, 2, False, 11566),
    ("fp32", 0, 8, 128, 1, True, 7300), ("bf16", 85, 16, 128, 1, False, 16900), ("bf16", 85, 16, 128, 1, False, 16920),
    ("bf16", 0, 16, 128, 1, True, 11570), ("bf16", 0, 16, 128, 1, True, 11560), ("bf16", 0, 16, 128, 1, False, 11570)])
def test_units_with_many_rows_to_score(dtype, sub, rank, D, hkv, skew, n):
    check_long_units(dtype, sub, n, rank, D, hkv, skew)


@pytest.mark.parametrize("n,hkv,L,D,G", [(3, 1, 16, 64, 2), (5000, 1, 16, 64, 2), (5000, 3, 16, 64, 2), (24576, 2, 16, 64, 2), (24577, 2, 16, 64, 2),
                                         (1023, 1, 64, 128, 4), (1024, 1, 64, 128, 4), (1025, 3, 64, 128, 4), (1024, 4, 64, 128, 4),
                                         (2048, 2, 64, 128, 8), (2048, 3, 64, 128, 8), (1023, 1, 128, 64, 1), (1024, 3, 128, 64, 1),
                                         (292, 152, 16, 128, 2), (300, 149, 16, 128, 1), (293, 185, 16, 128, 1), (293, 186, 16, 128, 1)])
def test_exact_selection_of_long_units(n, hkv, L, D, G):
    """The exact block masses of long contexts, on both sides of the lines between the kernels that take them: against direct sums
    in 64 bits."""
    B = _binding()
    topk, batch = 40, 1
    wl = synth.Workload("longx", batch, G * hkv, hkv, D, n * L, L, 16, rank=1, topk=topk, window=100, summary_dtype="bf16", seq_lens=[n * L - 5])
    inp = one_page_inputs(wl, n_pages=2 * n * (L // 16))
    cfg = B.make_config(wl)
    ws = B.alloc_workspace(cfg, "cuda")
    sel, cnt = torch.full((batch, hkv, topk), -7, dtype=torch.int32, device="cuda"), torch.zeros((batch, hkv), dtype=torch.int32, device="cuda")
    scores = torch.zeros((batch, hkv, n), device="cuda")
    B.cobs_exact_select(cfg, inp["q"], B.make_kv(inp), sel, cnt, scores, ws)
    assert B.cobs_read_status(ws) == 0
    n_sum = (n * L - 5) // L
    keys = inp["k_pages"][inp["page_table"][0].long()].transpose(0, 1).reshape(hkv, n, L, D).double()
    q = inp["q"][0].double().view(hkv, G, D) / math.sqrt(D)
    e = torch.logsumexp(torch.einsum("hnld,hgd->hgnl", keys, q), -1)[:, :, :n_sum]
    want = torch.softmax(e, -1).sum(1)
    assert float(((scores[0, :, :n_sum].double() - want).abs() / want).max()) <= SCORE_TOL
    n_cand = O.window_start(n * L - 5, 100, L) // L
    for h in range(hkv):
        ok, msg, _ = check_selection(sel[0, h].tolist(), want[h].cpu().numpy(), n_cand, topk)
        assert ok, (h, msg)
        assert int(cnt[0, h]) == min(topk, n_cand)
