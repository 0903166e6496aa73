"""Calls at the edges of what the entry points accept: very large pools, lengths that make no sense, buffers that overlap,
calls that follow one another without a host synchronisation."""

import pytest
import torch

from paper_2607_09052_b200 import synth

pytestmark = pytest.mark.gpu


def _binding():
    from paper_2607_09052_b200 import binding
    return binding


def to_dev(inp):
    return {k: (v.cuda() if isinstance(v, torch.Tensor) and k != "planted" else v) for k, v in inp.items()}


def test_pool_beyond_64_gib():
    """Pages whose bytes lie 64 GiB and more from the start of the pool: the same bits as from a small pool.  The first pages
    of the large pool, where an offset of 32 bits in 16-byte units would end up, hold other keys."""
    B = _binding()
    page_bytes, n_far = 16 * 128 * 2, 1 << 24                     # 4 KiB pages: page 2^24 begins at 64 GiB
    wl = synth.Workload("far", 1, 4, 1, 128, 24 * 64, 64, 16, rank=2, topk=5, window=100, summary_dtype="bf16",
                        key_model="block_offset", shuffle_pages=True, seed=19)
    if torch.cuda.mem_get_info()[0] < (n_far + 4096) * page_bytes + (2 << 30):
        pytest.skip("needs 67 GB of free device memory")
    inp = to_dev(synth.generate(wl))
    cfg = B.make_config(wl)
    n = inp["k_pages"].shape[0]
    summ = B.SummaryBuffers(cfg, "cuda")
    ws = B.alloc_workspace(cfg, "cuda")
    B.cobs_build_summaries(cfg, B.make_kv(inp), 0, wl.max_blocks, summ, ws)

    def calls(pool, table):
        kv = B.KV(pool.data_ptr(), pool.data_ptr(), table.data_ptr(), inp["seq_lens"].data_ptr(), pool.shape[0])
        sel = torch.full((1, 1, wl.topk), -7, dtype=torch.int32, device="cuda")
        cnt = torch.zeros((1, 1), dtype=torch.int32, device="cuda")
        scores = torch.zeros((1, 1, wl.max_blocks), device="cuda")
        outs = [torch.zeros((1, 4, 128), device="cuda") for _ in range(2)]
        B.cobs_exact_select(cfg, inp["q"], kv, sel, cnt, scores, ws)
        B.cobs_sparse_decode(cfg, inp["q"], kv, sel, cnt, outs[0], None, ws)
        B.cobs_decode_step(cfg, inp["q"], kv, summ, outs[1], None, None, None, ws)
        assert B.cobs_read_status(ws) == 0
        return [sel, cnt, scores] + outs

    want = calls(inp["k_pages"], inp["page_table"])
    far = torch.empty((n_far + n, 1, 16, 128), dtype=torch.bfloat16, device="cuda")
    far[:n] = inp["k_pages"].flip(0) * -1.0
    far[n_far:] = inp["k_pages"]
    got = calls(far, inp["page_table"] + n_far)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    del far
    torch.cuda.empty_cache()


def test_host_step_with_query_and_output_in_one_buffer():
    """The query at the start of the pinned buffer that receives the output: the query is read before anything is written,
    however many (sequence, KV head) units there are, as when it was copied to the device first."""
    B = _binding()
    wl = synth.Workload("alias", 96, 32, 8, 128, 16 * 64, 64, 64, rank=2, topk=4, window=100, summary_dtype="bf16",
                        key_model="block_offset", seed=5)
    inp = synth.generate(wl, "cuda")
    cfg = B.make_config(wl)
    kv = B.make_kv(inp)
    summ = B.SummaryBuffers(cfg, "cuda")
    ws = B.alloc_workspace(cfg, "cuda")
    B.cobs_build_summaries(cfg, kv, 0, wl.max_blocks, summ, ws)
    q = inp["q"].cpu().pin_memory()
    want = torch.zeros(q.shape).pin_memory()
    B.cobs_decode_step_host(cfg, q, kv, summ, want, None, None, ws)
    for at in (0, q.numel() // 2 - 64):                           # at the start of the output, and across its middle
        buf = torch.zeros(q.shape).pin_memory()
        inside = buf.view(-1)[at:at + q.numel() // 2].view(torch.bfloat16).view(q.shape)
        inside.copy_(q)
        B.cobs_decode_step_host(cfg, inside, kv, summ, buf, None, None, ws)
        assert torch.equal(buf, want)
    # the selection's arrays may lie over the query as well
    sel, cnt = torch.zeros((96, 8, 4), dtype=torch.int32).pin_memory(), torch.zeros((96, 8), dtype=torch.int32).pin_memory()
    out = torch.zeros_like(want)
    B.cobs_decode_step_host(cfg, q, kv, summ, out, sel, cnt, ws)
    q2 = q.clone().pin_memory()
    over = q2.view(-1).view(torch.int32)
    sel2, cnt2 = over[:sel.numel()].view(sel.shape), over[sel.numel():sel.numel() + cnt.numel()].view(cnt.shape)
    B.cobs_decode_step_host(cfg, q2, kv, summ, out, sel2, cnt2, ws)
    assert torch.equal(out, want) and torch.equal(sel2, sel) and torch.equal(cnt2, cnt)
    assert B.cobs_read_status(ws) == 0


def test_calls_in_a_row_without_host_synchronisation():
    """Appends, rebuilds and steps, and subspace builds with one basis after another on one workspace, enqueued back to back:
    every kernel is resident before the one in front of it has finished writing what it reads.  The same bits as with a
    synchronisation behind every call."""
    B = _binding()
    from paper_2607_09052_b200.decode_loop import DecodeLoop
    wl = synth.Workload("chain", 3, 8, 2, 128, 40 * 32, 32, 16, rank=4, topk=6, window=70, summary_dtype="bf16",
                        key_model="block_offset", shuffle_pages=True, seed=3, seq_lens=[32 * 20 + 30, 32 * 11 + 29, 32 * 31])
    cfg = B.make_config(wl)
    gen = torch.Generator().manual_seed(4)
    q, k, v = (torch.randn(shape, generator=gen).bfloat16().cuda() for shape in ((40, 3, 8, 128), (40, 3, 2, 128), (40, 3, 2, 128)))

    def loop(sync):
        inp = to_dev(synth.generate(wl))
        summ = B.SummaryBuffers(cfg, "cuda", skew=True)
        ws = B.alloc_workspace(cfg, "cuda")
        B.cobs_build_summaries(cfg, B.make_kv(inp), 0, wl.max_blocks, summ, ws)
        dl = DecodeLoop(wl, inp, summ, ws)
        out = torch.zeros((40, 3, 8, 128), device="cuda")
        torch.cuda.synchronize()
        for i in range(40):
            dl.step(q[i], k[i], v[i], out[i])
            if sync:
                torch.cuda.synchronize()
        assert B.cobs_read_status(ws) == 0
        return [out, summ.mean, summ.xi, summ.skew, inp["seq_lens"]]

    for a, b in zip(loop(False), loop(True)):
        assert torch.equal(a, b)

    wl = synth.Workload("bases", 2, 8, 2, 128, 64 * 64, 64, 16, rank=4, topk=6, window=70, summary_dtype="fp32", sub_dim=85,
                        key_model="block_offset", shuffle_pages=True, seed=6)
    cfg = B.make_config(wl)
    inp = to_dev(synth.generate(wl))
    kv = B.make_kv(inp)
    ws = B.alloc_workspace(cfg, "cuda")
    bases = [torch.linalg.qr(torch.randn((2, 128, 85), generator=gen))[0].contiguous().cuda() for _ in range(6)]

    def builds(sync):
        summs = [B.SummaryBuffers(cfg, "cuda", u) for u in bases * 2]
        torch.cuda.synchronize()
        for s in summs:
            B.cobs_build_summaries(cfg, kv, 0, wl.max_blocks, s, ws)
            if sync:
                torch.cuda.synchronize()
        assert B.cobs_read_status(ws) == 0
        return [s.xi for s in summs]

    want = builds(True)
    for _ in range(5):
        for a, b in zip(builds(False), want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("dtype,sub,skew", [("fp4", 0, False), ("bf16", 0, False), ("fp32", 0, False), ("fp4", 33, False), ("fp4", 0, True)])
def test_lengths_that_make_no_sense(dtype, sub, skew):
    """A negative length counts as an empty sequence in every call, one beyond the page table's row is reported and not
    followed; the sequences beside them get what they get without them."""
    B = _binding()
    L, D, big = 32, 64, 2 ** 31 - 1
    wl = synth.Workload("lens", 6, 8, 2, D, 70 * L, L, 16, rank=3, topk=7, window=100, summary_dtype=dtype, sub_dim=sub,
                        key_model="block_offset", shuffle_pages=True, seed=8)
    inp = to_dev(synth.generate(wl))
    cfg = B.make_config(wl)
    kv = B.make_kv(inp)
    summ = B.SummaryBuffers(cfg, "cuda", inp.get("u_q"), skew=skew)
    ws = B.alloc_workspace(cfg, "cuda")
    B.cobs_build_summaries(cfg, kv, 0, wl.max_blocks, summ, ws)
    shape = (6, 2, wl.topk)

    def calls(lens):
        inp["seq_lens"].copy_(torch.tensor(lens, dtype=torch.int32))
        sel, cnt = torch.full(shape, -7, dtype=torch.int32, device="cuda"), torch.full(shape[:2], -7, dtype=torch.int32, device="cuda")
        scores = torch.zeros((6, 2, wl.max_blocks), device="cuda")
        out, lse = torch.zeros((3, 6, 8, D), device="cuda"), torch.zeros((3, 6, 8), device="cuda")
        sel_x, cnt_x, sel_f, cnt_f = torch.full_like(sel, -7), torch.full_like(cnt, -7), torch.full_like(sel, -7), torch.full_like(cnt, -7)
        B.cobs_score_select(cfg, inp["q"], summ, inp["seq_lens"], sel, cnt, scores, ws)
        B.cobs_sparse_decode(cfg, inp["q"], kv, sel, cnt, out[0], lse[0], ws)
        B.cobs_adaptive_trim(cfg, scores, inp["seq_lens"], 0.3, 1, sel, cnt, ws)
        B.cobs_sparse_decode(cfg, inp["q"], kv, sel, cnt, out[1], lse[1], ws)
        B.cobs_decode_step(cfg, inp["q"], kv, summ, out[2], lse[2], sel_f, cnt_f, ws)
        B.cobs_exact_select(cfg, inp["q"], kv, sel_x, cnt_x, scores, ws)
        s2 = B.SummaryBuffers(cfg, "cuda", inp.get("u_q"), skew=skew)
        B.cobs_build_summaries(cfg, kv, 0, wl.max_blocks, s2, ws)
        # (outputs as their bits: an empty sequence's rows are not numbers)
        return [t.view(torch.int32) for t in (sel, cnt, sel_f, cnt_f, sel_x, cnt_x)] + \
               [t.view(torch.int32)[i] for t in (out, lse) for i in range(3)], [s2.mean, s2.xi, s2.scale]

    want, built = calls([70 * L, 0, 0, 9, 51 * L + 3, 0])
    assert B.cobs_read_status(ws) == 0
    got, built2 = calls([70 * L, -1, -70 * L, 9, 51 * L + 3, -2 ** 31])
    assert B.cobs_read_status(ws) == 0
    for a, b in zip(got + built2, want + built):
        assert torch.equal(a, b)
    assert torch.all(got[1][[1, 2, 5]] == 0) and torch.all(got[0][[1, 2, 5]] == -1)
    got, _ = calls([70 * L, big, 0, 9, 51 * L + 3, big - 15])
    assert B.cobs_read_status(ws) == 6
    B.cobs_reset_status(ws)
    for a, b in zip(got, want):
        assert torch.equal(a[[0, 2, 3, 4]], b[[0, 2, 3, 4]])

    # and no token is appended where there is no place for it
    lens = [70 * L, -1, big, 9, 51 * L + 3, -2 ** 31]
    inp["seq_lens"].copy_(torch.tensor(lens, dtype=torch.int32))
    k_new = torch.ones((6, 2, D), dtype=torch.bfloat16, device="cuda")
    pool = inp["k_pages"].clone()
    B.cobs_append_token(cfg, k_new, k_new, inp, ws)
    assert B.cobs_read_status(ws) == 6
    assert inp["seq_lens"].tolist() == [70 * L, -1, big, 10, 51 * L + 4, -2 ** 31]
    changed = (inp["k_pages"] != pool).any(-1).sum()
    assert int(changed) == 2 * 2
