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
