"""The step with more units than SMs: parity where the launch's plan changes (one wave and a rest in clusters, two CTAs of four
warps per SM, three waves of eight warps)."""

import pytest
import torch

from paper_2607_09052_b200 import synth
from test_parity_gpu import check_fused_equals_two_calls_on_every_unit, run_stage_s

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,hkv,blocks,rank,dtype,sub", [
    (149, 1, 140, 16, "fp32", 0), (23, 8, 140, 16, "fp32", 0), (185, 1, 140, 16, "fp32", 0), (31, 6, 140, 16, "fp32", 0),      # 149, 184, 185, 186 units
    (19, 8, 140, 16, "fp32", 64), (19, 8, 280, 16, "bf16", 0), (19, 8, 900, 16, "fp4", 0), (19, 8, 40, 16, "fp32", 0),
    (37, 8, 130, 4, "fp4", 0), (297, 1, 112, 4, "bf16", 0), (297, 1, 113, 4, "bf16", 0), (111, 4, 130, 4, "fp4", 33), (89, 5, 120, 4, "fp4", 0),      # 296 to 445
    (128, 4, 8, 4, "fp32", 0), (511, 1, 8, 4, "fp32", 33), (74, 4, 4, 4, "fp32", 0), (99, 3, 4, 4, "fp32", 0), (64, 16, 16, 8, "fp32", 0), (64, 17, 17, 8, "fp32", 0)])
def test_more_units_than_sms(batch, hkv, blocks, rank, dtype, sub):
    from paper_2607_09052_b200 import binding as B
    L = 16
    lens = [blocks * L - (5 * b) % (3 * L) for b in range(batch)]
    wl = synth.Workload("plan", batch, 2 * hkv, hkv, 128, blocks * L, L, 16, rank=rank, topk=5, window=2 * L + 5, sub_dim=sub,
                        summary_dtype=dtype, key_model="block_offset", shuffle_pages=True, seed=23, seq_lens=lens)
    inp = synth.generate(wl, "cuda")
    cfg = B.make_config(wl)
    summ = B.SummaryBuffers(cfg, "cuda", inp.get("u_q"))
    ws = B.alloc_workspace(cfg, "cuda")
    B.cobs_build_summaries(cfg, B.make_kv(inp), 0, wl.max_blocks, summ, ws)
    n = batch * hkv
    units = [divmod(u, hkv) for u in (0, 147, min(148, n - 1), n - 1)]
    run_stage_s(wl, inp_dev=inp, units=units, summ=summ)
    check_fused_equals_two_calls_on_every_unit(wl, inp, summ)
