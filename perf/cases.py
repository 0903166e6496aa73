"""What a user of this library has it do, as cases that can be timed.

The library serves one attention layer of a decoder: it builds a summary of every KV block as the cache fills
(prefill, and one block per sequence whenever a decode step fills one), and per decode step it scores all blocks,
selects the best and attends over them and the local window.  The cases call the ctypes binding and the decode loop
as a serving program does, from the one-sequence step whose latency counts to the long batch that fills the GPU.

Every kind of call:
  step      cobs_decode_step on device tensors: the fused decode step
  host      cobs_decode_step_host: the same with the query and the output in pinned host memory
  two_call  cobs_score_select, cobs_adaptive_trim, cobs_sparse_decode: the selection in the caller's hands
  exact     cobs_exact_select: the selection by exact block masses, the quality reference for the estimator
  tokens    DecodeLoop.step over several tokens of a ragged batch: append, rebuild the block that filled, step
  build     cobs_build_summaries over every block, as after a prefill

Steps take summaries that are not the builder's own (block means, and factors by a few rounds of subspace
iteration): a step's inputs are then a function of the seed alone."""

from __future__ import annotations

import math

import torch

from paper_2607_09052_b200 import binding as B
from paper_2607_09052_b200 import synth
from paper_2607_09052_b200.decode_loop import DecodeLoop


def _case(kind, **kw):
    """One case: the decode problem's sizes, the options, and the distribution of the keys and queries."""
    c = dict(kind=kind, batch=1, q_heads=32, kv_heads=8, head_dim=128, seq_len=32768, ragged=False, block=64, page=64,
             shuffled=False, rank=4, sub_dim=0, dtype="fp4", scale="fp32", skew=False, topk=16, window=512,
             keys="block_offset", planted=4, tokens=0)
    assert set(kw) <= set(c) | {"name"}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one short sequence, one KV head, fp32 summaries; only launches and latency count
        _case("step", name="step_2k_fp32", q_heads=4, kv_heads=1, head_dim=64, seq_len=2048, dtype="fp32", topk=4,
              window=64, keys="iid", planted=2),
        # interactive decode: one sequence of 32k tokens, bf16 summaries
        _case("step", name="step_32k_b1_bf16", dtype="bf16"),
        # the paper's descriptor (FP4 factors in an 85-dimensional query subspace) for a few sequences
        _case("step", name="step_32k_b4_subspace", batch=4, sub_dim=85),
        # serving: a ragged batch on 16-token pages in any order, an odd block count, small blocks, rank 6, fp16 scales
        _case("step", name="step_ragged_b24", batch=24, seq_len=375 * 32, ragged=True, block=32, page=16, shuffled=True,
              rank=6, scale="fp16", topk=24, window=256, keys="cov_perturb", planted=0),
        # the largest: sixteen sequences of 128k tokens, rank 8, scattered pages
        _case("step", name="step_128k_b16", batch=16, seq_len=131072, page=16, shuffled=True, rank=8, topk=64,
              keys="lowrank16", planted=0),
        # eight query heads per KV head, blocks of 128 tokens; query and output in the caller's host memory
        _case("host", name="host_step_64k_g8", batch=8, q_heads=64, seq_len=65536, block=128, page=128,
              keys="cov_perturb", planted=0),
        # the selection in the caller's hands: many blocks kept, trimmed to the share of the mass they hold
        _case("two_call", name="two_call_32k_k85", batch=4, topk=85),
        # how good the estimator's selection is: the same selection from every key
        _case("exact", name="exact_select_32k", batch=4),
        # sixteen tokens of a ragged batch of sixteen sequences, some of them filling a block on the way
        _case("tokens", name="tokens_16k_b16", batch=16, seq_len=16384, ragged=True, page=16, shuffled=True, planted=0,
              tokens=16),
        # after a prefill: every block of the long batch (four of its sequences), rank 8
        _case("build", name="build_128k_r8", batch=4, seq_len=131072, page=16, shuffled=True, rank=8,
              keys="lowrank16", planted=0),
        # blocks of 128 tokens
        _case("build", name="build_64k_l128", batch=8, q_heads=64, seq_len=65536, block=128, page=128,
              keys="cov_perturb", planted=0),
        # factors in the query subspace
        _case("build", name="build_32k_subspace", batch=4, sub_dim=85),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host", "two_call", "exact", "tokens", "build", "build", "build"])
    d = rng.choice([64, 128, 128])
    h = rng.choice([1, 2, 4, 8, 8])
    g = rng.choice([1, 2, 4, 4, 8])
    block = rng.choice([16, 32, 64, 64, 128])
    page = rng.choice([p for p in (16, 32, 64, 128) if p <= block])
    rank = rng.choice([1, 2, 3, 4, 4, 5, 6, 8, 8, 12, 16])
    # the builder's output is compared as it is stored, FP4: in a float type a factor whose two largest entries tie
    # could take either sign, which no bound on a difference allows
    dtype = "fp4" if kind in ("build", "tokens") else rng.choice(["fp4", "fp4", "fp4", "bf16", "bf16", "fp32"])
    sub = rng.randint(max(rank, d // 3), d - 1) if rng.random() < 0.3 else 0
    skew = dtype != "fp4" and sub == 0 and rng.random() < 0.3
    # capacity in blocks: any number of them; all sequences together no more than the largest listed case holds
    most = {"build": 1 << 22, "exact": 1 << 22, "tokens": 1 << 21}.get(kind, 1 << 24)
    if kind == "build" and (sub or rank > 8):
        most >>= 1
    n = max(2, _log(rng, 1024, 131072) // block)
    batch = _log(rng, 1, 64)
    if kind == "build":
        batch = max(batch, 4096 // (n * h * rank))
    batch = min(batch, max(1, most // (n * block * h)))
    keys = rng.choice(["iid", "block_offset", "lowrank16", "cov_perturb"])
    return _case(kind, batch=batch, q_heads=g * h, kv_heads=h, head_dim=d, seq_len=n * block, ragged=rng.random() < 0.5,
                 block=block, page=page, shuffled=rng.random() < 0.5, rank=rank, sub_dim=sub, dtype=dtype,
                 scale=rng.choice(["fp32", "fp16"]), skew=skew, topk=_log(rng, 4, 128), window=_log(rng, 32, 1024),
                 keys=keys, planted=rng.choice([0, 4]) if keys == "block_offset" and batch <= 8 else 0,
                 tokens=rng.randint(4, 16) if kind == "tokens" else 0)


def _lens(c):
    """Tokens in the cache per sequence: all of the capacity, or anything from a quarter of it up."""
    room = c["seq_len"] - c["tokens"]
    if not c["ragged"]:
        return [room] * c["batch"]
    return [max(1, room - (b * 7919 + 13) % max(1, 3 * room // 4)) for b in range(c["batch"])]


def _workload(c, seed):
    return synth.Workload(
        "case", c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"], c["seq_len"], c["block"], c["page"], c["rank"],
        c["topk"], c["window"], summary_dtype=c["dtype"], scale_dtype=c["scale"], sub_dim=c["sub_dim"],
        key_model=c["keys"], query_model="spectrum" if c["sub_dim"] and c["head_dim"] == 128 else "iid",
        planted=c["planted"], shuffle_pages=c["shuffled"], seed=seed, seq_lens=_lens(c))


def _fill_summaries(wl, cfg, inp, summ):
    """Summaries of every block, from torch: the mean, and r factors spanning (nearly) the leading directions."""
    nb, length, r, h, d = wl.max_blocks, wl.block_size, wl.rank, wl.n_kv_heads, wl.head_dim
    ds = wl.sub_dim or d
    xi = torch.empty((wl.batch, h, nb, r, ds), device="cuda")
    mean = torch.empty((wl.batch, h, nb, d), device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(wl.seed + 1)
    start = torch.randn((length, r), generator=gen, device="cuda")
    per = nb * length // wl.page_size
    for b in range(wl.batch):
        k = inp["k_pages"][inp["page_table"][b, :per].long()]                       # [pages, h, P, d]
        k = k.permute(1, 0, 2, 3).reshape(h, nb, length, d).float()
        m = k.mean(dim=2)
        kc = k - m[:, :, None]
        if wl.sub_dim:
            kc = torch.einsum("hnld,hds->hnls", kc, inp["u_q"])
        gram = kc @ kc.transpose(-1, -2)
        w = gram @ (gram @ (gram @ start))
        for i in range(r):                                                          # Gram-Schmidt
            for j in range(i):
                w[..., i] -= (w[..., i] * w[..., j]).sum(-1, keepdim=True) * w[..., j]
            w[..., i] /= w[..., i].norm(dim=-1, keepdim=True).clamp_min(1e-20)
        xi[b] = (w.transpose(-1, -2) @ kc) / math.sqrt(length)
        mean[b] = m
    mean_v, xi_v, scale_v = B.summary_views(cfg, summ)
    mean_v.copy_(mean)
    if wl.summary_dtype == "fp4":
        B.cobs_quantise_xi(cfg, xi.view(-1, ds), summ.xi, summ.scale)
    else:
        xi_v.copy_(xi)
    if summ.skew is not None:
        summ.skew.copy_(0.3 * torch.randn(summ.skew.shape, generator=gen, device="cuda"))


def prepare(case, seed):
    wl = _workload(case, seed)
    cfg = B.make_config(wl)
    inp = synth.generate(wl, device="cuda")
    kind, b, hq, h, d = case["kind"], wl.batch, wl.n_q_heads, wl.n_kv_heads, wl.head_dim
    s = {"kind": kind, "case": case, "cfg": cfg, "inp": inp, "kv": B.make_kv(inp), "ws": B.alloc_workspace(cfg, "cuda"),
         "q": inp["q"]}
    if kind != "exact":
        s["summ"] = B.SummaryBuffers(cfg, "cuda", inp.get("u_q"), skew=case["skew"])
        if kind != "build":
            _fill_summaries(wl, cfg, inp, s["summ"])
    s["sel"] = torch.full((b, h, wl.topk), -1, dtype=torch.int32, device="cuda")
    s["cnt"] = torch.zeros((b, h), dtype=torch.int32, device="cuda")
    s["out"] = torch.zeros((b, hq, d), device="cuda")
    s["lse"] = torch.zeros((b, hq), device="cuda")
    if kind == "host":
        s["q_host"] = inp["q"].cpu().pin_memory()
        s["out_host"] = torch.zeros((b, hq, d), pin_memory=True)
        s["sel_host"] = torch.full((b, h, wl.topk), -1, dtype=torch.int32, pin_memory=True)
        s["cnt_host"] = torch.zeros((b, h), dtype=torch.int32, pin_memory=True)
    if kind in ("two_call", "exact"):
        s["scores"] = torch.zeros((b, h, wl.max_blocks), device="cuda")
    if kind == "tokens":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n = case["tokens"]
        s["loop"] = DecodeLoop(wl, inp, s["summ"], s["ws"])
        s["lens"], s["lens_dev"] = list(s["loop"].lens), inp["seq_lens"].clone()
        s["qs"] = torch.randn((n, b, hq, d), generator=gen, device="cuda").bfloat16()
        s["ks"] = torch.randn((n, b, h, d), generator=gen, device="cuda").bfloat16()
        s["vs"] = torch.randn((n, b, h, d), generator=gen, device="cuda").bfloat16()
        s["outs"] = torch.zeros((n, b, hq, d), device="cuda")
    return s


def _summary_arrays(s):
    mean, xi, scale = B.summary_views(s["cfg"], s["summ"])
    return [mean, xi, scale, s["summ"].skew]


def run(s):
    cfg, ws, kind = s["cfg"], s["ws"], s["kind"]
    if kind == "step":
        B.cobs_decode_step(cfg, s["q"], s["kv"], s["summ"], s["out"], s["lse"], s["sel"], s["cnt"], ws)
        return [s["out"], s["lse"], s["sel"], s["cnt"]]
    if kind == "host":
        B.cobs_decode_step_host(cfg, s["q_host"], s["kv"], s["summ"], s["out_host"], s["sel_host"], s["cnt_host"], ws)
        return [s["out_host"], s["sel_host"], s["cnt_host"]]
    if kind == "two_call":
        B.cobs_score_select(cfg, s["q"], s["summ"], s["inp"]["seq_lens"], s["sel"], s["cnt"], s["scores"], ws)
        B.cobs_adaptive_trim(cfg, s["scores"], s["inp"]["seq_lens"], 0.05, 1, s["sel"], s["cnt"], ws)
        B.cobs_sparse_decode(cfg, s["q"], s["kv"], s["sel"], s["cnt"], s["out"], s["lse"], ws)
        return [s["out"], s["lse"], s["scores"], s["sel"], s["cnt"]]
    if kind == "exact":
        B.cobs_exact_select(cfg, s["q"], s["kv"], s["sel"], s["cnt"], s["scores"], ws)
        return [s["scores"], s["sel"], s["cnt"]]
    if kind == "build":
        B.cobs_build_summaries(cfg, s["kv"], 0, cfg.max_blocks, s["summ"], ws)
        return _summary_arrays(s)
    # tokens: from the same point of the sequences every time, as when speculated tokens are taken back
    loop = s["loop"]
    s["inp"]["seq_lens"].copy_(s["lens_dev"])
    loop.lens = list(s["lens"])
    for i in range(s["qs"].shape[0]):
        loop.step(s["qs"][i], s["ks"][i], s["vs"][i], s["outs"][i])
    return [s["outs"], s["inp"]["seq_lens"]] + _summary_arrays(s)


def _record_bytes(c):
    d, ds, r = c["head_dim"], c["sub_dim"] or c["head_dim"], c["rank"]
    skew = 4 * r if c["skew"] else 0
    if c["dtype"] == "fp32":
        return 4 * d + 4 * r * ds + skew
    if c["dtype"] == "bf16":
        return 2 * d + 2 * r * ds + skew
    return 2 * d + r * ((ds + 1) // 2 + (4 if c["scale"] == "fp32" else 2)) + skew


def work(case):
    """Bytes and operations of one pass that no implementation can do without."""
    c, d, h, length, r = case, case["head_dim"], case["kv_heads"], case["block"], case["rank"]
    g, ds = c["q_heads"] // h, c["sub_dim"] or d
    rec = _record_bytes(c)
    u_q = 4 * h * d * c["sub_dim"]
    n_bytes = flops = 0
    if c["kind"] == "build":
        n = sum(t // length for t in _lens(c)) * h
        # the Gram matrix (one half), its tridiagonal form, the factors; the projections where there is a subspace
        flops = n * (length * length * d + 4 * length ** 3 / 3 + 2 * r * length * d + (2 * r * d * ds if c["sub_dim"] else 0))
        return {"bytes": n * (length * d * 2 + rec) + u_q, "flops": flops}
    if c["kind"] == "exact":
        tok = sum(t // length * length for t in _lens(c))
        units = c["batch"] * h
        return {"bytes": tok * h * d * 2 + units * (c["topk"] * 4 + 4 + g * d * 2) + tok // length * h * 4,
                "flops": 2 * tok * h * g * d}
    for step in range(max(1, c["tokens"])):
        for t in _lens(c):
            t += step + 1 if c["tokens"] else 0
            ws = max(0, t - c["window"]) // length * length
            kv = min(c["topk"], ws // length) * length + t - ws
            n_sum = t // length
            n_bytes += h * (n_sum * rec + kv * d * 4) + c["q_heads"] * d * 6
            flops += h * g * (2 * n_sum * (d + r * ds) + 4 * kv * d)
            if c["kind"] == "two_call":
                n_bytes += 2 * h * n_sum * 4
            if c["tokens"]:
                n_bytes += h * d * 8
                if t % length == 0:
                    n_bytes += h * (length * d * 2 + rec)
                    flops += h * (length * length * d + 4 * length ** 3 / 3 + 2 * r * length * d)
        n_bytes += u_q
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    """Measured against the same computation in 64 bits (scores, attention) and against the library's other
    eigen-solver (build), times about four.  Two blocks whose scores differ by less than their rounding may change
    places at the end of a selection, about one unit in a thousand of the largest case: the output of such a unit moves
    by the weight of one block, which is what the bounds of the step allow; without one it agrees to 1e-5."""
    if case["kind"] == "build":
        return {"rel": 2e-4, "max": 0.5, "differ": 2e-3}          # nearly equal eigenvalues turn their factors
    if case["kind"] == "exact":
        return {"rel": 5e-5, "differ": 1e-2}
    return {"rel": 3e-3, "max": 0.3, "differ": 1e-2}
