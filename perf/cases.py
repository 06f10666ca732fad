"""Timing cases of the verification path: what a serving process has the library do, from one small float32 layer to
a 128K-token cache of 32 layers.

Kinds of pass
  step     the layer-batched step of `bench.py`: tree mask, full verification, commit with summaries, block scores,
           selection, gather, then tree mask, partial verification and commit into the buffer
  loop     one refresh period of a decode loop: a refresh over the partially verified chain and the tree, followed by
           partial steps whose accepted tokens fill the buffer
  block    the attention block the way a model runs it, layer after layer: rope table, then per layer the QKV
           projection, the verification (partial or full cache) and the output projection; `graph` replays the same
           calls from a CUDA graph
  attend   the verification alone, one call per layer
  prefill  what follows a prefill: summaries of the whole cache, first scores, selection and gather
  host     the entry point with step tensors in pinned host memory, full and partial verification

Geometries: the head shapes of LLaMA-3.1-8B and Qwen3-8B (32 query and 8 KV heads of 128), of Qwen3-14B (40 and 8),
head size 64, the tiny float32 configuration; pages of 16, 32 and 64 tokens; draft trees of 8 to 64 nodes, chains of up
to 42 tokens; budgets of 512 to 8192 tokens.  Verification over a cache in host memory is left out: it runs at the rate
of the host link.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_02337_b200 import binding as B
from paper_2512_02337_b200 import workloads as wl

BASE = dict(layers=32, hq=32, hkv=8, d=128, bs=64, dtype="bf16", m=60, depth=6, branch=4, budget=64, chain=0,
            partial_steps=1, reduce=0, score_mode=0, shared=False, shuffle=False, hidden=0, graph=False, cache="partial")


def _case(name, kind, ctx, **over):
    c = dict(BASE, kind=kind, ctx=ctx, **over)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the tiny float32 configuration: the smallest step, bound by launches and latency
        _case("fp32_tiny_step", "step", "2048", layers=1, hq=8, hkv=2, d=64, dtype="fp32", m=16, depth=4, budget=8),
        # context still shorter than the budget: every step verifies fully over a short cache, head size 64
        _case("short_full_d64", "attend", "1500,811", layers=16, d=64, m=26, depth=5, cache="full"),
        # one decode step of a LLaMA-3.1-8B-shaped model, layer after layer, 4096-token budget
        _case("block_partial_4k", "block", "16384", layers=32, hidden=4096),
        # the same captured once and replayed, a small tree and the 2048-token budget
        _case("block_partial_2k_graph", "block", "8192", layers=32, m=24, depth=5, budget=32, hidden=4096, graph=True),
        # a refresh step of Qwen3-14B's head geometry (five query heads per KV head), layer after layer
        _case("block_full_g5", "block", "12345", layers=10, hq=40, m=48, depth=5, hidden=5120, cache="full"),
        # the benchmark's step at 32K and at 128K
        _case("step_32k", "step", "32768"),
        _case("step_128k", "step", "131072"),
        # one refresh period of the 64K decode loop: chain of 42 and tree of 48, then partial steps
        _case("loop_64k", "loop", "65536", layers=36, m=48, depth=5, chain=42, partial_steps=6),
        # the paper's own settings: 16-token blocks, 512-token budget, buffer of 20 tokens beyond the tree
        _case("loop_pages16_60k", "loop", "61440", layers=16, bs=16, m=60, budget=32, chain=18, partial_steps=5),
        # ragged batch of four with a shuffled block table
        _case("batch4_ragged_step", "step", "98304,114688,122880,131072", layers=6, m=64, shuffle=True),
        # after the prefill of a 96K-token prompt
        _case("prefill_96k", "prefill", "98309", layers=32),
        # step tensors in host memory
        _case("host_32k", "host", "32768", layers=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "loop", "block", "block", "block", "attend", "prefill", "host"])
    m = rng.randint(8, 64)
    over = dict(m=m, depth=rng.randint(4, 7), branch=rng.randint(3, 5))
    geometry = rng.choice(["g4", "g4", "g4", "g4", "g5", "d64", "fp32"])
    if kind in ("loop", "prefill", "host") and geometry != "fp32":
        geometry = "g4"
    if geometry == "fp32":
        kind = rng.choice(["step", "attend"])
        over.update(dtype="fp32", layers=rng.randint(1, 4), hq=8, hkv=2, d=64, m=min(m, 32))
        ctx = [_log_int(rng, 600, 8192)]
        over["budget"] = 8
    else:
        if geometry == "g5":
            over.update(hq=40)
        if geometry == "d64":
            over.update(d=64)
        batch = rng.choice([1, 1, 1, 2, 3, 4])
        top = 131072 if geometry == "g4" else 16384
        longest = _log_int(rng, 3000, top)
        ctx = [longest if b == 0 else rng.randint(longest // 2, longest) for b in range(batch)]
        # layers so that the cache stays below 9 GB, and far below that for the shapes of the plain kernels
        most = (9e9 if geometry == "g4" else 0.35e9) / (batch * longest * 8 * 2 * 128 * 2)
        over["layers"] = max(1, min(rng.choice([8, 16, 24, 32, 36]), int(most)))
        over["bs"] = rng.choice([16, 32, 64, 64, 64])
        over["budget"] = rng.choice([1024, 2048, 2048, 4096, 4096, 8192]) // over["bs"]
        over["shuffle"] = rng.random() < 0.3
        over["reduce"] = rng.choice([0, 0, 0, 1, 2])
        over["score_mode"] = int(rng.random() < 0.15)
        over["shared"] = rng.random() < 0.15
        if kind == "loop":
            over["chain"] = rng.randint(4, 42)
            over["partial_steps"] = rng.randint(2, 6)
        if kind == "block":
            over["hidden"] = 5120 if geometry == "g5" else rng.choice([2560, 4096])
            over["graph"] = rng.random() < 0.5
        if kind in ("block", "attend"):
            over["cache"] = rng.choice(["partial", "full"])
    # the partial cache must be smaller than the context it is selected from
    while over["budget"] > 4 and over["budget"] * over.get("bs", 64) > min(ctx) // 2:
        over["budget"] //= 2
    sink, local = wl.sink_local_blocks(over.get("bs", 64))
    over["budget"] = max(over["budget"], sink + local + 1)
    case = _case(None, kind, ",".join(str(c) for c in ctx), **over)
    largest = work(next(c for c in listed() if c["name"] == "step_128k"))
    while any(work(case)[k] > 0.9 * largest[k] for k in largest):  # no more than the largest listed case
        case["layers"] -= case["layers"] // 4 or 1
    return case


# ---- what a program holds before the call --------------------------------------------------------------------------
ACCEPT = 4  # tokens accepted per step: the paper's mean accept length is 3.3-3.6, plus the root


def _ctx(case):
    return [int(c) for c in case["ctx"].split(",")]


def _buffer(case):
    return 20 + case["m"] if case["bs"] == 16 else case["chain"] + case["m"] + ACCEPT * case["partial_steps"]


def _parents(case, rng):
    return [wl.make_tree(case["m"], case["depth"], case["branch"], rng) for _ in _ctx(case)]


def _accepted(case, parents, device):
    """Chain rows, then a root-to-node path of the tree (indices into the step's rows)."""
    rows = []
    for p in parents:
        path = max((wl.path_to(p, n) for n in range(len(p))), key=lambda q: min(len(q), ACCEPT))[:ACCEPT]
        rows.append(path)
    n = len(rows[0])
    tree = np.stack([r[:n] for r in rows]).astype(np.int32)
    chain = np.tile(np.arange(case["chain"], dtype=np.int32), (len(parents), 1))
    refresh = np.concatenate([chain, tree + case["chain"]], axis=1)
    count = torch.full((len(parents),), n, dtype=torch.int32, device=device)
    return (torch.from_numpy(np.ascontiguousarray(tree)).to(device), count,
            torch.from_numpy(np.ascontiguousarray(refresh)).to(device), count + case["chain"])


def prepare(case, seed):
    dev = torch.device("cuda")
    L, hq, hkv, d, bs, m, chain = (case[k] for k in ("layers", "hq", "hkv", "d", "bs", "m", "chain"))
    ctx, rows = _ctx(case), case["m"] + case["chain"]
    kind = case["kind"]
    host_rng = np.random.default_rng(seed)
    w = wl.make_workload("tiny_fp32" if case["dtype"] == "fp32" else "llama_32k", device=dev, n_layers=L, spare_tokens=128,
                         index=int(seed), Hq=hq, Hkv=hkv, d=d, bs=bs, ctx=ctx, M=rows, depth=rows, branch=2,
                         shuffle=case["shuffle"])
    batch, dt = len(ctx), wl.torch_dtype(case["dtype"])
    sink, local = wl.sink_local_blocks(bs)
    buffer = _buffer(case)
    cfg = B.make_config(L, hq, hkv, d, bs, case["dtype"], sink, local, case["budget"], buffer, reduce=case["reduce"],
                        score_mode=case["score_mode"], select_shared=int(case["shared"]))
    per_call = 1 if kind in ("block", "attend") else L
    max_len = max(ctx) + 128
    s = dict(case=case, cfg=cfg, w=w, L=L, m=m, rows=rows, batch=batch, parents=_parents(case, host_rng))
    s["ws"] = B.new_workspace(cfg, per_call, batch, max_len, rows, device=dev)
    s["full"] = B.Cache(w.k_pool, w.v_pool, w.block_table, w.seq_lens, max_len)
    ppb = case["budget"] + (buffer + bs - 1) // bs + 1
    pk = torch.zeros((L, batch * ppb, hkv, bs, d), dtype=dt, device=dev)
    ptable = torch.arange(batch * ppb, dtype=torch.int32, device=dev).reshape(batch, ppb).contiguous()
    s["partial"] = B.Cache(pk, torch.zeros_like(pk), ptable, torch.zeros(batch, dtype=torch.int32, device=dev),
                           case["budget"] * bs + buffer)
    s["kmax"] = torch.zeros((L, batch, hkv, w.max_blocks, d), dtype=dt, device=dev)
    s["kmin"] = torch.zeros_like(s["kmax"])
    s["scores"] = torch.zeros((L, batch, hkv, w.max_blocks), dtype=torch.float32, device=dev)
    s["idx"] = torch.zeros((L, batch, hkv, case["budget"]), dtype=torch.int32, device=dev)
    s["count"] = torch.zeros(batch, dtype=torch.int32, device=dev)
    s["last"] = torch.full((batch,), chain, dtype=torch.int32, device=dev)  # the tree's root
    s["lens0"] = w.seq_lens.clone()
    s["accepted"], s["n_accepted"], s["accepted_refresh"], s["n_refresh"] = _accepted(case, s["parents"], dev)
    words, twords = (rows + 63) // 64, (m + 63) // 64
    s["mask_host"] = torch.zeros((batch, rows, words), dtype=torch.int64).pin_memory()
    s["tmask_host"] = torch.zeros((batch, m, twords), dtype=torch.int64).pin_memory()
    s["mask"], s["tmask"] = s["mask_host"].to(dev), s["tmask_host"].to(dev)
    s["out"] = torch.zeros((L, batch, rows, hq, d), dtype=dt, device=dev)
    s["lse"] = torch.zeros((L, batch, rows, hq), dtype=torch.float32, device=dev)
    # the tree's own step tensors in a partial step
    s["tq"], s["tk"], s["tv"] = (t[:, :, chain:].contiguous() for t in (w.q, w.k_new, w.v_new))
    s["touts"] = [torch.zeros((L, batch, m, hq, d), dtype=dt, device=dev) for _ in range(case["partial_steps"])]
    s["tlses"] = [torch.zeros((L, batch, m, hq), dtype=torch.float32, device=dev) for _ in range(case["partial_steps"])]
    if kind != "prefill":
        B.specpv_update_block_summaries(cfg, 0, L, s["full"], None, w.max_blocks, s["kmax"], s["kmin"], s["ws"])
    if kind in ("host", "block", "attend"):
        # a partial cache filled by an earlier refresh
        B.specpv_score_blocks(cfg, 0, L, w.q, None, rows, s["last"], s["kmax"], s["kmin"], s["full"], s["scores"], s["ws"])
        B.specpv_select_partial_kv(cfg, L, s["scores"], w.seq_lens, batch, w.max_blocks, s["idx"], s["count"], s["ws"])
        B.specpv_refresh_partial(cfg, s["full"], s["idx"], s["count"], s["partial"], s["partial"].seq_lens, s["ws"])
        _masks(s, refresh=False)
    if kind == "host":
        s["host"] = [t.cpu().pin_memory() for t in (s["tq"], s["tk"], s["tv"])]
        s["host_out"] = [torch.zeros((L, batch, m, hq, d), dtype=dt).pin_memory() for _ in range(2)]
        s["host_lse"] = [torch.zeros((L, batch, m, hq), dtype=torch.float32).pin_memory() for _ in range(2)]
    if kind in ("block", "attend"):
        cache = s["cache"] = s["partial"] if case["cache"] == "partial" else s["full"]
        hid = case["hidden"]
        layers = []
        if hid:
            bw = s["bw"] = wl.make_block_weights("llama_32k", device=dev, n_layers=L, M=m, hidden=hid, index=int(seed), Hq=hq,
                                                 Hkv=hkv, d=d, ctx=ctx)
            s["y"] = torch.zeros_like(bw.x)
            s["base"] = w.seq_lens.clone()
            s["cos_sin"] = torch.zeros((batch, m, d // 2, 2), dtype=torch.float32, device=dev)
        for i in range(L):  # a layer's own buffers, as the module of that layer would hold them
            views = [t[i:i + 1] for t in (s["tq"], s["tk"], s["tv"], s["touts"][0], s["tlses"][0])]
            layers.append(views + ([t[i:i + 1] for t in (bw.x, bw.residual, s["y"])] if hid else []))
        s["layers"] = layers
        if case["graph"]:
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                _layers(s)
            torch.cuda.current_stream().wait_stream(side)
            torch.cuda.synchronize()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                _layers(s)
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------
def _masks(s, refresh):
    name, chain = ("mask", s["case"]["chain"]) if refresh else ("tmask", 0)
    host = s[name + "_host"].numpy().view(np.uint64)
    for b in range(s["batch"]):
        host[b] = B.specpv_build_tree_mask(s["parents"][b], chain, host.shape[2])
    s[name].copy_(s[name + "_host"], non_blocking=True)


def _refresh(s):
    cfg, w, L, rows, ws, full, partial = s["cfg"], s["w"], s["L"], s["rows"], s["ws"], s["full"], s["partial"]
    _masks(s, refresh=True)
    B.specpv_verify_full(cfg, 0, L, w.q, w.k_new, w.v_new, s["mask"], None, rows, full, s["out"], s["lse"], ws)
    acc = s["accepted_refresh"]
    B.specpv_commit_accepted(cfg, 0, L, w.k_new, w.v_new, rows, acc, s["n_refresh"], acc.shape[1], full, s["kmax"],
                             s["kmin"], ws)
    B.specpv_score_blocks(cfg, 0, L, w.q, None, rows, s["last"], s["kmax"], s["kmin"], full, s["scores"], ws)
    B.specpv_select_partial_kv(cfg, L, s["scores"], w.seq_lens, s["batch"], w.max_blocks, s["idx"], s["count"], ws)
    B.specpv_refresh_partial(cfg, full, s["idx"], s["count"], partial, partial.seq_lens, ws)


def _partial_step(s, i):
    cfg, L, m, ws, partial, acc = s["cfg"], s["L"], s["m"], s["ws"], s["partial"], s["accepted"]
    _masks(s, refresh=False)
    B.specpv_verify_partial(cfg, 0, L, s["tq"], s["tk"], s["tv"], s["tmask"], None, m, partial, s["touts"][i],
                            s["tlses"][i], ws)
    B.specpv_commit_accepted(cfg, 0, L, s["tk"], s["tv"], m, acc, s["n_accepted"], acc.shape[1], partial, None, None, ws)


def _layers(s):
    cfg, case, m, ws, cache, batch = s["cfg"], s["case"], s["m"], s["ws"], s["cache"], s["batch"]
    verify = B.specpv_verify_partial if case["cache"] == "partial" else B.specpv_verify_full
    hid = case["hidden"]
    if hid:
        bw = s["bw"]
        B.specpv_rope_table(cfg, s["tmask"], None, s["base"], batch, m, bw.rope_theta, s["cos_sin"])
    for i, views in enumerate(s["layers"]):
        q, k, v, out, lse = views[:5]
        if hid:
            x, residual, y = views[5:]
            B.specpv_qkv_rope(cfg, i, 1, x, hid, bw.w_qkv, s["cos_sin"], batch, m, q, k, v, ws)
        verify(cfg, i, 1, q, k, v, s["tmask"], None, m, cache, out, lse, ws)
        if hid:
            B.specpv_o_proj(cfg, i, 1, out, bw.w_o, hid, residual, batch, m, y, ws)


def run(state):
    s, kind, w = state, state["case"]["kind"], state["w"]
    partial = s["partial"]
    if kind in ("step", "loop"):
        _refresh(s)
        for i in range(s["case"]["partial_steps"]):
            _partial_step(s, i)
        w.seq_lens.copy_(s["lens0"], non_blocking=True)  # the next pass starts from the same lengths
        return {"out": s["out"], "lse": s["lse"], "scores": s["scores"], "idx": s["idx"], "count": s["count"],
                "partial_out": s["touts"], "partial_lse": s["tlses"], "partial_k": partial.k_pool,
                "partial_v": partial.v_pool, "partial_lens": partial.seq_lens, "kmax": s["kmax"], "kmin": s["kmin"]}
    if kind in ("block", "attend"):
        if s["case"]["graph"]:
            s["graph"].replay()
        else:
            _layers(s)
        outs = {"out": s["touts"][0], "lse": s["tlses"][0]}
        return dict(outs, y=s["y"], q=s["tq"], k=s["tk"], v=s["tv"]) if s["case"]["hidden"] else outs
    if kind == "prefill":
        cfg, L, ws, full = s["cfg"], s["L"], s["ws"], s["full"]
        B.specpv_update_block_summaries(cfg, 0, L, full, None, w.max_blocks, s["kmax"], s["kmin"], ws)
        B.specpv_score_blocks(cfg, 0, L, w.q, None, s["rows"], s["last"], s["kmax"], s["kmin"], full, s["scores"], ws)
        B.specpv_select_partial_kv(cfg, L, s["scores"], w.seq_lens, s["batch"], w.max_blocks, s["idx"], s["count"], ws)
        B.specpv_refresh_partial(cfg, full, s["idx"], s["count"], partial, partial.seq_lens, ws)
        return {"kmax": s["kmax"], "kmin": s["kmin"], "scores": s["scores"], "idx": s["idx"], "partial_k": partial.k_pool,
                "partial_v": partial.v_pool, "partial_lens": partial.seq_lens}
    cfg, L, m, ws, (q, k, v) = s["cfg"], s["L"], s["m"], s["ws"], s["host"]
    for i, (mode, cache) in enumerate(((B.MODE_FULL, s["full"]), (B.MODE_PARTIAL, partial))):
        B.specpv_verify_host(cfg, mode, 0, L, q, k, v, s["tmask_host"], m, cache, s["host_out"][i], s["host_lse"][i], ws)
    return {"out": s["host_out"], "lse": s["host_lse"]}


# ---- what a pass cannot do without ---------------------------------------------------------------------------------
def work(case):
    L, hq, hkv, d, bs, m, chain = (case[k] for k in ("layers", "hq", "hkv", "d", "bs", "m", "chain"))
    es = 4 if case["dtype"] == "fp32" else 2
    ctx, kind, rows = _ctx(case), case["kind"], case["m"] + case["chain"]
    part = [min(c, case["budget"] * bs) for c in ctx]
    blocks = sum((c + bs - 1) // bs for c in ctx)
    summaries = 2 * L * blocks * hkv * d * es

    def attention(tokens, r):
        n = len(tokens)
        nbytes = L * (sum(tokens) * hkv * 2 * d * es + n * r * (2 * hq + 2 * hkv) * d * es + n * r * hq * 4)
        return nbytes, sum(4.0 * L * r * hq * (t + r) * d for t in tokens)

    def refresh_rest(r):
        nbytes = summaries + L * len(ctx) * r * hq * d * es + 2 * L * sum(part) * hkv * 2 * d * es
        return nbytes, 4.0 * L * r * hq * blocks * d

    def total(*parts):
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}

    if kind in ("step", "loop"):
        steps = [attention([p + i * ACCEPT for p in part], m) for i in range(case["partial_steps"])]
        return total(attention(ctx, rows), refresh_rest(rows), *steps)
    if kind == "prefill":
        return total((L * sum(ctx) * hkv * d * es, 2.0 * L * sum(ctx) * hkv * d), (summaries, 0.0), refresh_rest(rows))
    if kind == "host":
        return total(attention(ctx, m), attention(part, m))
    parts = [attention(part if case["cache"] == "partial" else ctx, m)]
    if case["hidden"]:
        hid, n = case["hidden"], len(ctx) * m
        feats = (hq + 2 * hkv) * d + hq * d
        parts.append((L * es * (feats * hid + n * (3 * hid + (hq + 2 * hkv) * d + hq * d)), 2.0 * L * n * feats * hid))
    return total(*parts)


def tolerance(case):
    # measured against float64: bf16 outputs rel 1.9e-3 (1.7e-3 of it the rounding of the output), max 1.5e-2 (P is
    # rounded to bf16 before P V); float32 outputs rel 6e-7, max 3e-6 (sums in another order).  Copies and maxima are
    # exact; block lists may differ where two scores tie within rounding.
    if case["dtype"] == "fp32":
        return {"rel": 3e-6, "max": 3e-5, "differ": 2e-3}
    return {"rel": 8e-3, "max": 6e-2, "differ": 2e-3}
