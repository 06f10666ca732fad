"""GPU parity of the whole hot path on the tiny float32 config and on a small bfloat16 shape:
summaries, scores, selection, gather, partial and full verification, commit -- each compared with the
CPU oracle through the C ABI."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_02337_b200 import binding as B
from paper_2512_02337_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu


def run_pipeline(name, n_layers=None, reduce=0, score_mode=0, select_shared=0, **over):
    w = wl.make_workload(name, device="cuda", n_layers=n_layers, spare_tokens=256, **over)
    c = w.cfg
    L, Hq, Hkv, d, bs, M = c["n_layers"], c["Hq"], c["Hkv"], c["d"], c["bs"], c["M"]
    batch = w.batch
    cfg = util.config_for(w, reduce=reduce, score_mode=score_mode, select_shared=select_shared)
    full = util.full_cache(w)
    full.max_seq_len = int(max(c["ctx"])) + 256
    ws = B.new_workspace(cfg, L, batch, full.max_seq_len, M)
    dt = wl.torch_dtype(c["dtype"])
    dev = w.device
    mask = util.device_masks(w.parents, M)
    last_query = torch.zeros(batch, dtype=torch.int32, device=dev)

    # ---- Eq. 1 summaries: bit-exact
    kmax = torch.zeros((L, batch, Hkv, w.max_blocks, d), dtype=dt, device=dev)
    kmin = torch.zeros_like(kmax)
    B.specpv_update_block_summaries(cfg, 0, L, full, None, w.max_blocks, kmax, kmin, ws)
    # ---- Eq. 2-3 scores
    scores = torch.full((L, batch, Hkv, w.max_blocks), float("nan"), dtype=torch.float32, device=dev)
    B.specpv_score_blocks(cfg, 0, L, w.q, None, M, last_query, kmax, kmin, full, scores, ws)
    # ---- selection
    idx = torch.full((L, batch, Hkv, cfg.budget_blocks), -7, dtype=torch.int32, device=dev)
    count = torch.zeros(batch, dtype=torch.int32, device=dev)
    B.specpv_select_partial_kv(cfg, L, scores, w.seq_lens, batch, w.max_blocks, idx, count, ws)
    # ---- gather into the partial cache (pages of sequence b: [b*ppb, (b+1)*ppb), identity table)
    ppb = cfg.budget_blocks + (cfg.buffer_tokens + bs - 1) // bs + 1
    pk = torch.zeros((L, batch * ppb, Hkv, bs, d), dtype=dt, device=dev)
    pv = torch.zeros_like(pk)
    ptable = torch.arange(batch * ppb, dtype=torch.int32, device=dev).reshape(batch, ppb)
    plens = torch.zeros(batch, dtype=torch.int32, device=dev)
    partial = B.Cache(pk, pv, ptable, plens, cfg.budget_blocks * bs + cfg.buffer_tokens)
    B.specpv_refresh_partial(cfg, full, idx, count, partial, plens, ws)
    # ---- verification
    out_full = torch.zeros((L, batch, M, Hq, d), dtype=torch.float32, device=dev)
    lse_full = torch.zeros((L, batch, M, Hq), dtype=torch.float32, device=dev)
    out_part, lse_part = torch.zeros_like(out_full), torch.zeros_like(lse_full)
    B.specpv_verify_full(cfg, 0, L, w.q, w.k_new, w.v_new, mask, None, M, full, out_full, lse_full, ws)
    B.specpv_verify_partial(cfg, 0, L, w.q, w.k_new, w.v_new, mask, None, M, partial, out_part, lse_part, ws)
    if c["dtype"] == "bf16":  # the bfloat16 output is the float32 one, rounded
        cfg16 = util.config_for(w, reduce=reduce, score_mode=score_mode, select_shared=select_shared, out_f32=0)
        o16f, o16p = torch.zeros_like(out_full, dtype=dt), torch.zeros_like(out_full, dtype=dt)
        B.specpv_verify_full(cfg16, 0, L, w.q, w.k_new, w.v_new, mask, None, M, full, o16f, None, ws)
        B.specpv_verify_partial(cfg16, 0, L, w.q, w.k_new, w.v_new, mask, None, M, partial, o16p, None, ws)
        util.same_as_rounded(o16f, out_full)
        util.same_as_rounded(o16p, out_part)
    util.sync_status(ws)

    seq_lens = w.seq_lens.cpu().numpy()
    table = w.block_table.cpu().numpy()
    kp, vp = wl.to_numpy(w.k_pool), wl.to_numpy(w.v_pool)
    qn, knn, vnn = wl.to_numpy(w.q), wl.to_numpy(w.k_new), wl.to_numpy(w.v_new)
    kmax_g, kmin_g = util.widen_t(kmax), util.widen_t(kmin)
    scores_g, idx_g, count_g = scores.cpu().numpy(), idx.cpu().numpy(), count.cpu().numpy()
    pk_g, pv_g, plens_g = wl.to_numpy(pk), wl.to_numpy(pv), plens.cpu().numpy()
    sink, local = cfg.sink_blocks, cfg.local_blocks
    for l in range(L):
        for b in range(batch):
            sl = int(seq_lens[b])
            nb = (sl + bs - 1) // bs
            okmax, okmin = oracle.block_summaries(kp[l], table[b], sl)
            assert np.array_equal(kmax_g[l, b, :, :nb], okmax) and np.array_equal(kmin_g[l, b, :, :nb], okmin)
            osc = oracle.block_scores(qn[l, b], okmax, okmin, Hkv, reduce=reduce, last_query=0, score_mode=score_mode)
            np.testing.assert_allclose(scores_g[l, b, :, :nb], osc, rtol=2e-3 if c["dtype"] == "bf16" else 2e-5,
                                       atol=2e-2 if c["dtype"] == "bf16" else 2e-4)
            assert np.all(np.isnan(scores_g[l, b, :, nb:]))  # untouched beyond the context
            n_keep = min(nb, cfg.budget_blocks)
            assert count_g[b] == n_keep
            if select_shared:  # one list per (layer, sequence), ranked on the mean over the heads
                for h in range(1, Hkv):
                    assert np.array_equal(idx_g[l, b, h, :n_keep], idx_g[l, b, 0, :n_keep])
                util.check_shared_selection(idx_g[l, b, 0, :n_keep], scores_g[l, b, :, :nb], sink, local,
                                            cfg.budget_blocks, f"shared selection l{l} b{b}")
                oidx = idx_g[l, b, :, :n_keep].copy()  # the list the gather below has to follow
            else:
                oidx = np.stack([oracle.select(scores_g[l, b, h, :nb].astype(np.float64), sink, local, cfg.budget_blocks)
                                 for h in range(Hkv)])
                assert np.array_equal(idx_g[l, b, :, :n_keep], oidx)  # bit-exact given the same float32 scores
            opk, opv = np.zeros_like(pk_g[l]), np.zeros_like(pv_g[l])
            oplen = oracle.gather(kp[l], vp[l], table[b], sl, oidx, opk, opv, first_page=b * ppb)
            assert plens_g[b] == oplen
            first, last = b * ppb, b * ppb + n_keep
            gk, gv = pk_g[l, first:last].copy(), pv_g[l, first:last].copy()
            tail = oplen - (n_keep - 1) * bs
            gk[-1, :, tail:], gv[-1, :, tail:] = 0, 0   # tokens past the ragged end are unspecified
            assert np.array_equal(gk, opk[first:last]) and np.array_equal(gv, opv[first:last])
            omask = oracle.tree_mask(w.parents[b])
            assert np.array_equal(omask, B.specpv_build_tree_mask(w.parents[b]))
            o_out, o_lse = oracle.tree_attention(qn[l, b], knn[l, b], vnn[l, b], omask, kp[l], vp[l], table[b], sl)
            util.compare(util.widen_t(out_full[l, b]), o_out, c["dtype"], f"full out l{l} b{b}")
            np.testing.assert_allclose(lse_full[l, b].cpu().numpy(), o_lse, atol=2e-5 if c["dtype"] == "fp32" else 5e-3)
            p_out, p_lse = oracle.tree_attention(qn[l, b], knn[l, b], vnn[l, b], omask, opk, opv,
                                                 ptable[b].cpu().numpy(), oplen)
            util.compare(util.widen_t(out_part[l, b]), p_out, c["dtype"], f"partial out l{l} b{b}")
            np.testing.assert_allclose(lse_part[l, b].cpu().numpy(), p_lse, atol=2e-5 if c["dtype"] == "fp32" else 5e-3)
    return w, cfg, full, partial, ws, (kmax, kmin)


def test_tiny_fp32_config_every_step_matches_oracle():
    run_pipeline("tiny_fp32")


@pytest.mark.parametrize("reduce", [1, 2])
def test_tiny_fp32_other_reductions(reduce):
    run_pipeline("tiny_fp32", reduce=reduce)


def test_small_bf16_llama_shape_pipeline():
    # the 32K LLaMA geometry cut down to 2 layers and 6K tokens so that the oracle covers every row
    run_pipeline("llama_32k", n_layers=2, ctx=[6144 + 37], M=60)


@pytest.mark.parametrize("reduce", [1, 2])
def test_small_bf16_other_reductions(reduce):
    # max / last reductions through the tensor-core score kernel, M = 20 (80 query rows: one Q tile)
    run_pipeline("llama_32k", n_layers=1, reduce=reduce, ctx=[64 * 150 + 11], M=20)


@pytest.mark.parametrize("reduce", [0, 1])
def test_channelwise_score_mode_fp32_and_bf16(reduce):
    # score_mode 1: the maximum is taken per channel; selection, gather and partial verification follow from it
    run_pipeline("tiny_fp32", reduce=reduce, score_mode=1)
    run_pipeline("llama_32k", n_layers=1, reduce=reduce, score_mode=1, ctx=[64 * 90 + 3], M=33)


def test_head_shared_selection_fp32_and_bf16():
    # one block set per (layer, sequence): every head gathers and attends the blocks ranked on the heads' mean score
    run_pipeline("tiny_fp32", select_shared=1)
    run_pipeline("llama_32k", n_layers=2, select_shared=1, ctx=[64 * 120 + 9], M=25)


def test_ragged_batch_shuffled_table_pipeline():
    run_pipeline("stress_b4", n_layers=1, ctx=[4096 + 5, 4800, 5120 - 1, 5120], M=64)


def test_commit_appends_and_updates_summaries():
    w, cfg, full, partial, ws, (kmax, kmin) = run_pipeline("tiny_fp32")
    c = w.cfg
    L, Hkv, d, bs, M = c["n_layers"], c["Hkv"], c["d"], c["bs"], c["M"]
    dev = w.device
    path = wl.path_to(w.parents[0], int(np.argmax([len(wl.path_to(w.parents[0], n)) for n in range(M)])))
    A_max = 8
    acc = torch.zeros((1, A_max), dtype=torch.int32, device=dev)
    acc[0, :len(path)] = torch.from_numpy(path).to(dev)
    n_acc = torch.tensor([len(path)], dtype=torch.int32, device=dev)
    kp0, vp0 = wl.to_numpy(w.k_pool).copy(), wl.to_numpy(w.v_pool).copy()
    sl0 = int(w.seq_lens[0])
    pl0 = int(partial.seq_lens[0])
    ppk0, ppv0 = wl.to_numpy(partial.k_pool).copy(), wl.to_numpy(partial.v_pool).copy()
    # full cache (with summaries) and partial cache (buffer append, no summaries)
    B.specpv_commit_accepted(cfg, 0, L, w.k_new, w.v_new, M, acc, n_acc, A_max, full, kmax, kmin, ws)
    B.specpv_commit_accepted(cfg, 0, L, w.k_new, w.v_new, M, acc, n_acc, A_max, partial, None, None, ws)
    util.sync_status(ws)
    assert int(w.seq_lens[0]) == sl0 + len(path) and int(partial.seq_lens[0]) == pl0 + len(path)
    table = w.block_table.cpu().numpy()
    knn, vnn = wl.to_numpy(w.k_new), wl.to_numpy(w.v_new)
    for l in range(L):
        new_len = oracle.commit(knn[l, 0], vnn[l, 0], path, kp0[l], vp0[l], table[0], sl0)
        assert new_len == sl0 + len(path)
        oracle.commit(knn[l, 0], vnn[l, 0], path, ppk0[l], ppv0[l], partial.block_table[0].cpu().numpy(), pl0)
        okmax, okmin = oracle.block_summaries(kp0[l], table[0], new_len)
        nb = (new_len + bs - 1) // bs
        assert np.array_equal(util.widen_t(kmax[l, 0])[:, :nb], okmax)
        assert np.array_equal(util.widen_t(kmin[l, 0])[:, :nb], okmin)
    assert np.array_equal(wl.to_numpy(w.k_pool), kp0) and np.array_equal(wl.to_numpy(w.v_pool), vp0)
    assert np.array_equal(wl.to_numpy(partial.k_pool), ppk0) and np.array_equal(wl.to_numpy(partial.v_pool), ppv0)
    # incremental summaries == full recompute
    kmax2, kmin2 = torch.zeros_like(kmax), torch.zeros_like(kmin)
    B.specpv_update_block_summaries(cfg, 0, L, full, None, w.max_blocks, kmax2, kmin2, ws)
    nb = (sl0 + len(path) + bs - 1) // bs
    assert torch.equal(kmax[:, :, :, :nb], kmax2[:, :, :, :nb]) and torch.equal(kmin[:, :, :, :nb], kmin2[:, :, :, :nb])


@pytest.mark.parametrize("dtype,Hkv,d,bs,shift", [("bf16", 1, 64, 16, 0), ("bf16", 8, 128, 64, 0), ("bf16", 9, 128, 32, 1),
                                                  ("fp32", 3, 64, 64, 0), ("fp32", 12, 128, 16, 1)])
def test_summaries_of_ragged_blocks_are_exact(dtype, Hkv, d, bs, shift):
    """Eq. 1 with one token up to a whole block valid, head counts around the eight a CTA takes, NaN and signed zeros among
    the keys, summaries that start off a 16-byte boundary (``shift`` elements): bit-exact, max and min are."""
    dt, dev, L = wl.torch_dtype(dtype), "cuda", 2
    lens = [1, bs - 1, bs * 3, bs * 5 + 1]
    g = torch.Generator().manual_seed(Hkv + d)
    mb = 6
    k = torch.randn((L, mb * len(lens), Hkv, bs, d), generator=g)
    k[torch.rand(k.shape, generator=g) < 0.01] = float("nan")
    k[torch.rand(k.shape, generator=g) < 0.05] = -0.0
    k = k.to(dt).to(dev)
    table = torch.randperm(mb * len(lens), generator=g).to(torch.int32).view(len(lens), mb).to(dev)
    cache = B.Cache(k, k, table, torch.tensor(lens, dtype=torch.int32, device=dev), mb * bs)
    cfg = B.make_config(L, Hkv, Hkv, d, bs, dtype, 1, 1, 3, bs)
    n = L * len(lens) * Hkv * mb * d
    flat = [torch.full((n + 8,), 5.0, dtype=dt, device=dev)[shift:shift + n] for _ in range(2)]
    kmax, kmin = (f.view(L, len(lens), Hkv, mb, d) for f in flat)
    ws = torch.zeros(4096, dtype=torch.uint8, device=dev)
    B.specpv_update_block_summaries(cfg, 0, L, cache, None, mb, kmax, kmin, ws)
    util.sync_status(ws)
    for b, n_tok in enumerate(lens):
        nb = (n_tok + bs - 1) // bs
        keys = k[:, table[b, :nb].long()].permute(0, 2, 1, 3, 4).float().reshape(L, Hkv, nb * bs, d)[:, :, :n_tok]
        for i in range(nb):
            blk = keys[:, :, i * bs:(i + 1) * bs]
            hi = torch.where(blk.isnan(), torch.full_like(blk, -float("inf")), blk).amax(2)
            lo = torch.where(blk.isnan(), torch.full_like(blk, float("inf")), blk).amin(2)
            assert torch.equal(kmax[:, b, :, i].float(), hi) and torch.equal(kmin[:, b, :, i].float(), lo)
        assert torch.all(kmax[:, b, :, nb:].float() == 5.0) and torch.all(kmin[:, b, :, nb:].float() == 5.0)


@pytest.mark.parametrize("dtype,d,bs,n", [("bf16", 128, 64, 46), ("bf16", 64, 16, 46), ("fp32", 128, 32, 1), ("fp32", 64, 64, 0),
                                          ("bf16", 128, 16, 16)])
def test_commit_across_blocks_and_ragged_batches(dtype, d, bs, n):
    """A commit of up to 46 rows (a refresh's chain and path) that starts inside a block, at its end and at its first token,
    over several sequences: rows, summaries of every touched block and lengths against the oracle, twice in a row."""
    w = wl.make_workload("llama_32k", device="cuda", n_layers=2, spare_tokens=256, Hq=6, Hkv=3, d=d, bs=bs, dtype=dtype, M=48,
                         ctx=[bs * 5 + 3, bs * 4, bs * 6 - 1], shuffle=True)
    c = w.cfg
    L, Hkv, M, batch = c["n_layers"], c["Hkv"], c["M"], w.batch
    cfg = util.config_for(w)
    full = util.full_cache(w)
    full.max_seq_len = int(max(c["ctx"])) + 256
    ws = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    kmax = torch.zeros((L, batch, Hkv, w.max_blocks, d), dtype=wl.torch_dtype(dtype), device="cuda")
    kmin = torch.zeros_like(kmax)
    B.specpv_update_block_summaries(cfg, 0, L, full, None, w.max_blocks, kmax, kmin, ws)
    kp, vp = wl.to_numpy(w.k_pool).copy(), wl.to_numpy(w.v_pool).copy()
    lens = [int(x) for x in c["ctx"]]
    table = w.block_table.cpu().numpy()
    knn, vnn = wl.to_numpy(w.k_new), wl.to_numpy(w.v_new)
    rng = np.random.default_rng(n + bs)
    for _ in range(2):
        acc = rng.integers(0, M, size=(batch, 46)).astype(np.int32)
        counts = [n, max(n - 3, 0), n]
        B.specpv_commit_accepted(cfg, 0, L, w.k_new, w.v_new, M, torch.from_numpy(acc).cuda(),
                                 torch.tensor(counts, dtype=torch.int32, device="cuda"), 46, full, kmax, kmin, ws)
        util.sync_status(ws)
        for b in range(batch):
            for l in range(L):
                new_len = oracle.commit(knn[l, b], vnn[l, b], acc[b, :counts[b]], kp[l], vp[l], table[b], lens[b])
                okmax, okmin = oracle.block_summaries(kp[l], table[b], new_len)
                nb = (new_len + bs - 1) // bs
                assert np.array_equal(util.widen_t(kmax[l, b])[:, :nb], okmax) and np.array_equal(util.widen_t(kmin[l, b])[:, :nb], okmin)
            lens[b] += counts[b]
            assert int(w.seq_lens[b]) == lens[b]
        assert np.array_equal(wl.to_numpy(w.k_pool), kp) and np.array_equal(wl.to_numpy(w.v_pool), vp)


def test_commit_in_layer_groups_matches_the_oracle():
    """A step's commit issued in two layer groups, in ascending order: every group writes its rows at the lengths as
    they stand and the lengths advance with the group that holds the model's last layer."""
    w = wl.make_workload("llama_32k", device="cuda", n_layers=3, spare_tokens=64, ctx=[64 * 20 + 9], M=20)
    c = w.cfg
    L, M = c["n_layers"], c["M"]
    cfg = util.config_for(w)
    full = util.full_cache(w)
    ws = B.new_workspace(cfg, L, 1, int(max(c["ctx"])) + 64, M)
    path = wl.path_to(w.parents[0], int(np.argmax([len(wl.path_to(w.parents[0], n)) for n in range(M)])))
    acc = torch.zeros((1, 8), dtype=torch.int32, device="cuda")
    acc[0, :len(path)] = torch.from_numpy(path).cuda()
    n_acc = torch.tensor([len(path)], dtype=torch.int32, device="cuda")
    kp0, vp0 = wl.to_numpy(w.k_pool).copy(), wl.to_numpy(w.v_pool).copy()
    sl0 = int(w.seq_lens[0])
    B.specpv_commit_accepted(cfg, 0, 2, w.k_new[0:2], w.v_new[0:2], M, acc, n_acc, 8, full, None, None, ws)
    torch.cuda.synchronize()
    assert int(w.seq_lens[0]) == sl0                      # not yet: the last layer is not in this group
    B.specpv_commit_accepted(cfg, 2, 1, w.k_new[2:3], w.v_new[2:3], M, acc, n_acc, 8, full, None, None, ws)
    util.sync_status(ws)
    assert int(w.seq_lens[0]) == sl0 + len(path)
    table = w.block_table.cpu().numpy()
    knn, vnn = wl.to_numpy(w.k_new), wl.to_numpy(w.v_new)
    for l in range(L):
        assert oracle.commit(knn[l, 0], vnn[l, 0], path, kp0[l], vp0[l], table[0], sl0) == sl0 + len(path)
    assert np.array_equal(wl.to_numpy(w.k_pool), kp0) and np.array_equal(wl.to_numpy(w.v_pool), vp0)


def test_commits_of_two_caches_on_two_streams_share_a_workspace():
    """A commit keeps nothing in the workspace but the status word: commits of the full cache on one stream and of the partial
    cache on another, unordered, over one workspace, advance either cache's lengths by what was accepted, every time, and
    leave the workspace as it was."""
    dev, L, Hkv, d, bs, M, steps = "cuda", 36, 8, 128, 64, 8, 25
    cfg = B.make_config(L, 32, Hkv, d, bs, "bf16", 1, 2, 8, bs)
    k_new, v_new = (torch.randn((L, 1, M, Hkv, d), device=dev).to(torch.bfloat16) for _ in range(2))
    caches = []
    for n_pages in (12, 6):
        pool = torch.zeros((2, L, n_pages, Hkv, bs, d), dtype=torch.bfloat16, device=dev)
        caches.append(B.Cache(pool[0], pool[1], torch.arange(n_pages, dtype=torch.int32, device=dev)[None],
                              torch.tensor([3], dtype=torch.int32, device=dev), n_pages * bs))
    acc = torch.tensor([[4, 0, 6, 1]], dtype=torch.int32, device=dev)
    counts = [torch.tensor([n], dtype=torch.int32, device=dev) for n in (4, 2)]
    ws = torch.zeros(B.WORKSPACE_HEAD_BYTES, dtype=torch.uint8, device=dev)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(steps):
        for s, cache, n in zip(streams, caches, counts):
            B.specpv_commit_accepted(cfg, 0, L, k_new, v_new, M, acc, n, 4, cache, None, None, ws, stream=s)
    torch.cuda.synchronize()
    assert not ws.any()
    for cache, n in zip(caches, (4, 2)):
        assert int(cache.seq_lens[0]) == 3 + steps * n
        for pool, new in ((cache.k_pool, k_new), (cache.v_pool, v_new)):
            flat = pool.permute(0, 1, 3, 2, 4).reshape(L, -1, Hkv, d)
            assert torch.equal(flat[:, 3:3 + steps * n], new[:, 0][:, acc[0, :n].long()].repeat(1, steps, 1, 1))


@pytest.mark.parametrize("nb,budget", [(300, 40), (2048, 64), (4099, 128), (9000, 1000)])
def test_selection_alone_on_synthetic_scores_with_ties_and_nan(nb, budget):
    """The selection kernel on its own: several of its forms, repeated scores (ties go to the lower index), NaN (ranks last),
    -0 / +0; bit-exact against the oracle."""
    dev = "cuda"
    rng = np.random.default_rng(nb)
    Hkv, L, batch, bs = 3, 2, 2, 64
    sc = rng.standard_normal((L, batch, Hkv, nb)).astype(np.float32)
    sc[:, :, 0] = np.round(sc[:, :, 0] * 4) / 4          # many exact ties
    sc[0, 0, 1, rng.integers(0, nb, size=nb // 7)] = np.nan
    sc[1, 1, 2, ::5] = -0.0
    sc[1, 1, 2, 1::5] = 0.0
    lens = np.array([nb * bs - 3, (nb - 5) * bs], dtype=np.int32)  # ragged last block; a shorter second sequence
    cfg = B.make_config(L, 8 * Hkv, Hkv, 128, bs, "bf16", 1, 2, budget, 64)
    scores = torch.from_numpy(sc).to(dev)
    idx = torch.full((L, batch, Hkv, budget), -7, dtype=torch.int32, device=dev)
    count = torch.zeros(batch, dtype=torch.int32, device=dev)
    ws = torch.zeros(4096, dtype=torch.uint8, device=dev)
    B.specpv_select_partial_kv(cfg, L, scores, torch.from_numpy(lens).to(dev), batch, nb, idx, count, ws)
    util.sync_status(ws)
    got = idx.cpu().numpy()
    for b in range(batch):
        n = (int(lens[b]) + bs - 1) // bs
        assert int(count[b]) == min(n, budget)
        for l in range(L):
            for h in range(Hkv):
                want = oracle.select(sc[l, b, h, :n].astype(np.float64), 1, 2, budget)
                assert np.array_equal(got[l, b, h, :len(want)], want), (l, b, h)


@pytest.mark.parametrize("name,L,over", [("tiny_fp32", 1, {}), ("llama_32k", 5, dict(ctx=[5000])),
                                         ("llama_32k", 11, dict(ctx=[1500])), ("stress_b4", 3, dict(ctx=[900, 2100, 64, 1300]))])
def test_verify_host_matches_the_device_call_and_the_oracle(name, L, over):
    """The end-to-end entry point (pinned host step tensors in, host outputs back; layers pipelined in up to four groups, the copies in
    being what these calls take) against the device-pointer call and, on one layer, the oracle."""
    w = wl.make_workload(name, device="cuda", n_layers=L, spare_tokens=256, **over)  # the bytes of run_pipeline's caches
    c = w.cfg
    Hq, d, M, batch = c["Hq"], c["d"], c["M"], w.batch
    cfg = util.config_for(w)
    full = util.full_cache(w)
    ws = B.new_workspace(cfg, L, batch, int(max(c["ctx"])) + 256, M)
    mask = util.device_masks(w.parents, M)
    out_d = torch.zeros((L, batch, M, Hq, d), dtype=torch.float32, device="cuda")
    lse_d = torch.zeros((L, batch, M, Hq), dtype=torch.float32, device="cuda")
    B.specpv_verify_full(cfg, 0, L, w.q, w.k_new, w.v_new, mask, None, M, full, out_d, lse_d, ws)
    host = [t.cpu().pin_memory() for t in (w.q, w.k_new, w.v_new)]
    mask_h = mask.cpu().pin_memory()
    out_h = torch.full((L, batch, M, Hq, d), float("nan"), dtype=torch.float32).pin_memory()
    lse_h = torch.full((L, batch, M, Hq), float("nan"), dtype=torch.float32).pin_memory()
    for _ in range(2):  # twice: the staging area and the copy streams are reused
        B.specpv_verify_host(cfg, B.MODE_FULL, 0, L, host[0], host[1], host[2], mask_h, M, full, out_h, lse_h, ws)
    util.sync_status(ws)
    # the layer groups may be split over the KV range differently from the one-launch call: two results that are each
    # within the bar of the oracle, not bit-equal to each other
    tol = 2e-5 if c["dtype"] == "fp32" else 4e-2
    assert torch.isfinite(out_h).all() and torch.isfinite(lse_h).all()
    assert (out_h - out_d.cpu()).abs().max().item() <= tol
    assert (lse_h - lse_d.cpu()).abs().max().item() <= tol
    l, b = L - 1, batch - 1
    o_out, o_lse = oracle.tree_attention(wl.to_numpy(w.q[l, b]), wl.to_numpy(w.k_new[l, b]), wl.to_numpy(w.v_new[l, b]),
                                         oracle.tree_mask(w.parents[b]), wl.to_numpy(w.k_pool[l]),
                                         wl.to_numpy(w.v_pool[l]), wl.to_numpy(w.block_table[b]), int(c["ctx"][b]))
    util.compare(out_h[l, b].numpy(), o_out, c["dtype"], "verify_host")
    np.testing.assert_allclose(lse_h[l, b].numpy(), o_lse, atol=5e-3)


@pytest.mark.parametrize("dtype,Hq,d", [("fp32", 8, 64), ("fp32", 8, 128), ("bf16", 10, 128), ("bf16", 8, 64),
                                        ("bf16", 66, 64)])
@pytest.mark.parametrize("reduce,score_mode", [(B.REDUCE_MEAN, 0), (B.REDUCE_MAX, 1), (B.REDUCE_LAST, 0)])
def test_scores_of_the_plain_kernel(dtype, Hq, d, reduce, score_mode):
    """What the tensor-core score kernel does not take: float32, more than 1024 rows per KV head (33 x 33), and head size 64 or a
    group size that does not divide 128 with per-sequence row counts; a few blocks more or less than the 8 a CTA of the plain
    kernel takes (fewer than 296 CTAs), row counts that leave lanes without rows."""
    w = wl.make_workload("llama_32k", device="cuda", n_layers=2, Hq=Hq, Hkv=2, d=d, dtype=dtype, M=33,
                         ctx=[64 * 31 + 9, 64 * 33, 64])
    c = w.cfg
    Hkv, M, batch, L = c["Hkv"], c["M"], w.batch, c["n_layers"]
    cfg = util.config_for(w, reduce=reduce, score_mode=score_mode)
    full = util.full_cache(w)
    ws = B.new_workspace(cfg, L, batch, int(max(c["ctx"])), M)
    kmax = torch.zeros((L, batch, Hkv, w.max_blocks, d), dtype=wl.torch_dtype(dtype), device="cuda")
    kmin = torch.zeros_like(kmax)
    B.specpv_update_block_summaries(cfg, 0, L, full, None, w.max_blocks, kmax, kmin, ws)
    q_lens = torch.tensor([33, 2, 7], dtype=torch.int32, device="cuda")
    last = torch.tensor([30, 1, 0], dtype=torch.int32, device="cuda")
    scores = torch.full((L, batch, Hkv, w.max_blocks), float("nan"), dtype=torch.float32, device="cuda")
    B.specpv_score_blocks(cfg, 0, L, w.q, q_lens, M, last, kmax, kmin, full, scores, ws)
    util.sync_status(ws)
    for l in range(L):
        for b in range(batch):
            sl, m = int(c["ctx"][b]), int(q_lens[b])
            nb = (sl + c["bs"] - 1) // c["bs"]
            okmax, okmin = oracle.block_summaries(wl.to_numpy(w.k_pool[l]), wl.to_numpy(w.block_table[b]), sl)
            osc = oracle.block_scores(wl.to_numpy(w.q[l, b, :m]), okmax, okmin, Hkv, reduce=reduce, last_query=int(last[b]),
                                      score_mode=score_mode)
            # products of the stored values summed in float32: d terms per dot product, then up to 165 rows
            np.testing.assert_allclose(scores[l, b, :, :nb].cpu().numpy(), osc, rtol=2e-5, atol=2e-4, err_msg=f"{l} {b}")
            assert torch.isnan(scores[l, b, :, nb:]).all()


@pytest.mark.parametrize("Hq,d,M", [(2, 64, 1), (6, 128, 85), (6, 64, 86), (10, 128, 51), (10, 64, 52), (14, 128, 37),
                                    (8, 64, 64), (96, 128, 6), (256, 64, 5)])
@pytest.mark.parametrize("reduce,score_mode", [(B.REDUCE_MEAN, 0), (B.REDUCE_MAX, 0), (B.REDUCE_LAST, 1), (B.REDUCE_MEAN, 1)])
def test_scores_of_any_group_size_on_the_tensor_core_kernel(Hq, d, M, reduce, score_mode):
    """One to 128 query heads per KV head, both head sizes, ragged row counts: rows just below, at and just above the 256 of a
    pass and the 128 of an epilogue half, contractions a little wider than their rows; blocks around the 128 of a tile.  (With
    per-sequence row counts these shapes run on the plain kernel; test_mean_scores_on_the_tensor_core_kernel has such
    shapes without.)"""
    w = wl.make_workload("llama_32k", device="cuda", n_layers=2, Hq=Hq, Hkv=2, d=d, M=M, ctx=[64 * 128, 64 * 129 - 3, 64 * 5])
    c = w.cfg
    Hkv, batch, L = c["Hkv"], w.batch, c["n_layers"]
    cfg = util.config_for(w, reduce=reduce, score_mode=score_mode)
    full = util.full_cache(w)
    ws = B.new_workspace(cfg, L, batch, int(max(c["ctx"])), M)
    kmax = torch.zeros((L, batch, Hkv, w.max_blocks, d), dtype=torch.bfloat16, device="cuda")
    kmin = torch.zeros_like(kmax)
    B.specpv_update_block_summaries(cfg, 0, L, full, None, w.max_blocks, kmax, kmin, ws)
    q_lens = torch.tensor([M, max(M - 3, 1), (M + 1) // 2], dtype=torch.int32, device="cuda")
    last = torch.tensor([M - 1, 0, 0], dtype=torch.int32, device="cuda")
    scores = torch.full((L, batch, Hkv, w.max_blocks), float("nan"), dtype=torch.float32, device="cuda")
    B.specpv_score_blocks(cfg, 0, L, w.q, q_lens, M, last, kmax, kmin, full, scores, ws)
    util.sync_status(ws)
    for l in range(L):
        for b in range(batch):
            sl, m = int(c["ctx"][b]), int(q_lens[b])
            nb = (sl + c["bs"] - 1) // c["bs"]
            okmax, okmin = oracle.block_summaries(wl.to_numpy(w.k_pool[l]), wl.to_numpy(w.block_table[b]), sl)
            osc = oracle.block_scores(wl.to_numpy(w.q[l, b, :m]), okmax, okmin, Hkv, reduce=reduce, last_query=int(last[b]),
                                      score_mode=score_mode)
            # exact products summed in float32, d (twice d in the channel-wise form) to a dot product: as the plain kernel
            np.testing.assert_allclose(scores[l, b, :, :nb].cpu().numpy(), osc, rtol=2e-5, atol=2e-4, err_msg=f"{l} {b}")
            assert torch.isnan(scores[l, b, :, nb:]).all()  # blocks past the context are left alone


def score_call(Hq, Hkv, d, M, kmax, kmin, q, lens, bs=64, q_lens=None, reduce=0, score_mode=0):
    """Scores of one layer for given summaries [batch][Hkv][blocks][d] and queries; -7 where nothing was written."""
    batch, blocks = kmax.shape[0], kmax.shape[2]
    cfg = B.make_config(1, Hq, Hkv, d, bs, "bf16", 1, 2, 4, bs, reduce=reduce, score_mode=score_mode)
    pool = torch.zeros((1, 1, Hkv, bs, d), dtype=torch.bfloat16, device="cuda")
    cache = B.Cache(pool, pool, torch.zeros((batch, blocks), dtype=torch.int32, device="cuda"),
                    torch.tensor(lens, dtype=torch.int32, device="cuda"), max(lens))
    ws = torch.zeros(B.WORKSPACE_HEAD_BYTES, dtype=torch.uint8, device="cuda")
    scores = torch.full((1, batch, Hkv, blocks), -7.0, device="cuda")
    rows = None if q_lens is None else torch.tensor(q_lens, dtype=torch.int32, device="cuda")
    B.specpv_score_blocks(cfg, 0, 1, q, rows, M, None, kmax, kmin, cache, scores, ws)
    util.sync_status(ws)
    return scores[0]


def score_reference(kmax, kmin, q, Hkv, reduce, score_mode):
    """[Hkv][blocks] float64 scores of one sequence: kmax, kmin [Hkv][blocks][d], q [rows][Hq][d]."""
    d = q.shape[-1]
    rows = q.double().reshape(q.shape[0], Hkv, -1, d)
    if reduce == B.REDUCE_LAST:
        rows = rows[:1]
    rows = rows.permute(1, 0, 2, 3).reshape(Hkv, -1, d)
    a, z = kmax.double().transpose(1, 2), kmin.double().transpose(1, 2)
    s = torch.maximum(rows @ a, rows @ z) if score_mode == 0 else rows.clamp(min=0) @ a + rows.clamp(max=0) @ z
    return s.amax(1) if reduce == B.REDUCE_MAX else s.mean(1)


@pytest.mark.parametrize("Hq,Hkv,d,M", [(8, 2, 64, 8), (8, 2, 64, 64), (10, 2, 128, 51), (10, 2, 128, 52), (14, 2, 128, 37),
                                        (256, 2, 64, 5), (2, 2, 64, 32), (7, 1, 128, 90), (96, 2, 128, 6)])
def test_mean_scores_on_the_tensor_core_kernel(Hq, Hkv, d, M):
    """Head size 64 and group sizes that do not divide 128 without per-sequence row counts: 32 rows and just above, just below
    and above the 256 of a pass, three passes; blocks around the 128 of a tile."""
    lens = [64 * 128, 64 * 129 - 3, 64 * 5]
    g = torch.Generator().manual_seed(Hq + M)
    key = torch.randn((2, 3, Hkv, 129, d), generator=g)
    kmax, kmin = (t.to(torch.bfloat16).cuda() for t in (key.amax(0), key.amin(0)))
    q = torch.randn((1, 3, M, Hq, d), generator=g).to(torch.bfloat16).cuda()
    got = score_call(Hq, Hkv, d, M, kmax, kmin, q, lens)
    for b, n in enumerate(lens):
        nb = (n + 63) // 64
        want = score_reference(kmax[b, :, :nb], kmin[b, :, :nb], q[0, b], Hkv, 0, 0)
        torch.testing.assert_close(got[b, :, :nb].double(), want, rtol=2e-5, atol=2e-4)
        assert (got[b, :, nb:] == -7.0).all()


@pytest.mark.parametrize("Hq,Hkv,d", [(8, 2, 64), (10, 2, 128), (3, 1, 128)])
@pytest.mark.parametrize("M,reduce,score_mode", [(60, B.REDUCE_MAX, 0), (60, B.REDUCE_LAST, 0), (60, B.REDUCE_MEAN, 1),
                                                 (1, B.REDUCE_MEAN, 0), (40, B.REDUCE_MEAN, 0)])
def test_scores_are_rounded_not_truncated(Hq, Hkv, d, M, reduce, score_mode):
    """Head size 64 and group sizes that do not divide 128: float32 products, rounded sums.  Rounding errors have either sign, at
    2^-24 sqrt(d) = 6.7e-7 a score at most over 4000 scores they leave 1e-8 between the scores' mean size and the exact one; truncated
    sums are 4.6e-8 (d = 64) to 14e-8 (d = 128) too small.  The mean of the full dot products over 32 rows or more stays on the tensor
    cores, whose error there is below that of the plain kernel's long sums: 1.6e-7 bounds both."""
    blocks = 2048
    g = torch.Generator().manual_seed(d + M + reduce)
    u = torch.randn((Hkv, 1, d), generator=g)
    u = 6.0 * u / u.norm(dim=-1, keepdim=True)
    key = torch.randn((2, 1, Hkv, blocks, d), generator=g) + u * torch.rand((Hkv, blocks, 1), generator=g)
    kmax, kmin = (t.to(torch.bfloat16).cuda() for t in (key.amax(0), key.amin(0)))
    q = (torch.randn((1, 1, M, Hq, d), generator=g) + u[:, 0].repeat_interleave(Hq // Hkv, 0)).to(torch.bfloat16).cuda()
    got = score_call(Hq, Hkv, d, M, kmax, kmin, q, [blocks * 64], reduce=reduce, score_mode=score_mode)[0].double()
    want = score_reference(kmax[0], kmin[0], q[0, 0], Hkv, reduce, score_mode)
    drift = (((got - want) * want).sum() / (want * want).sum()).abs().item()
    assert drift < (1.6e-7 if reduce == B.REDUCE_MEAN and score_mode == 0 and M > 1 else 2.5e-8)


@pytest.mark.parametrize("Hq,Hkv,d", [(8, 2, 64), (10, 2, 128)])
def test_scores_without_rows_and_with_infinite_keys(Hq, Hkv, d):
    """Head size 64 and group sizes that do not divide 128: a sequence with no rows in this step has a mean of NaN, a maximum of
    -infinity and row 0 as its last row; a channel whose maximum is infinite counts, channel-wise, for the queries that are positive
    there and for no others."""
    g = torch.Generator().manual_seed(d)
    key = torch.randn((2, 2, Hkv, 40, d), generator=g)
    kmax, kmin = (t.to(torch.bfloat16).cuda() for t in (key.amax(0), key.amin(0)))
    q = torch.randn((1, 2, 6, Hq, d), generator=g).to(torch.bfloat16).cuda()
    lens = [64 * 40, 64 * 39 + 1]
    for reduce in (B.REDUCE_MEAN, B.REDUCE_MAX, B.REDUCE_LAST):
        got = score_call(Hq, Hkv, d, 6, kmax, kmin, q, lens, q_lens=[0, 6], reduce=reduce)
        if reduce == B.REDUCE_MEAN:
            assert got[0].isnan().all()
        elif reduce == B.REDUCE_MAX:
            assert (got[0] == -float("inf")).all()
        else:
            torch.testing.assert_close(got[0].double(), score_reference(kmax[0], kmin[0], q[0, 0], Hkv, reduce, 0), rtol=2e-5, atol=2e-4)
        torch.testing.assert_close(got[1].double(), score_reference(kmax[1], kmin[1], q[0, 1], Hkv, reduce, 0), rtol=2e-5, atol=2e-4)
    q[..., 3] = -q[..., 3].abs() - 0.1
    plain = score_call(Hq, Hkv, d, 6, kmax, kmin, q, lens, score_mode=1)
    kmax[:, :, 5, 3] = float("inf")
    assert torch.equal(score_call(Hq, Hkv, d, 6, kmax, kmin, q, lens, score_mode=1), plain)
    q[:, :, 0, :, 3] = 1.0
    got = score_call(Hq, Hkv, d, 6, kmax, kmin, q, lens, score_mode=1)
    assert (got[:, :, 5] == float("inf")).all() and got[:, :, :5].isfinite().all()


@pytest.mark.parametrize("score_mode", [0, 1])
@pytest.mark.parametrize("reduce", [B.REDUCE_MEAN, B.REDUCE_MAX, B.REDUCE_LAST])
def test_scores_of_a_refresh_step_with_more_rows_than_one_accumulator(reduce, score_mode):
    """A refresh scores with the chain and the tree together: 90 and 77 tokens x 4 heads = 360 and 308 query rows per
    KV head, which the tensor-core kernel takes in two passes of 64 tokens (the second sequence's second pass is
    ragged); the "last" row sits in the second pass for one sequence and in the first for the other."""
    w = wl.make_workload("llama_32k", device="cuda", n_layers=2, M=90, ctx=[64 * 140 + 9, 64 * 300 + 1])
    c = w.cfg
    Hkv, d, M, batch, L = c["Hkv"], c["d"], c["M"], w.batch, c["n_layers"]
    cfg = util.config_for(w, reduce=reduce, score_mode=score_mode)
    full = util.full_cache(w)
    ws = B.new_workspace(cfg, L, batch, int(max(c["ctx"])), M)
    kmax = torch.zeros((L, batch, Hkv, w.max_blocks, d), dtype=torch.bfloat16, device="cuda")
    kmin = torch.zeros_like(kmax)
    B.specpv_update_block_summaries(cfg, 0, L, full, None, w.max_blocks, kmax, kmin, ws)
    q_lens = torch.tensor([90, 77], dtype=torch.int32, device="cuda")
    last = torch.tensor([71, 5], dtype=torch.int32, device="cuda")
    scores = torch.full((L, batch, Hkv, w.max_blocks), float("nan"), dtype=torch.float32, device="cuda")
    B.specpv_score_blocks(cfg, 0, L, w.q, q_lens, M, last, kmax, kmin, full, scores, ws)
    util.sync_status(ws)
    for l in range(L):
        for b in range(batch):
            sl = int(c["ctx"][b])
            nb = (sl + c["bs"] - 1) // c["bs"]
            okmax, okmin = oracle.block_summaries(wl.to_numpy(w.k_pool[l]), wl.to_numpy(w.block_table[b]), sl)
            m = int(q_lens[b])
            osc = oracle.block_scores(wl.to_numpy(w.q[l, b, :m]), okmax, okmin, Hkv, reduce=reduce, last_query=int(last[b]),
                                      score_mode=score_mode)
            got = scores[l, b, :, :nb].cpu().numpy().astype(np.float64)
            assert np.isfinite(got).all()
            np.testing.assert_allclose(got, osc, rtol=2e-3, atol=2e-2, err_msg=f"layer {l} seq {b}")
            assert torch.isnan(scores[l, b, :, nb:]).all()  # blocks past the context are left alone


@pytest.mark.parametrize("nb,budget", [(7, 5), (259, 100), (1024, 5), (1025, 64), (4096, 4095), (4097, 64), (16387, 128), (16500, 64)])
def test_selection_at_the_edges_of_its_register_forms(nb, budget):
    """Candidate counts either side of 1024, 4096 and 16384, around which the forms of the selection kernel change, few candidates to
    choose, and all but one."""
    test_selection_alone_on_synthetic_scores_with_ties_and_nan(nb, budget)


@pytest.mark.parametrize("blocks,layers", [(1, 1), (8, 1), (9, 1), (31, 75), (33, 75)])
@pytest.mark.parametrize("M,d", [(16, 64), (17, 128), (33, 64)])
def test_plain_scores_in_both_forms(blocks, layers, M, d):
    """One block per warp and, with CTAs enough (75 layers x 2 heads x 2 groups of 32 blocks), four; 64, 68 and 132 rows around
    the 64 that are staged at a time."""
    w = wl.make_workload("tiny_fp32", device="cuda", n_layers=layers, Hq=8, Hkv=2, d=d, M=M, ctx=[64 * blocks - 5])
    cfg, full = util.config_for(w, reduce=B.REDUCE_MEAN), util.full_cache(w)
    ws = B.new_workspace(cfg, layers, 1, 64 * blocks, M)
    kmax = torch.zeros((layers, 1, 2, w.max_blocks, d), dtype=torch.float32, device="cuda")
    kmin = torch.zeros_like(kmax)
    B.specpv_update_block_summaries(cfg, 0, layers, full, None, w.max_blocks, kmax, kmin, ws)
    scores = torch.full((layers, 1, 2, w.max_blocks), float("nan"), dtype=torch.float32, device="cuda")
    B.specpv_score_blocks(cfg, 0, layers, w.q, None, M, torch.zeros(1, dtype=torch.int32, device="cuda"), kmax, kmin, full, scores, ws)
    util.sync_status(ws)
    for l in {0, layers - 1}:
        want = oracle.block_scores(wl.to_numpy(w.q[l, 0]), wl.to_numpy(kmax[l, 0])[:, :blocks],
                                   wl.to_numpy(kmin[l, 0])[:, :blocks], 2, reduce=B.REDUCE_MEAN)
        # products of the stored values summed in float32: d terms per dot product, then up to 132 rows
        np.testing.assert_allclose(scores[l, 0, :, :blocks].cpu().numpy(), want, rtol=2e-5, atol=2e-4)
        assert torch.isnan(scores[l, 0, :, blocks:]).all()


@pytest.mark.parametrize("dtype,Hkv,batch,bs,A", [("fp32", 1, 1, 64, 4), ("fp32", 2, 2, 64, 4), ("bf16", 1, 4, 16, 16), ("bf16", 4, 1, 32, 5),
                                                  ("fp32", 3, 1, 16, 17)])
def test_commit_of_few_units_in_one_launch(dtype, Hkv, batch, bs, A):
    """Up to four units of work (block touched, KV head, sequence) share a CTA, up to eight are a cluster, either of which advances the
    lengths itself; nine, the last case, take two launches.  Three commits in a row, of which the second appends nothing to the first sequence."""
    d, M = 64, 24
    w = wl.make_workload("tiny_fp32", device="cuda", n_layers=1, spare_tokens=256, Hq=2 * Hkv, Hkv=Hkv, d=d, bs=bs, dtype=dtype, M=M,
                         ctx=[bs * 3 + 5 * b - 1 for b in range(batch)])
    cfg, full = B.make_config(1, 2 * Hkv, Hkv, d, bs, dtype, 1, 1, 3, bs), util.full_cache(w)
    full.max_seq_len = int(max(w.cfg["ctx"])) + 256
    ws = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    kmax = torch.zeros((1, batch, Hkv, w.max_blocks, d), dtype=wl.torch_dtype(dtype), device="cuda")
    kmin = torch.zeros_like(kmax)
    B.specpv_update_block_summaries(cfg, 0, 1, full, None, w.max_blocks, kmax, kmin, ws)
    kp, vp = wl.to_numpy(w.k_pool).copy(), wl.to_numpy(w.v_pool).copy()
    lens, table = [int(x) for x in w.cfg["ctx"]], w.block_table.cpu().numpy()
    knn, vnn = wl.to_numpy(w.k_new), wl.to_numpy(w.v_new)
    rng = np.random.default_rng(bs + A)
    for turn in range(3):
        acc = rng.integers(0, M, size=(batch, A)).astype(np.int32)
        counts = [0 if turn == 1 and b == 0 else A - b % 2 for b in range(batch)]
        before = B.specpv_kernel_launches()
        B.specpv_commit_accepted(cfg, 0, 1, w.k_new, w.v_new, M, torch.from_numpy(acc).cuda(),
                                 torch.tensor(counts, dtype=torch.int32, device="cuda"), A, full, kmax, kmin, ws)
        assert B.specpv_kernel_launches() - before == (2 if Hkv == 3 else 1)
        util.sync_status(ws)
        for b in range(batch):
            new_len = oracle.commit(knn[0, b], vnn[0, b], acc[b, :counts[b]], kp[0], vp[0], table[b], lens[b])
            okmax, okmin = oracle.block_summaries(kp[0], table[b], new_len)
            nb = (new_len + bs - 1) // bs
            assert np.array_equal(util.widen_t(kmax[0, b])[:, :nb], okmax) and np.array_equal(util.widen_t(kmin[0, b])[:, :nb], okmin)
            lens[b] += counts[b]
            assert int(w.seq_lens[b]) == lens[b]
        assert np.array_equal(wl.to_numpy(w.k_pool), kp) and np.array_equal(wl.to_numpy(w.v_pool), vp)


@pytest.mark.parametrize("n,L", [(33, 1), (1024, 2), (1025, 1), (2048, 2), (2049, 2), (2049, 20), (4096, 20), (4097, 2), (4097, 20), (8192, 20),
                                 (8193, 1), (16384, 1), (16385, 1)])
@pytest.mark.parametrize("shared", [0, 1])
def test_selection_of_one_and_of_tied_candidates(n, L, shared):
    """Either side of every form's most candidates, on fewer lists than SMs and on more (20 layers x 8 heads), with k = 1 and 61 of them to
    choose: the search from the keys' common bits, past its second look, and the one key that is left.  Scores are multiples of 1/4, so that
    the mean over the 8 heads is exact and many tie; layer 0 has one value everywhere, layer 1 NaN throughout its first list but
    for one score, and one that is larger than the rest by far."""
    dev, Hkv, bs = "cuda", 8, 16
    rng = np.random.default_rng(n + L)
    nb = n + 3  # 1 sink and 2 local blocks beside the candidates
    sc = np.round(rng.standard_normal((L, 1, Hkv, nb)) * 16).astype(np.float32) / 4
    sc[0] = -1.25
    if L > 1:
        sc[1, 0, 0] = np.nan
        sc[1, 0, :, n // 2 + 1] = 1e30
    scores = torch.from_numpy(sc).to(dev)
    lens = torch.tensor([nb * bs], dtype=torch.int32, device=dev)
    ws = torch.zeros(4096, dtype=torch.uint8, device=dev)
    for budget in (4, 64) if n > 61 else (4,):
        cfg = B.make_config(L, 4 * Hkv, Hkv, 128, bs, "bf16", 1, 2, budget, 64, select_shared=shared)
        idx = torch.full((L, 1, Hkv, budget), -7, dtype=torch.int32, device=dev)
        count = torch.zeros(1, dtype=torch.int32, device=dev)
        B.specpv_select_partial_kv(cfg, L, scores, lens, 1, nb, idx, count, ws)
        util.sync_status(ws)
        got = idx.cpu().numpy()
        for l in {0, min(1, L - 1), L - 1}:
            mean = sc[l, 0].astype(np.float64).sum(0) / Hkv
            for h in range(Hkv):
                want = oracle.select(mean if shared else sc[l, 0, h].astype(np.float64), 1, 2, budget)
                assert np.array_equal(got[l, 0, h], want), (budget, l, h)


@pytest.mark.parametrize("dtype,batch,A", [("fp32", 1, 1), ("bf16", 1, 17), ("bf16", 2, 16), ("fp32", 1, 49), ("bf16", 3, 16), ("bf16", 1, 81), ("fp32", 1, 112),
                                           ("bf16", 4, 7)])
def test_commit_of_any_number_of_units(dtype, batch, A):
    """Two to eight units, with up to as many tokens as the touched blocks hold."""
    test_commit_of_few_units_in_one_launch(dtype, 1, batch, 16, A)


@pytest.mark.parametrize("dtype,Hq,d,M", [("fp32", 2, 64, 16), ("fp32", 8, 128, 4), ("fp32", 8, 128, 5), ("bf16", 8, 64, 17), ("bf16", 10, 128, 3),
                                          ("bf16", 10, 128, 13), ("bf16", 2, 64, 1)])
@pytest.mark.parametrize("reduce,score_mode", [(B.REDUCE_MEAN, 0), (B.REDUCE_MAX, 1), (B.REDUCE_LAST, 0), (B.REDUCE_LAST, 1)])
@pytest.mark.parametrize("layers,shift", [(1, 0), (75, 0), (75, 1)])
def test_plain_scores_with_few_rows_and_summaries_anywhere(dtype, Hq, d, M, reduce, score_mode, layers, shift):
    """Up to 16 rows of a group, of which eight lanes share one, and just more; one block per warp and (75 layers) four; per-sequence row
    counts, whose last sequence has none; summaries that start on a 16-byte boundary and one element past it."""
    Hkv, lens, blocks = 2, [64 * 33 - 5, 64 * 8, 64 * 9 - 63], 33
    dt = wl.torch_dtype(dtype)
    g = torch.Generator().manual_seed(Hq + M + layers)
    key = torch.randn((2, layers, 3, Hkv, blocks, d), generator=g)
    n = key[0].numel()
    flat = [torch.zeros(n + 8, dtype=dt, device="cuda")[shift:shift + n] for _ in range(2)]
    kmax, kmin = (f.view(layers, 3, Hkv, blocks, d).copy_(t.to(dt)) for f, t in zip(flat, (key.amax(0), key.amin(0))))
    q = torch.randn((layers, 3, M, Hq, d), generator=g).to(dt).cuda()
    cfg = B.make_config(layers, Hq, Hkv, d, 64, dtype, 1, 2, 4, 64, reduce=reduce, score_mode=score_mode)
    pool = torch.zeros((layers, 1, Hkv, 64, d), dtype=dt, device="cuda")
    cache = B.Cache(pool, pool, torch.zeros((3, blocks), dtype=torch.int32, device="cuda"), torch.tensor(lens, dtype=torch.int32, device="cuda"), max(lens))
    ws = torch.zeros(B.WORKSPACE_HEAD_BYTES, dtype=torch.uint8, device="cuda")
    scores = torch.full((layers, 3, Hkv, blocks), -7.0, device="cuda")
    rows = [M, (M + 1) // 2, 0]
    B.specpv_score_blocks(cfg, 0, layers, q, torch.tensor(rows, dtype=torch.int32, device="cuda"), M, torch.zeros(3, dtype=torch.int32, device="cuda"),
                          kmax, kmin, cache, scores, ws)
    util.sync_status(ws)
    for l in {0, layers // 2, layers - 1}:
        for b in range(3):
            nb = (lens[b] + 63) // 64
            got = scores[l, b]
            assert (got[:, nb:] == -7.0).all()  # blocks past the context are left alone
            if rows[b] == 0 and reduce != B.REDUCE_LAST:
                assert got[:, :nb].isnan().all() if reduce == B.REDUCE_MEAN else (got[:, :nb] == -float("inf")).all()
                continue
            want = score_reference(kmax[l, b, :, :nb], kmin[l, b, :, :nb], q[l, b, :max(rows[b], 1)], Hkv, reduce, score_mode)
            # products of the stored values summed in float32: d terms per dot product, then up to 85 rows
            torch.testing.assert_close(got[:, :nb].double(), want, rtol=2e-5, atol=2e-4)


@pytest.mark.parametrize("mode", [B.MODE_FULL, B.MODE_PARTIAL])
@pytest.mark.parametrize("Hq,Hkv,M,ctx,L,out_f32", [
    (32, 8, 2, [3000], 7, 0),      # attention outlasts the copies: groups of 1, 1, 4, 1 layers with their own keys and values
    (32, 8, 60, [9000], 5, 1),     # attention at 0.6 of the copies in: groups of 2, 2, 1
    (32, 8, 60, [1500], 7, 0),     # keys and values first: queries in groups of 1, 3, 2, 1
    (32, 8, 24, [900, 400], 3, 1),  # the same with outputs longer than the queries, a short delay
    (8, 8, 100, [300], 8, 1),      # and a delay too long for that
])
def test_verify_host_in_every_order_of_its_copies(mode, Hq, Hkv, M, ctx, L, out_f32):
    """Every layer of the host call against the device-pointer call, every sequence of the last layer against the oracle."""
    w = wl.make_workload("llama_32k", device="cuda", n_layers=L, spare_tokens=256, Hq=Hq, Hkv=Hkv, M=M, ctx=ctx)
    c, batch, d = w.cfg, w.batch, w.cfg["d"]
    cfg = util.config_for(w, out_f32=out_f32, budget_blocks=4, buffer_tokens=64)
    cache = util.full_cache(w)
    ws = B.new_workspace(cfg, L, batch, int(max(ctx)) + 256, M)
    mask = util.device_masks(w.parents, M)
    dt = torch.float32 if out_f32 else torch.bfloat16
    out_d = torch.zeros((L, batch, M, Hq, d), dtype=dt, device="cuda")
    lse_d = torch.zeros((L, batch, M, Hq), dtype=torch.float32, device="cuda")
    verify = B.specpv_verify_full if mode == B.MODE_FULL else B.specpv_verify_partial
    verify(cfg, 0, L, w.q, w.k_new, w.v_new, mask, None, M, cache, out_d, lse_d, ws)
    host = [t.cpu().pin_memory() for t in (w.q, w.k_new, w.v_new)]
    mask_h = mask.cpu().pin_memory()
    out_h = torch.full((L, batch, M, Hq, d), float("nan"), dtype=dt).pin_memory()
    lse_h = torch.full((L, batch, M, Hq), float("nan"), dtype=torch.float32).pin_memory()
    for _ in range(2):  # twice: the staging area and the copy streams are reused
        out_h.fill_(float("nan"))
        B.specpv_verify_host(cfg, mode, 0, L, host[0], host[1], host[2], mask_h, M, cache, out_h, lse_h, ws)
    util.sync_status(ws)
    # as above: the groups may split the KV range differently from the one launch.  A bfloat16 output adds half a unit in the last place
    # of values up to 16 on either side, 2 x 2^-5
    assert torch.isfinite(out_h).all() and torch.isfinite(lse_h).all()
    assert (out_h.float() - out_d.cpu().float()).abs().max().item() <= (4e-2 if out_f32 else 4e-2 + 2 ** -4)
    assert (lse_h - lse_d.cpu()).abs().max().item() <= 4e-2
    l = L - 1
    for b in range(batch):
        o_out, o_lse = oracle.tree_attention(wl.to_numpy(w.q[l, b]), wl.to_numpy(w.k_new[l, b]), wl.to_numpy(w.v_new[l, b]),
                                             oracle.tree_mask(w.parents[b]), wl.to_numpy(w.k_pool[l]),
                                             wl.to_numpy(w.v_pool[l]), wl.to_numpy(w.block_table[b]), int(ctx[b]))
        if out_f32:
            util.compare(out_h[l, b].numpy(), o_out, "bf16", "verify_host")
        else:
            assert np.abs(out_h[l, b].float().numpy() - o_out).max() <= 2e-2 + 2 ** -5
        np.testing.assert_allclose(lse_h[l, b].numpy(), o_lse, atol=5e-3)
