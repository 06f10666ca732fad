"""GPU parity of the verification attention over a sweep of small shapes and edge cases
(ragged last block, empty context, one-node trees, M not a multiple of 8, refresh chains,
per-sequence row counts, every group size and block size), element by element against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_02337_b200 import binding as B
from paper_2512_02337_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, params=["single", "pair"])
def attention_kernel(request, monkeypatch):
    """Every case runs on both tensor-core kernels: the default (one CTA per KV range) and the CTA-pair kernel,
    which the library uses on request for shapes with more than 128 query rows per KV head."""
    if request.param == "pair":
        monkeypatch.setenv("SPECPV_ATTN_KERNEL", "pair")
    else:
        monkeypatch.delenv("SPECPV_ATTN_KERNEL", raising=False)
    return request.param


def run_case(dtype, Hq, Hkv, d, bs, ctx, Ms, depth=4, branch=3, n_chain=0, n_layers=1, shuffle=True, seed=0,
             partial_entry=False, float32_weights=False):
    """One verify call on random data; Ms lists the tree size of every sequence (ragged q_lens).  ``float32_weights``: hold the
    results to what float32 weights give (see test_weights_keep_their_float32_precision)."""
    rng = np.random.default_rng(seed)
    dev = "cuda"
    batch = len(ctx)
    dt = wl.torch_dtype(dtype)
    M_max = max(Ms) + n_chain
    blocks = [(c + bs - 1) // bs + 1 for c in ctx]
    n_pages = sum(blocks) + 2
    max_blocks = max(blocks)
    pages = rng.permutation(n_pages) if shuffle else np.arange(n_pages)
    table = np.zeros((batch, max_blocks), dtype=np.int32)
    off = 0
    for b in range(batch):
        table[b, :blocks[b]] = pages[off:off + blocks[b]]
        off += blocks[b]
    g = torch.Generator(device="cpu").manual_seed(seed)
    k_pool = torch.randn((n_layers, n_pages, Hkv, bs, d), generator=g).to(dt).to(dev)
    v_pool = torch.randn((n_layers, n_pages, Hkv, bs, d), generator=g).to(dt).to(dev)
    q = (torch.randn((n_layers, batch, M_max, Hq, d), generator=g) * 1.5).to(dt).to(dev)
    k_new = torch.randn((n_layers, batch, M_max, Hkv, d), generator=g).to(dt).to(dev)
    v_new = torch.randn((n_layers, batch, M_max, Hkv, d), generator=g).to(dt).to(dev)
    parents = [wl.make_tree(m, min(depth, m - 1), branch, rng) for m in Ms]
    W = (M_max + 63) // 64
    masks = np.zeros((batch, M_max, W), dtype=np.uint64)
    for b in range(batch):
        m = B.specpv_build_tree_mask(parents[b], n_chain, W)
        masks[b, :m.shape[0]] = m
    q_lens = torch.tensor([m + n_chain for m in Ms], dtype=torch.int32, device=dev)
    seq_lens = torch.tensor(ctx, dtype=torch.int32, device=dev)
    cfg = B.make_config(n_layers, Hq, Hkv, d, bs, dtype, 1, 1, 3, bs, out_f32=1)
    cache = B.Cache(k_pool, v_pool, torch.from_numpy(table).to(dev), seq_lens, max(ctx))
    ws = B.new_workspace(cfg, n_layers, batch, max(max(ctx), 1), M_max)
    out = torch.full((n_layers, batch, M_max, Hq, d), 77.0, dtype=torch.float32, device=dev)
    lse = torch.full((n_layers, batch, M_max, Hq), 77.0, dtype=torch.float32, device=dev)
    fn = B.specpv_verify_partial if partial_entry else B.specpv_verify_full
    mask_dev = torch.from_numpy(masks.view(np.int64)).to(dev)
    fn(cfg, 0, n_layers, q, k_new, v_new, mask_dev, q_lens, M_max, cache, out, lse, ws)
    if dtype == "bf16":  # the bfloat16 output is the float32 one, rounded
        cfg16 = B.make_config(n_layers, Hq, Hkv, d, bs, dtype, 1, 1, 3, bs, out_f32=0)
        out16 = torch.full((n_layers, batch, M_max, Hq, d), 77.0, dtype=dt, device=dev)
        fn(cfg16, 0, n_layers, q, k_new, v_new, mask_dev, q_lens, M_max, cache, out16, None, ws)
        util.same_as_rounded(out16, out)
    util.sync_status(ws)
    kp, vp = wl.to_numpy(k_pool), wl.to_numpy(v_pool)
    qn, knn, vnn = wl.to_numpy(q), wl.to_numpy(k_new), wl.to_numpy(v_new)
    for l in range(n_layers):
        for b in range(batch):
            m = Ms[b] + n_chain
            omask = oracle.tree_mask(parents[b], n_chain)
            assert np.array_equal(omask, masks[b, :m, :omask.shape[1]])
            o_out, o_lse = oracle.tree_attention(qn[l, b, :m], knn[l, b, :m], vnn[l, b, :m], omask, kp[l], vp[l],
                                                 table[b], ctx[b])
            util.compare(util.widen_t(out[l, b, :m]), o_out, dtype, f"out l{l} b{b}")
            np.testing.assert_allclose(lse[l, b, :m].cpu().numpy(), o_lse, atol=2e-5 if dtype == "fp32" else 5e-3)
            if float32_weights:
                err = out[l, b, :m].double().cpu().numpy() - o_out
                assert np.sqrt((err ** 2).mean() / (o_out ** 2).mean()) < 1.2e-5
                np.testing.assert_allclose(lse[l, b, :m].cpu().numpy(), o_lse, rtol=3e-7, atol=2e-6)
            # rows past q_lens[b] are not written
            assert torch.all(out[l, b, m:].float() == 77.0)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("Hq,Hkv,d,bs", [(8, 2, 64, 64), (32, 8, 128, 64), (4, 4, 128, 16), (16, 2, 64, 32),
                                          (8, 4, 128, 64)])
def test_shapes_ragged_context(dtype, Hq, Hkv, d, bs):
    run_case(dtype, Hq, Hkv, d, bs, ctx=[bs * 9 + 5, bs * 4], Ms=[13, 7], seed=Hq + d + bs)


@pytest.mark.parametrize("bs", [16, 32])
def test_small_pages_on_the_tensor_core_path(bs):
    """16- and 32-token pages (the paper's block size is 16): eight or four pages per 128-token tile, shuffled
    table, a context long enough to be split over many CTAs with a ragged last page, two layers, refresh rows."""
    run_case("bf16", 32, 8, 128, bs, ctx=[bs * 531 + bs - 3, bs * 7 + 1, 0], Ms=[60, 9, 2], depth=6, branch=4,
             n_layers=2, seed=40 + bs)
    run_case("bf16", 8, 2, 128, bs, ctx=[128 * 20 + 5], Ms=[48], depth=5, branch=4, n_chain=20, seed=41 + bs)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_empty_context_and_single_node_tree(dtype):
    run_case(dtype, 8, 2, 128, 64, ctx=[0, 1, 64], Ms=[5, 1, 1], seed=3)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_refresh_rows_chain_plus_tree(dtype):
    # partially verified chain of 42 tokens in front of a 48-node tree: 90 rows, two mask words
    run_case(dtype, 32, 8, 128, 64, ctx=[64 * 40 + 17], Ms=[48], depth=5, branch=4, n_chain=42, seed=4)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_maximum_rows_and_long_split_context(dtype):
    # M_max = 128 (the kernels' limit) and a context long enough to be split across many CTAs
    run_case(dtype, 8, 2, 128, 64, ctx=[64 * 300 + 63], Ms=[128], depth=8, branch=4, seed=5)


@pytest.mark.parametrize("Hq,Hkv,d", [(10, 2, 128), (12, 2, 64), (7, 1, 128), (8, 2, 64), (24, 2, 128)])
@pytest.mark.parametrize("bs,ctx,Ms,n_chain", [
    (64, [0, 127, 128, 129], [1, 25, 24, 9], 0),      # one row tile; none, one, one and two context tiles
    (16, [128 * 2, 128 * 3 + 1], [26, 10], 0),         # an even and an odd number of tiles between the two streams
    (32, [128 * 5 - 1], [33], 20),                     # two and three row tiles
])
def test_packed_rows_and_alternating_streams(Hq, Hkv, d, bs, ctx, Ms, n_chain):
    """Group sizes that do not divide 128 (rows of a tile left over), head size 64, and sequences of one row tile,
    whose two streams take alternate K/V tiles: 0 to 5 context tiles, ragged last tiles, row counts at the tile edge."""
    run_case("bf16", Hq, Hkv, d, bs, ctx=ctx, Ms=Ms, n_chain=n_chain, seed=Hq + d + len(ctx))


@pytest.mark.parametrize("Hq,Hkv,d", [(8, 2, 64), (1, 1, 64), (10, 2, 128), (7, 1, 128), (130, 1, 64)])
@pytest.mark.parametrize("bs,ctx,Ms,n_layers", [
    (64, [0, 129], [9, 7], 1),             # no context; a tile and one token
    (16, [128 * 11 + 5], [26], 24),        # one and two row tiles, few KV splits
    (32, [128 * 9, 100], [64, 33], 1),     # one CTA per few tiles, merged
])
def test_weights_keep_their_float32_precision(Hq, Hkv, d, bs, ctx, Ms, n_layers):
    """bfloat16 caches with head size 64 or a group size that does not divide 128 (and, on the plain kernel, more than 128
    query heads per KV head): weights in float32, or in two bfloat16 terms that hold them to 2^-16, 2.6e-6 rms.  The tensor core
    cuts a sum to 2^-24 of itself after every 16 tokens and term, 16 times a tile: for 12 tiles 192 x 6e-8 = 1.1e-5 at most.  (One
    bfloat16 term is off by 2^-9 / sqrt(3) = 1.1e-3 a weight.)  A log-sum-exp is rounded once, 2^-24 = 6e-8 of itself, and holds the
    error of the scores, d / 16 cuts of 2^-24 = 4.8e-7 of a score at most, 2.4e-7 on average, before the mean is put back."""
    run_case("bf16", Hq, Hkv, d, bs, ctx=ctx, Ms=Ms, n_layers=n_layers, seed=Hq + d + len(ctx), float32_weights=True)


@pytest.mark.parametrize("Hq,Hkv,d", [(8, 2, 64), (5, 1, 128)])
@pytest.mark.parametrize("bs,ctx,Ms,n_chain", [
    (64, [0, 1, 63, 64], [16, 1, 13, 12], 0),         # no context to one 64-token tile, row counts around 64
    (16, [65, 64 * 9], [65, 17], 0),                   # the step's own tokens in two tiles
    (32, [64 * 40 + 33], [60], 68),                    # 128 step tokens, several row tiles, many splits
])
def test_float32_kernel_tile_edges(Hq, Hkv, d, bs, ctx, Ms, n_chain):
    """The plain kernel's 64-row and 64-token tiles at their edges, one and many KV splits."""
    run_case("fp32", Hq, Hkv, d, bs, ctx=ctx, Ms=Ms, n_chain=n_chain, seed=Hq + bs)


@pytest.mark.parametrize("dtype,Hq,Hkv,d", [("bf16", 8, 2, 64), ("bf16", 10, 2, 128), ("bf16", 8, 2, 128), ("fp32", 8, 2, 64)])
@pytest.mark.parametrize("scale", [0.31, 1.0, 2.0 ** -23 + 2.0 ** -46, 1e-40])
def test_softmax_scale(dtype, Hq, Hkv, d, scale):
    """A softmax scale of the caller's, down to one that makes all visible keys count alike: masked keys still count nothing."""
    dev, bs, M, ctx = "cuda", 64, 21, 333
    dt = wl.torch_dtype(dtype)
    g = torch.Generator().manual_seed(d + Hq)
    mk = lambda *shape: (0.5 * torch.randn(shape, generator=g)).to(dt).to(dev)  # noqa: E731
    pools, q = mk(2, 1, 6, Hkv, bs, d), mk(1, 1, M, Hq, d)
    k_new, v_new = mk(2, 1, 1, M, Hkv, d)
    table = torch.arange(6, dtype=torch.int32, device=dev)[None]
    cache = B.Cache(pools[0], pools[1], table, torch.tensor([ctx], dtype=torch.int32, device=dev), ctx)
    parents = wl.make_tree(M, 5, 4, np.random.default_rng(1))
    cfg = B.make_config(1, Hq, Hkv, d, bs, dtype, 1, 1, 3, bs, softmax_scale=scale, out_f32=1)
    ws = B.new_workspace(cfg, 1, 1, ctx, M)
    out, lse = torch.zeros((1, 1, M, Hq, d), device=dev), torch.zeros((1, 1, M, Hq), device=dev)
    B.specpv_verify_full(cfg, 0, 1, q, k_new, v_new, util.device_masks([parents], M), None, M, cache, out, lse, ws)
    util.sync_status(ws)
    o_out, o_lse = oracle.tree_attention(wl.to_numpy(q[0, 0]), wl.to_numpy(k_new[0, 0]), wl.to_numpy(v_new[0, 0]),
                                         oracle.tree_mask(parents), wl.to_numpy(pools[0, 0]), wl.to_numpy(pools[1, 0]),
                                         table[0].cpu().numpy(), ctx, float(np.float32(scale)))
    util.compare(out[0, 0].cpu().numpy(), o_out, dtype, f"scale {scale}")
    np.testing.assert_allclose(lse[0, 0].cpu().numpy(), o_lse, atol=2e-5 if dtype == "fp32" else 5e-3)


@pytest.mark.parametrize("Hq,Hkv,d", [(8, 2, 64), (10, 2, 128), (8, 2, 128)])
def test_infinite_values_stay_infinite(Hq, Hkv, d):
    """A channel in which a visible token's value is infinite is infinite in the output (the weight is positive, however it is held),
    NaN where infinities of both signs meet, and the other channels know nothing of it."""
    dev, bs, M, ctx = "cuda", 64, 30, 900
    g = torch.Generator().manual_seed(d + Hq)
    bf = lambda *shape: torch.randn(shape, generator=g).to(torch.bfloat16).to(dev)  # noqa: E731
    pools, q = bf(2, 1, 15, Hkv, bs, d), bf(1, 1, M, Hq, d)
    k_new, v_new = bf(2, 1, 1, M, Hkv, d)
    cache = B.Cache(pools[0], pools[1], torch.arange(15, dtype=torch.int32, device=dev)[None],
                    torch.tensor([ctx], dtype=torch.int32, device=dev), ctx)
    mask = util.device_masks([wl.make_tree(M, 5, 4, np.random.default_rng(1))], M)
    cfg = B.make_config(1, Hq, Hkv, d, bs, "bf16", 1, 1, 3, bs, out_f32=1)
    ws = B.new_workspace(cfg, 1, 1, ctx, M)
    out = torch.zeros_like(q, dtype=torch.float32)
    call = lambda: B.specpv_verify_full(cfg, 0, 1, q, k_new, v_new, mask, None, M, cache, out, None, ws)  # noqa: E731
    call()
    plain, inf = out.clone(), float("inf")
    for t in range(0, 128, 3):  # whatever bits the weights have
        cache.v_pool[0, t // bs, :, t % bs, 1] = inf
    cache.v_pool[0, 5, :, 7, 2] = -inf
    cache.v_pool[0, 5, :, 8, 3], cache.v_pool[0, 6, :, 8, 3] = inf, -inf
    v_new[0, 0, 0, :, 4] = inf  # the root, which every row sees
    call()
    util.sync_status(ws)
    assert (out[..., 1] == inf).all() and (out[..., 2] == -inf).all() and out[..., 3].isnan().all() and (out[..., 4] == inf).all()
    assert torch.equal(out[..., 5:], plain[..., 5:]) and torch.equal(out[..., 0], plain[..., 0])


@pytest.mark.parametrize("Hq,Hkv,d,ctx,n_layers", [(8, 2, 64, 3000, 1), (10, 2, 128, 3000, 1), (32, 8, 128, 700, 1),
                                                   (32, 8, 128, 6000, 4)])
def test_workspace_off_a_32_byte_boundary(Hq, Hkv, d, ctx, n_layers):
    """A workspace needs 16-byte alignment and no more: 16 bytes past a multiple of 32, as large as the call asks for and not a
    byte larger, gives what an aligned one gives, and nothing before or behind it is written."""
    dev, bs, M = "cuda", 64, 20
    g = torch.Generator().manual_seed(ctx + d)
    bf = lambda *shape: torch.randn(shape, generator=g).to(torch.bfloat16).to(dev)  # noqa: E731
    n_pages = (ctx + bs - 1) // bs
    pools, q = bf(2, n_layers, n_pages, Hkv, bs, d), bf(n_layers, 1, M, Hq, d)
    k_new, v_new = bf(2, n_layers, 1, M, Hkv, d)
    cache = B.Cache(pools[0], pools[1], torch.arange(n_pages, dtype=torch.int32, device=dev)[None],
                    torch.tensor([ctx], dtype=torch.int32, device=dev), ctx)
    mask = util.device_masks([wl.make_tree(M, 5, 4, np.random.default_rng(1))], M)
    cfg = B.make_config(n_layers, Hq, Hkv, d, bs, "bf16", 1, 1, 3, bs, out_f32=1)
    n = B.specpv_workspace_bytes(cfg, n_layers, 1, ctx, M)
    results = []
    for offset in (0, 16):
        buf = torch.full((n + 4096,), 0x5A, dtype=torch.uint8, device=dev)
        ws = buf[1024 + offset:1024 + offset + n]
        assert ws.data_ptr() % 32 == offset
        ws.zero_()
        out, lse = torch.zeros_like(q, dtype=torch.float32), torch.zeros((n_layers, 1, M, Hq), device=dev)
        B.specpv_verify_full(cfg, 0, n_layers, q, k_new, v_new, mask, None, M, cache, out, lse, ws)
        util.sync_status(ws)
        assert (buf[:1024 + offset] == 0x5A).all() and (buf[1024 + offset + n:] == 0x5A).all()
        results.append((out, lse))
    assert torch.equal(results[0][0], results[1][0]) and torch.equal(results[0][1], results[1][1])


@pytest.mark.parametrize("d,value", [(64, 0.1), (128, 0.7)])
def test_float32_kernel_sums_over_long_ranges(d, value):
    """Equal weights and equal values over 4096 tokens that one CTA walks (enough heads that the KV range is not split): the output
    is that value.  Sums of 64 tokens added up are off by some 64 x 2^-25 = 1.9e-6 at most, 9e-7 when simulated; one chain
    of 4096 additions drifts by 4e-5 for these values."""
    dev = "cuda"
    Hkv, bs, n, batch = 8, 64, 4096, 74
    cfg = B.make_config(1, Hkv, Hkv, d, bs, "fp32", 1, 1, 3, bs)
    k_pool = torch.randn((1, n // bs, Hkv, bs, d), generator=torch.Generator().manual_seed(d)).to(dev)
    v_pool = torch.full_like(k_pool, value)
    table = torch.arange(n // bs, dtype=torch.int32, device=dev).repeat(batch, 1)
    cache = B.Cache(k_pool, v_pool, table, torch.full((batch,), n, dtype=torch.int32, device=dev), n)
    q = torch.zeros((1, batch, 1, Hkv, d), device=dev)  # equal weights
    kv_new = torch.full((1, batch, 1, Hkv, d), value, device=dev)
    mask = torch.ones((batch, 1, 1), dtype=torch.int64, device=dev)
    ws = B.new_workspace(cfg, 1, batch, n, 1)
    out = torch.zeros_like(q)
    B.specpv_verify_full(cfg, 0, 1, q, kv_new, kv_new, mask, None, 1, cache, out, None, ws)
    util.sync_status(ws)
    want = kv_new[0, 0, 0, 0, 0].double()
    assert ((out.double() - want).abs().max() / want).item() < 2e-6


@pytest.mark.parametrize("M,n_layers", [(60, 20), (90, 12), (26, 24)])
def test_many_layers_and_one_layer_agree_with_the_oracle(M, n_layers):
    """The row tiles per CTA and the KV splits depend on how many CTAs a launch has: two row tiles without splits, a last
    row group of one tile behind the full ones, and one row tile with splits, on the same ragged context."""
    run_case("bf16", 32, 8, 128, 64, ctx=[128 * 6 + 70], Ms=[M], n_layers=n_layers, seed=M)
    run_case("bf16", 32, 8, 128, 64, ctx=[128 * 6 + 70], Ms=[M], n_layers=1, seed=M + 1)


@pytest.mark.parametrize("M,n_layers", [(8, 1), (9, 24), (40, 1), (41, 20)])
def test_warps_without_rows(M, n_layers):
    """Row counts at the 32 rows of a warp: warps without a row in the first and in the second row tile, a second row tile
    that only one sequence uses, one tile of the step's own tokens and several K/V tiles, one and many KV splits."""
    run_case("bf16", 32, 8, 128, 64, ctx=[128 * 5 + 70, 0, 128 * 3], Ms=[M, max(M - 33, 1), M // 2], n_layers=n_layers, seed=M)


def test_partial_entry_point_multi_layer_bf16():
    run_case("bf16", 32, 8, 128, 64, ctx=[64 * 64 + 20, 64 * 70], Ms=[60, 33], depth=6, branch=4, n_layers=3,
             seed=6, partial_entry=True)


def test_chain_tree_matches_torch_causal_sdpa():
    # independent witness on the GPU side as well: a chain tree is causal attention (library SDPA)
    dev = "cuda"
    Hq, Hkv, d, bs, L, M = 8, 2, 64, 64, 64 * 5 + 9, 12
    g = torch.Generator().manual_seed(1)
    n_pages = (L + bs - 1) // bs
    k_pool = torch.randn((1, n_pages, Hkv, bs, d), generator=g).to(dev)
    v_pool = torch.randn((1, n_pages, Hkv, bs, d), generator=g).to(dev)
    q = torch.randn((1, 1, M, Hq, d), generator=g).to(dev)
    k_new = torch.randn((1, 1, M, Hkv, d), generator=g).to(dev)
    v_new = torch.randn((1, 1, M, Hkv, d), generator=g).to(dev)
    mask = util.device_masks([np.arange(-1, M - 1, dtype=np.int32)], M)
    cfg = B.make_config(1, Hq, Hkv, d, bs, "fp32", 1, 1, 3, 64)
    cache = B.Cache(k_pool, v_pool, torch.arange(n_pages, dtype=torch.int32, device=dev)[None],
                    torch.tensor([L], dtype=torch.int32, device=dev), L)
    ws = B.new_workspace(cfg, 1, 1, L, M)
    out = torch.zeros_like(q)
    B.specpv_verify_full(cfg, 0, 1, q, k_new, v_new, mask, None, M, cache, out, None, ws)
    util.sync_status(ws)
    k_all = torch.cat([k_pool[0].permute(0, 2, 1, 3).reshape(-1, Hkv, d)[:L], k_new[0, 0]]).double().cpu()
    v_all = torch.cat([v_pool[0].permute(0, 2, 1, 3).reshape(-1, Hkv, d)[:L], v_new[0, 0]]).double().cpu()
    q_full = torch.cat([torch.zeros((L, Hq, d), dtype=torch.float64), q[0, 0].double().cpu()])
    G = Hq // Hkv
    want = torch.nn.functional.scaled_dot_product_attention(
        q_full.permute(1, 0, 2)[None], k_all.permute(1, 0, 2).repeat_interleave(G, 0)[None],
        v_all.permute(1, 0, 2).repeat_interleave(G, 0)[None], is_causal=True)[0].permute(1, 0, 2)[L:]
    assert (out[0, 0].double().cpu() - want).abs().max() < 1e-5


@pytest.mark.parametrize("where", ["late", "early", "middle_twice"])
def test_large_score_jumps_take_the_general_path(where):
    """The tensor-core kernel keeps a row's reference maximum across full context tiles and only checks the row sum
    for overflow; keys whose scores exceed the reference by hundreds of nats (far beyond float32 range of the
    weights) must send it back over the tile, rescale, and still match the oracle."""
    dev = "cuda"
    Hq, Hkv, d, bs, M = 32, 8, 128, 64, 40
    L_ctx = 64 * 48 + 21
    g = torch.Generator().manual_seed(17)
    n_pages = (L_ctx + bs - 1) // bs + 1
    k_pool = torch.randn((1, n_pages, Hkv, bs, d), generator=g)
    v_pool = torch.randn((1, n_pages, Hkv, bs, d), generator=g)
    q = torch.randn((1, 1, M, Hq, d), generator=g)
    # blocks whose keys are the queries' mean direction, scaled: their logits jump by hundreds of nats
    direction = q[0, 0].mean(dim=(0, 1))
    direction = direction / direction.norm()
    q = q + 8.0 * direction
    boost = {"late": [(40, 400.0)], "early": [(0, 400.0)], "middle_twice": [(9, 150.0), (30, 500.0)]}[where]
    for page, scale in boost:
        k_pool[0, page, :, 5:9] = scale * direction
    to = lambda t: t.to(torch.bfloat16).to(dev)  # noqa: E731
    k_pool, v_pool, q = to(k_pool), to(v_pool), to(q)
    k_new = to(torch.randn((1, 1, M, Hkv, d), generator=g))
    v_new = to(torch.randn((1, 1, M, Hkv, d), generator=g))
    rng = np.random.default_rng(3)
    parents = [wl.make_tree(M, 5, 4, rng)]
    mask = util.device_masks(parents, M)
    cfg = B.make_config(1, Hq, Hkv, d, bs, "bf16", 1, 1, 3, bs, out_f32=1)
    table = torch.arange(n_pages, dtype=torch.int32, device=dev)[None].contiguous()
    cache = B.Cache(k_pool, v_pool, table, torch.tensor([L_ctx], dtype=torch.int32, device=dev), L_ctx)
    ws = B.new_workspace(cfg, 1, 1, L_ctx, M)
    out = torch.zeros((1, 1, M, Hq, d), dtype=torch.float32, device=dev)
    lse = torch.zeros((1, 1, M, Hq), dtype=torch.float32, device=dev)
    B.specpv_verify_full(cfg, 0, 1, q, k_new, v_new, mask, None, M, cache, out, lse, ws)
    util.sync_status(ws)
    o_out, o_lse = oracle.tree_attention(wl.to_numpy(q[0, 0]), wl.to_numpy(k_new[0, 0]), wl.to_numpy(v_new[0, 0]),
                                         oracle.tree_mask(parents[0]), wl.to_numpy(k_pool[0]), wl.to_numpy(v_pool[0]),
                                         table[0].cpu().numpy(), L_ctx)
    assert np.abs(o_lse).max() > 200  # the jump really is beyond what unscaled float32 weights could hold
    util.compare(out[0, 0].cpu().numpy(), o_out, "bf16", f"jump {where}")
    np.testing.assert_allclose(lse[0, 0].cpu().numpy(), o_lse, rtol=2e-5, atol=5e-3)


@pytest.mark.parametrize("Hq,Hkv,d", [(8, 8, 128), (40, 8, 128), (32, 8, 64)])
@pytest.mark.parametrize("tiles", [0, 1, 3, 4, 6])
def test_short_walks_of_one_cta(Hq, Hkv, d, tiles):
    """Enough heads that no KV range is split: a CTA walks `tiles` context tiles of 128 tokens (the last one ragged) and the step's
    own, one tile (nothing for the second stream), as many as the short walk of the two-term form takes, and more."""
    run_case("bf16", Hq, Hkv, d, 64, ctx=[max(128 * tiles - 27, 0)], Ms=[6], n_layers=19, seed=60 + tiles, float32_weights=d == 64 or Hq == 40)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("splits", [2, 15, 16, 17, 32, 33, 63, 64])
def test_float32_merge_around_its_groups_of_splits(d, splits):
    """One tile of 64 tokens per split (64 of them at most): counts around the 16 (32 with 128 channels) that a group of lanes merges."""
    run_case("fp32", 8, 2, d, 64, ctx=[64 * (splits - 1) - 7], Ms=[5], seed=90 + splits)
