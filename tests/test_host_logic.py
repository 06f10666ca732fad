"""CPU-only checks: the C-ABI library loads and exports every symbol the header declares, the host
functions (tree mask, mode rule) agree bit-for-bit with the oracle, and argument validation rejects
bad requests before anything is launched."""
import ctypes
import os
import re
from pathlib import Path

import numpy as np
import pytest
import torch

import oracle
from paper_2512_02337_b200 import binding as B
from paper_2512_02337_b200 import build as build_mod
from paper_2512_02337_b200 import workloads as wl

ROOT = Path(__file__).resolve().parent.parent


@pytest.fixture(scope="module", autouse=True)
def built():
    build_mod.build()


def test_library_exports_every_declared_symbol():
    header = (ROOT / "include" / "specpv.h").read_text()
    declared = set(re.findall(r"\b(specpv_[a-z_0-9]+)\s*\(", header))
    assert declared == set(B.EXPORTS)
    selftest = (ROOT / "include" / "specpv_selftest.h").read_text()
    declared_selftest = set(re.findall(r"\b(specpv_[a-z_0-9]+)\s*\(", selftest))
    assert declared_selftest == set(B.SELFTEST_EXPORTS)
    lib = B.lib()
    for name in declared | declared_selftest:
        assert getattr(lib, name) is not None


@pytest.mark.parametrize("M,depth,branch,chain", [(1, 0, 1, 0), (16, 4, 4, 0), (60, 6, 4, 0), (64, 6, 4, 0),
                                                  (48, 5, 4, 42), (100, 8, 3, 28), (128, 10, 2, 0), (5, 4, 1, 123)])
def test_tree_mask_bit_exact_with_oracle(M, depth, branch, chain):
    rng = np.random.default_rng(M + chain)
    for _ in range(5):
        parents = wl.make_tree(M, depth, branch, rng)
        assert np.array_equal(B.specpv_build_tree_mask(parents, chain), oracle.tree_mask(parents, chain))
    wide = B.specpv_build_tree_mask(parents, chain, row_words=4)
    assert np.array_equal(wide[:, : (M + chain + 63) // 64], oracle.tree_mask(parents, chain))
    assert not wide[:, (M + chain + 63) // 64:].any()


def test_tree_mask_rejects_bad_trees():
    for bad in ([0], [-1, 1], [-1, 0, 5], [-1, -1], [-1, 0, -2]):
        with pytest.raises(B.SpecPVError) as e:
            B.specpv_build_tree_mask(np.array(bad, dtype=np.int32))
        assert e.value.status == 5
    with pytest.raises(B.SpecPVError) as e:
        B.specpv_build_tree_mask(np.arange(-1, 69, dtype=np.int32), row_words=1)
    assert e.value.status == 4


def test_mode_rule_matches_oracle_on_a_grid():
    for ctx in (0, 100, 4095, 4096, 4097, 100000):
        for budget in (512, 4096):
            for npv in (0, 1, 20, 21, 60):
                for ncand in (1, 48, 60):
                    for buf in (20, 68, 80):
                        for init in (0, 1):
                            assert B.specpv_select_mode(ctx, budget, npv, ncand, buf, init) == \
                                oracle.select_mode(ctx, budget, npv, ncand, buf, init)


def test_config_validation_happens_on_the_host():
    good = dict(n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, block_tokens=64, dtype="fp32", sink_blocks=1,
                local_blocks=2, budget_blocks=8, buffer_tokens=64)
    assert B.specpv_workspace_bytes(B.make_config(**good), 2, 1, 2048, 16) > 256
    for key, val in [("n_q_heads", 7), ("head_dim", 96), ("block_tokens", 48), ("dtype", 5), ("budget_blocks", 3),
                     ("local_blocks", 0), ("reduce", 3), ("score_mode", 2), ("softmax_scale", -1.0)]:
        assert B.specpv_workspace_bytes(B.make_config(**{**good, key: val}), 2, 1, 2048, 16) == 0, key
    # null pointers / bad layer ranges are refused before any CUDA call (works without a GPU)
    cfg = B.make_config(**good)
    lib = B.lib()
    kv = B.PagedKV(0, 0, 0, 0, 1, 4, 4, 256)
    st = lib.specpv_verify_full(ctypes.byref(cfg), 0, 1, None, None, None, None, None, 16, ctypes.byref(kv), None,
                                None, None, ctypes.c_size_t(0), None)
    assert st == 1
    assert B.specpv_status_string(0) == "ok" and "capacity" in B.specpv_status_string(4)


def test_projection_and_offload_calls_validate_on_the_host():
    """Bad shapes and null pointers of the linear maps and of the offloaded verification are refused before any CUDA
    call (so this runs without a GPU); 16-byte aligned host buffers stand in for device pointers."""
    cfg = B.make_config(n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, block_tokens=64, dtype="fp32", sink_blocks=1,
                        local_blocks=2, budget_blocks=8, buffer_tokens=64)
    lib = B.lib()
    buf = np.zeros(4096, dtype=np.float32)
    ptr = ctypes.c_void_p(buf.ctypes.data + (-buf.ctypes.data) % 16)
    size = ctypes.c_size_t(1024)

    def qkv(hidden=512, layer0=0, n_layers=1, x=ptr, cos_sin=ptr, ws=ptr):
        return lib.specpv_qkv_rope(ctypes.byref(cfg), layer0, n_layers, x, hidden, ptr, cos_sin, 1, 16, ptr, ptr, ptr, ws,
                                   size, None)
    assert qkv(hidden=100) == 2          # hidden not a multiple of 16
    assert qkv(hidden=0) == 2
    assert qkv(x=None) == 1
    assert qkv(cos_sin=None) == 1
    assert qkv(ws=None) == 1
    assert qkv(layer0=2) == 1            # outside the two layers of the pool
    assert qkv(n_layers=3) == 1
    assert qkv(x=ctypes.c_void_p(ptr.value + 4)) == 1  # misaligned

    def o_proj(hidden=512, attn=ptr, y=ptr):
        return lib.specpv_o_proj(ctypes.byref(cfg), 0, 1, attn, ptr, hidden, None, 1, 16, y, ptr, size, None)
    assert o_proj(hidden=24) == 2
    assert o_proj(attn=None) == 1 and o_proj(y=None) == 1

    def table(theta=1.0e4, batch=1, M=16, mask=ptr):
        return lib.specpv_rope_table(ctypes.byref(cfg), mask, None, ptr, batch, M, ctypes.c_double(theta), ptr, None)
    assert table(theta=1.0) == 1 and table(theta=float("inf")) == 1 and table(theta=float("nan")) == 1
    assert table(batch=0) == 1 and table(mask=None) == 1
    assert table(M=129) == 4             # more rows than the mask words the kernels handle

    off = B.OffloadedKV(ptr, ptr, ptr, ptr, ptr, ptr, 1, 4, 4, 256)
    def staged(kv=off, q=ptr, layer0=0, n_layers=1, M=16):
        return lib.specpv_verify_full_offloaded(ctypes.byref(cfg), layer0, n_layers, q, ptr, ptr, ptr, None, M,
                                                ctypes.byref(kv) if kv is not None else None, ptr, None, ptr, size, None,
                                                None)
    assert staged(kv=None) == 1 and staged(q=None) == 1 and staged(n_layers=3) == 1
    assert staged(kv=B.OffloadedKV(None, ptr, ptr, ptr, ptr, ptr, 1, 4, 4, 256)) == 1
    assert staged(kv=B.OffloadedKV(ptr, ptr, ptr, ptr, ptr, ptr, 1, 4, 4, 257)) == 4   # longer than the table covers
    assert staged(M=129) == 4
    assert staged() == 4                 # a 1 KB workspace cannot hold the split partials


def test_workspace_grows_with_the_request():
    cfg = B.make_config(32, 32, 8, 128, 64, "bf16", 1, 2, 64, 80)
    a = B.specpv_workspace_bytes(cfg, 1, 1, 131072, 60)
    b = B.specpv_workspace_bytes(cfg, 32, 1, 131072, 60)
    c = B.specpv_workspace_bytes(cfg, 32, 4, 131072, 64)
    assert 256 < a < b < c


def _rank_main(rank, world, port, q):
    import torch.distributed as dist
    import torch

    import bench
    dist.init_process_group("gloo", init_method=f"tcp://127.0.0.1:{port}", rank=rank, world_size=world)
    try:
        # each replica reports its own device-timed figures; the job's figure is the slowest replica's
        got = bench.max_over_ranks([10.0 + rank, 5.0 - rank], torch.device("cpu"))
        q.put((rank, got))
    finally:
        dist.destroy_process_group()


def test_replica_timings_are_reduced_with_max_over_ranks_gloo():
    """bench.py --gpus N runs N independent replicas (the path has no exchange step); the only multi-rank
    logic is the MAX reduction of the timings, exercised here with two gloo ranks on the CPU."""
    import socket
    import torch.multiprocessing as mp
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    procs = [ctx.Process(target=_rank_main, args=(r, 2, port, q)) for r in range(2)]
    for p in procs:
        p.start()
    results = dict(q.get(timeout=120) for _ in range(2))
    for p in procs:
        p.join(timeout=60)
        assert p.exitcode == 0
    assert results[0] == results[1] == [11.0, 5.0]


@pytest.fixture(params=["native", "ctypes"])
def conversion(request, monkeypatch, tmp_path):
    """The step's calls with their arguments converted in native code and, where that has not been built, through ctypes."""
    monkeypatch.setattr(B, "_pycalls", None)
    if request.param == "ctypes":
        monkeypatch.setattr(B, "PYCALLS_PATH", tmp_path / "missing.so")
    assert isinstance(B._native(), B._CtypesCalls) == (request.param == "ctypes")
    return request.param


def verify_full_args(**over):
    """Arguments of a call that the library refuses for its null query tensor (so no CUDA call is made)."""
    cfg = B.make_config(n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, block_tokens=64, dtype="fp32", sink_blocks=1,
                        local_blocks=2, budget_blocks=8, buffer_tokens=64)
    t = torch.zeros(2, 4, 2, 64, 64)
    cache = B.Cache(t, t, torch.zeros(1, 4, dtype=torch.int32), torch.zeros(1, dtype=torch.int32), 256)
    return dict(dict(cfg=cfg, layer0=0, n_layers=1, q=None, k_new=np.zeros(64, np.float32), v_new=t, tree_mask=t, q_lens=None,
                     M_max=16, full=cache, out=t, lse=None, workspace=t, stream=0), **over)


@pytest.mark.parametrize("bad,error", [("strided", AssertionError), ("list", TypeError), ("word", TypeError),
                                       ("config", TypeError), ("cache", AttributeError), (None, B.SpecPVError)])
def test_native_argument_conversion(bad, error, conversion):
    """Tensors, NumPy arrays and None are taken as pointers, everything else is refused before the library is called; the
    library then refuses the null query tensor."""
    t = torch.zeros(2, 4, 2, 64, 64)
    args = verify_full_args(**{"strided": dict(v_new=t.transpose(0, 1)), "list": dict(v_new=[1.0]), "word": dict(M_max="16"),
                               "config": dict(cfg=t.numpy()), "cache": dict(full=t), None: {}}[bad])
    with pytest.raises((error, ctypes.ArgumentError) if bad == "word" else error) as e:
        B.specpv_verify_full(**args)
    assert bad is not None or e.value.status == 1


def test_conversion_takes_what_ctypes_takes_and_refuses_the_rest(conversion):
    """A configuration is a ctypes structure, its own or another that begins alike, and no other buffer of that size; sizes may be
    c_int; a cache is asked for its own desc() where it has one, a subclass of Cache as well as any other object."""
    args = verify_full_args()
    cfg = args["cfg"]
    for other in (bytes(cfg), bytearray(bytes(cfg)), np.frombuffer(bytes(cfg), dtype=np.uint8)):
        with pytest.raises(TypeError):
            B.specpv_verify_full(**dict(args, cfg=other))

    class Longer(ctypes.Structure):
        _fields_ = B.Config._fields_ + [("more", ctypes.c_int32)]
    longer = Longer.from_buffer_copy(bytes(cfg) + bytes(4))

    def too_long():  # 257 tokens in a table of 4 pages of 64: SPECPV_ERR_CAPACITY, where the cache itself gives INVALID_ARG
        kv = B.Cache.desc(args["full"])
        kv.max_seq_len = 257
        return kv

    class Subclass(B.Cache):
        def desc(self):
            return too_long()

    class Other:
        desc = staticmethod(too_long)

    class Wrong:
        def desc(self):
            return b"0" * ctypes.sizeof(B.PagedKV)
    sub = Subclass(**vars(args["full"]))
    for over, status in ((dict(cfg=longer), 1), (dict(M_max=ctypes.c_int(16), layer0=ctypes.c_int32(0)), 1), (dict(full=sub), 4),
                         (dict(full=Other()), 4)):
        with pytest.raises(B.SpecPVError) as e:
            B.specpv_verify_full(**dict(args, **over))
        assert e.value.status == status, over
    with pytest.raises(TypeError):
        B.specpv_verify_full(**dict(args, full=Wrong()))


def test_both_conversions_know_the_same_calls():
    """The table of pycalls.c and the binding's, and the library's functions of those names."""
    source = (ROOT / "paper_2512_02337_b200" / "csrc" / "pycalls.c").read_text()
    assert dict(re.findall(r'X\((specpv_\w+), "(\w+)", call_', source)) == B._STEP_CALLS
    assert set(B._SIGNATURES) == set(B.EXPORTS[3:] + B.SELFTEST_EXPORTS)


def test_build_does_without_a_c_compiler_and_builds_per_interpreter(monkeypatch, tmp_path):
    """Where the argument conversion cannot be compiled the library is built all the same, a stale one is removed, and the calls
    go through ctypes; its file name carries the interpreter's ABI, so that another interpreter does not load it."""
    import sysconfig
    assert build_mod.PYCALLS == B.PYCALLS_PATH and build_mod.PYCALLS.name == "pycalls" + sysconfig.get_config_var("EXT_SUFFIX")
    stale = tmp_path / build_mod.PYCALLS.name
    stale.touch()
    os.utime(stale, (0, 0))
    monkeypatch.setattr(build_mod, "PYCALLS", stale)
    for compiler in ("/nonexistent/cc", "false --some-flag"):
        monkeypatch.setenv("CC", compiler)
        with pytest.warns(UserWarning, match="through ctypes"):
            assert build_mod.build() == build_mod.LIB
        assert not stale.exists()
    monkeypatch.setenv("CC", "gcc -g0")  # a command with arguments
    build_mod.build()
    assert stale.exists() and not build_mod.needs_build(stale)


def test_overlapped_kernels_load_nothing_through_the_read_only_path():
    """A kernel launched as a programmatic dependent runs while its predecessor may still be writing what it will read, so no
    source that launches one holds a non-coherent load: __ldg, ld.global.nc, or const __restrict__ kernel parameters."""
    sources = {p.name: re.sub(r"//[^\n]*", "", p.read_text()) for p in sorted((ROOT / "paper_2512_02337_b200" / "csrc").glob("*.cu"))}
    overlapped = {n: s for n, s in sources.items() if re.search(r"\blaunch_pdl(_if)?\(|SPECPV_LAUNCH\(", s)}
    assert {"attn_tc.cu", "attn_simt.cu", "aux_kernels.cu", "proj_tc.cu", "score_tc.cu"} <= set(overlapped)
    for name, text in overlapped.items():
        assert not re.findall(r"__ldg\s*\(|ld\.global\.nc|__restrict__", text), name


@pytest.mark.parametrize("source", ["attn_tc.cu", "attn_pair.cu", "score_tc.cu", "proj_tc.cu"])
def test_lanes_of_a_warp_give_up_together(source):
    """A wait that can give up returns a value per lane, and so does a look at the abort flag: an exit, a condition of a loop or of a
    vote that depends on one comes after a vote of the whole warp, or the loop has no place where the lanes meet.  (Lanes that disagreed would wait for one another in different
    places, without a limit.)  Checked on the source: such a case cannot be brought about on a GPU that works."""
    own, loop = False, 0  # whether `ok` may differ between lanes
    lines = (build_mod.CSRC / source).read_text().split("\n")
    for n, line in enumerate(lines, 1):
        code = line.split("//")[0]
        if re.search(r"\bbool ok = ", code):
            own = False
        if re.search(r"\bfor \(", code) and code.startswith("    for ("):
            loop = n  # the outermost loop of a role
        if re.search(r"if \(!ok\) (break|return)|if \(ok\) ok = __all_sync", code):
            if "each lane by itself" in line:  # allowed in loops whose lanes meet nowhere
                end = next(i for i in range(n, len(lines)) if lines[i] == "    }")
                assert not re.search(r"_sync\(|__syncwarp", "\n".join(x.split("//")[0] for x in lines[loop - 1:end])), f"{source}:{n}"
            else:
                assert not own, f"{source}:{n} leaves without a vote"
        if re.search(r"\bok &?= .*__all_sync\(0xffffffffu, ", code):
            own = False if "ok &=" not in code else own
        elif re.search(r"\bok &?= (mbar|pair)_wait\(|\*abort_flag\) ok = ", code):
            own = True
