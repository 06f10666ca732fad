"""Builds libspecpv.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the binding's argument conversion beside it."""
from __future__ import annotations

import os
import shlex
import subprocess
import sys
import sysconfig
import warnings
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "lib" / "libspecpv.so"
PYCALLS = PKG / "lib" / ("pycalls" + sysconfig.get_config_var("EXT_SUFFIX"))  # per interpreter: another one builds its own
SOURCES = ["api.cu", "aux_kernels.cu", "attn_simt.cu", "attn_tc.cu", "attn_pair.cu", "score_tc.cu", "proj_tc.cu", "offload.cu", "selftest.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC,-fvisibility=hidden",
    "--expt-relaxed-constexpr",
]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if Path(cand).exists() else "nvcc"


def needs_build(target: Path = LIB) -> bool:
    if not target.exists():
        return True
    newest = max(p.stat().st_mtime for p in list(CSRC.iterdir()) + [PKG.parent / "include" / "specpv.h"])
    return newest > target.stat().st_mtime


def _build_pycalls() -> None:
    """The argument conversion needs a C compiler and Python's headers, which the library itself does without: where they are
    missing the binding converts through ctypes."""
    tmp = PYCALLS.with_suffix(f".{os.getpid()}.tmp")
    try:
        subprocess.run([*shlex.split(os.environ.get("CC") or "gcc"), "-O2", "-std=gnu11", "-Wall", "-fPIC", "-fvisibility=hidden",
                        "-shared", "-I", sysconfig.get_paths()["include"], str(CSRC / "pycalls.c"), "-o", str(tmp),
                        "-L", str(LIB.parent), "-lspecpv", "-Wl,-rpath,$ORIGIN"], check=True)
    except (OSError, subprocess.CalledProcessError) as e:
        PYCALLS.unlink(missing_ok=True)  # one of an older source must not be used
        warnings.warn(f"{PYCALLS.name} was not built ({e}): the binding's calls are converted through ctypes")
    else:
        os.replace(tmp, PYCALLS)


def build(force: bool = False, verbose: bool = False) -> Path:
    """Compile every .cu of the library into lib/libspecpv.so (static cudart, no libcuda link), then the argument conversion."""
    LIB.parent.mkdir(exist_ok=True)
    if force or needs_build():
        _build_lib(verbose)
    if force or needs_build(PYCALLS):
        _build_pycalls()
    return LIB


def _build_lib(verbose: bool) -> None:
    objdir = PKG / "lib" / "obj"
    objdir.mkdir(exist_ok=True)
    objs = []
    procs = []
    for src in SOURCES:
        obj = objdir / (src + ".o")
        cmd = [_nvcc(), *NVCC_FLAGS, "-c", str(CSRC / src), "-o", str(obj)]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(str(obj))
    failed = False
    for src, proc in procs:
        out, _ = proc.communicate()
        if proc.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= proc.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB.with_suffix(f".{os.getpid()}.tmp")
    subprocess.run([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", str(tmp), *objs,
                    "-cudart", "static"], check=True)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
