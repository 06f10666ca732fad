"""Builds libspecpv.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the binding's argument conversion beside it."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "lib" / "libspecpv.so"
PYCALLS = PKG / "lib" / "pycalls.so"
SOURCES = ["api.cu", "aux_kernels.cu", "attn_simt.cu", "attn_tc.cu", "attn_pair.cu", "score_tc.cu", "proj_tc.cu", "offload.cu", "selftest.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC,-fvisibility=hidden",
    "--expt-relaxed-constexpr",
]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if Path(cand).exists() else "nvcc"


def needs_build() -> bool:
    if not LIB.exists() or not PYCALLS.exists():
        return True
    newest = max(p.stat().st_mtime for p in list(CSRC.iterdir()) + [PKG.parent / "include" / "specpv.h"])
    return newest > min(LIB.stat().st_mtime, PYCALLS.stat().st_mtime)


def _build_pycalls() -> None:
    tmp = PYCALLS.with_suffix(f".{os.getpid()}.tmp")
    subprocess.run([os.environ.get("CC") or "gcc", "-O2", "-std=gnu11", "-Wall", "-fPIC", "-fvisibility=hidden", "-shared",
                    "-I", sysconfig.get_paths()["include"], str(CSRC / "pycalls.c"), "-o", str(tmp),
                    "-L", str(LIB.parent), "-lspecpv", "-Wl,-rpath,$ORIGIN"], check=True)
    os.replace(tmp, PYCALLS)


def build(force: bool = False, verbose: bool = False) -> Path:
    """Compile every .cu of the library into lib/libspecpv.so (static cudart, no libcuda link), then lib/pycalls.so."""
    if not force and not needs_build():
        return LIB
    LIB.parent.mkdir(exist_ok=True)
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
    _build_pycalls()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
