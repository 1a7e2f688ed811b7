"""Build libfact.so in-tree with nvcc for sm_100a, and the Python extension beside it (no JIT cache, no pip install).

    python -m paper_2604_26666_b200.build [--force] [--verbose]

FACT_EXPERIMENTS=1 in the environment adds -DFACT_EXPERIMENTS: a library for timing experiments whose kernels
honour the work-skipping FACT_DEBUG_FLAGS bits (loads, products or stores left out; results are garbage).
The default build has no such code.
"""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys
import sysconfig
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "libfact.so"
STAMP = PKG / "libfact.so.srchash"
BIND_SOURCE = CSRC / "bind.cpp"
BIND_LIB = PKG / "_fact_bind.so"  # the ordinary call's marshalling (CPython extension, linked to libfact.so beside it)
BIND_STAMP = PKG / "_fact_bind.so.srchash"

SOURCES = ["fact_api.cu"]
HEADERS = ["gemm_kernel.cuh", "grouped_kernel.cuh", "skinny_kernel.cuh", "kcluster_kernel.cuh", "attention_kernel.cuh", "attention_tiles_kernel.cuh", "attention_decode_kernel.cuh",
           "norm_kernel.cuh", "tune_kernels.cuh", "ptx.cuh"]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "--shared", "-Xcompiler", "-fPIC",
    "--expt-relaxed-constexpr",
]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if os.path.exists(cand) else "nvcc"


def _flags() -> list:
    return NVCC_FLAGS + (["-DFACT_EXPERIMENTS"] if os.environ.get("FACT_EXPERIMENTS") == "1" else [])


def source_hash() -> str:
    h = hashlib.sha1()
    for f in [CSRC / s for s in SOURCES + HEADERS] + [ROOT / "include" / "fact.h"]:
        h.update(f.read_bytes())
    h.update(" ".join(_flags()).encode())
    return h.hexdigest()


def is_current() -> bool:
    return LIB.exists() and STAMP.exists() and STAMP.read_text().strip() == source_hash()


def build(force: bool = False, verbose: bool = False) -> Path:
    if is_current() and not force:
        return LIB
    cmd = [_nvcc(), *_flags(), "-I", str(ROOT / "include"), "-I", str(CSRC)]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [str(CSRC / s) for s in SOURCES]
    tmp = LIB.with_suffix(f".tmp{os.getpid()}.so")
    cmd += ["-o", str(tmp)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(r.stderr)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    os.replace(tmp, LIB)
    STAMP.write_text(source_hash() + "\n")
    return LIB


def bind_hash() -> str:
    import torch

    h = hashlib.sha1()
    for f in (BIND_SOURCE, ROOT / "include" / "fact.h"):
        h.update(f.read_bytes())
    h.update(f"{torch.__version__} {sys.version}".encode())
    return h.hexdigest()


def build_bind(force: bool = False) -> Path:
    """The extension that binding.py calls; needs libfact.so (which it links to) and torch's headers."""
    if not force and BIND_LIB.exists() and BIND_STAMP.exists() and BIND_STAMP.read_text().strip() == bind_hash():
        return BIND_LIB
    import torch

    t = Path(torch.__file__).resolve().parent
    tmp = BIND_LIB.with_suffix(f".tmp{os.getpid()}.so")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-isystem", str(t / "include"), "-isystem", str(t / "include" / "torch" / "csrc" / "api" / "include"),
           "-isystem", str(Path(_nvcc()).resolve().parent.parent / "include"), "-I", sysconfig.get_paths()["include"],
           "-I", str(ROOT / "include"), str(BIND_SOURCE), "-o", str(tmp), f"-L{PKG}", "-l:libfact.so", f"-L{t / 'lib'}",
           "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("the binding extension failed to build:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    os.replace(tmp, BIND_LIB)
    BIND_STAMP.write_text(bind_hash() + "\n")
    return BIND_LIB


def bind_problem():
    """Why the extension in the tree cannot be used, or None."""
    if not BIND_LIB.exists():
        return f"{BIND_LIB} is missing"
    if BIND_STAMP.exists() and BIND_SOURCE.exists() and BIND_STAMP.read_text().strip() != bind_hash():
        return f"{BIND_LIB} was built from other sources, or for another torch or Python"
    return None


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
    print(build_bind(force="--force" in sys.argv))
