"""Builds the CUDA library (sm_100a only) in-tree with nvcc; no GPU is needed to compile."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmoc_ffn.so")
FRONT_SOURCE = "torch_front.cpp"
FRONT = os.path.join(HERE, "_front.so")   # the PyTorch entry points' host side, linked against LIB
SOURCES = ["api.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "-Xcompiler", "-Wall", "--expt-relaxed-constexpr",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def front_built_for() -> str:
    """The interpreter and torch that a _front.so built now belongs to (it uses torch's C++ interface, which has no stable ABI)."""
    import sysconfig

    import torch
    return f"{sysconfig.get_config_var('SOABI')}, torch {torch.__version__}"


def _front_is_current() -> bool:
    if not os.path.exists(FRONT):
        return False
    with open(FRONT, "rb") as fh:
        if f"[{front_built_for()}]".encode() not in fh.read():
            return False
    have = os.path.getmtime(FRONT)
    include = os.path.join(os.path.dirname(HERE), "include")
    sources = [os.path.join(CSRC, FRONT_SOURCE)] + [os.path.join(include, n) for n in os.listdir(include)]
    return all(have >= os.path.getmtime(p) for p in sources)


def build_front() -> str:
    """Compile csrc/torch_front.cpp into _front.so, a CPython module that calls libmoc_ffn.so; returns its path."""
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    tmp = FRONT + ".tmp.%d" % os.getpid()
    libs = cpp_extension.library_paths(device_type="cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-Wall",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DMOC_FRONT_BUILT_FOR="[{front_built_for()}]"']
    cmd += ["-isystem" + p for p in cpp_extension.include_paths(device_type="cuda") + [sysconfig.get_paths()["include"]]]
    cmd += [os.path.join(CSRC, FRONT_SOURCE), "-o", tmp, "-L" + HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
    cmd += ["-L" + p for p in libs] + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
        raise RuntimeError("building _front.so failed")
    os.replace(tmp, FRONT)
    return FRONT


def _newest_source_mtime() -> float:
    newest = 0.0
    for root in (CSRC, os.path.join(os.path.dirname(HERE), "include")):
        for name in os.listdir(root):
            if name.endswith((".cu", ".cuh", ".h")):
                newest = max(newest, os.path.getmtime(os.path.join(root, name)))
    return newest


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libmoc_ffn.so and csrc/torch_front.cpp into _front.so, next to this file; returns the
    library's path."""
    if force or not os.path.exists(LIB) or os.path.getmtime(LIB) < _newest_source_mtime():
        _build_library(verbose)
    if force or not _front_is_current():
        build_front()
    return LIB


def _build_library(verbose: bool) -> None:
    tmp = LIB + ".tmp.%d" % os.getpid()
    extra = os.environ.get("MOC_FFN_NVCC_FLAGS", "").split()   # further compiler flags
    cmd = [_nvcc()] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + \
        [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
        raise RuntimeError("nvcc failed while building libmoc_ffn.so")
    if verbose:
        sys.stderr.write(proc.stdout + proc.stderr)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
