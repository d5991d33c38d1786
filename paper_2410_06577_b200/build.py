"""Builds the CUDA library in-tree: ``nvcc`` for sm_100a, one shared object beside the package, and
the CPython module that marshals its arguments.

    python -m paper_2410_06577_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
INCLUDE = os.path.join(_ROOT, "include")
LIB_PATH = os.path.join(_PKG, "librodimus_ddts.so")
BINDING_PATH = os.path.join(_PKG, "_binding.so")

SOURCES = ["rodimus_ddts.cu", "ddts_step.cu", "ddts_fwd_simt.cu", "ddts_plan.cu", "ddts_fwd_tc.cu", "ddts_fwd_pair.cu", "ddts_fwd_scan.cu", "ddts_noalloc.cu", "ddts_probe.cu", "ddts_bwd.cu", "ddts_bwd_tc.cu", "swska_fwd.cu", "swska_fwd_tc.cu"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale(target: str, suffixes) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(suffixes)] + \
           [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return any(os.path.getmtime(d) > t for d in deps)


def _build_binding() -> None:
    """The CPython module, against the headers and libraries of the installed PyTorch."""
    import torch
    root = os.path.dirname(torch.__file__)
    tmp = BINDING_PATH + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-o", tmp,
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", INCLUDE, "-I", sysconfig.get_paths()["include"], "-I", "/usr/local/cuda/include",
           "-I", os.path.join(root, "include"),
           "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(CSRC, "binding.cpp"), "-L", os.path.join(root, "lib"),
           "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, BINDING_PATH)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every ``.cu`` file for sm_100a and link ``librodimus_ddts.so``; returns its path."""
    if force or _stale(BINDING_PATH, (".cpp",)):
        _build_binding()
    if not force and not _stale(LIB_PATH, (".cu", ".cuh")):
        return LIB_PATH
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC, "-o", tmp]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
