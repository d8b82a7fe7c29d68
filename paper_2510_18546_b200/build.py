"""Builds ``libenl.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and ``_enl.so``, the Python binding of its
per-layer calls (CPython C API, gcc), beside it."""
from __future__ import annotations

import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libenl.so")
BINDING = os.path.join(HERE, "_enl.so")
BINDING_SOURCE = os.path.join(CSRC, "enl_py.c")
SOURCES = ["enl_host.cu", "enl_attn_sm100.cu", "enl_attn_mass_sm100.cu", "enl_attn_small_sm100.cu", "enl_decode_sm100.cu", "enl_decode_cluster_sm100.cu", "enl_aux_kernels.cu", "enl_static_scratch.cu", "enl_cluster.cu", "enl_rope.cu", "enl_select.cpp"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared"]


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def _stale() -> bool:
    return _older(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "enl_py.c"] + [os.path.join(HERE, "..", "include", "enl.h")])


def build_library(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + \
              [os.path.join(CSRC, s) for s in SOURCES]
        subprocess.run(cmd, check=True)
    if force or _older(BINDING, [BINDING_SOURCE, os.path.join(HERE, "..", "include", "enl.h")]):
        subprocess.run(["gcc", "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-o", BINDING, BINDING_SOURCE,
                        "-L", HERE, "-lenl", "-Wl,-rpath,$ORIGIN"], check=True)
    return LIB


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
