"""Build libthc.so in-tree with nvcc for sm_100a, and the CPython module that marshals calls to it.

    python -m paper_2302_08545_b200._build [--force]

Flags that matter for reproducibility: -fmad=false (only the fmaf() calls written in the
sources are fused) and no fast-math (denormals kept, IEEE division and square root).
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libthc.so")
BINDING = os.path.join(HERE, "_binding.so")
BINDING_SOURCE = os.path.join(CSRC, "binding.c")
SOURCES = ["thc.cu", "thc_block.cu", "thc_noalloc.cu"]
HEADERS = ["thc_device.cuh", "thc_pipeline.cuh", "thc_block.h", os.path.join("..", "..", "include", "thc.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-fmad=false", "-prec-div=true", "-prec-sqrt=true", "-ftz=false",
    "-Xcompiler", "-fPIC", "-shared",
    "-cudart", "shared",
    "--threads", "3",                # the source files side by side
]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(p) > t for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        _build_library(verbose)
    _build_binding(force)
    return LIB


def _build_library(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
        ["-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed building libthc.so")
    if verbose:
        sys.stderr.write(res.stderr)


def _build_binding(force: bool) -> None:
    """Linked to libthc.so by soname and $ORIGIN, so that it uses the copy next to it."""
    deps = [BINDING_SOURCE, os.path.join(CSRC, HEADERS[-1]), os.path.abspath(__file__)]
    if not force and os.path.exists(BINDING) and all(os.path.getmtime(p) <= os.path.getmtime(BINDING) for p in deps):
        return
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-std=c11", "-Wall", "-fPIC", "-shared",
           "-I" + sysconfig.get_paths()["include"], "-o", BINDING, BINDING_SOURCE,
           "-L" + HERE, "-l:libthc.so", "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("gcc failed building _binding.so")


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
