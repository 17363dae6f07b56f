"""Builds libpowerattn.so (nvcc, sm_100a; cross-compiles without a GPU) and the CPython module _calls.so over it,
in-tree."""
from __future__ import annotations

import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(PKG, "libpowerattn.so")
CALLS = os.path.join(PKG, "_calls.so")
SOURCES = ["api.cu", "layout.cu", "decode.cu", "prefill_sm100.cu", "backward.cu", "backward_sm100.cu"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(out: str, deps) -> bool:
    return not os.path.exists(out) or any(os.path.getmtime(d) > os.path.getmtime(out) for d in deps)


def _build_calls() -> None:
    torch_dir = os.path.dirname(importlib.util.find_spec("torch").origin)
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    cmd = ["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden", "-I", INCLUDE,
           "-isystem", sysconfig.get_path("include"), "-isystem", os.path.join(torch_dir, "include"),
           "-isystem", os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"), "-o", CALLS, os.path.join(CSRC, "calls.cpp"),
           LIB, "-L" + os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
           "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + os.path.join(torch_dir, "lib")]
    subprocess.run(cmd, check=True)


def build(force: bool = False, verbose: bool = False) -> str:
    header = os.path.join(INCLUDE, "powerattn.h")
    calls_src = os.path.join(CSRC, "calls.cpp")
    cuda_deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))] + [header]
    if force or _stale(LIB, cuda_deps):
        cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O3", "-lineinfo",
               "-Xcompiler", "-fPIC", "-shared", "-Xlinker", "-soname=libpowerattn.so", "-I", INCLUDE, "-I", CSRC, "-o", LIB]
        if verbose:
            cmd += ["-Xptxas", "-v"]
        cmd += [os.path.join(CSRC, s) for s in SOURCES]
        subprocess.run(cmd, check=True)
    if force or _stale(CALLS, [calls_src, header]):
        _build_calls()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
