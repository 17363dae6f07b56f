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
CALLS_STAMP = os.path.join(PKG, "_calls.stamp")  # what _calls.so was built against
SOURCES = ["api.cu", "layout.cu", "decode.cu", "prefill_sm100.cu", "backward.cu", "backward_sm100.cu"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(out: str, deps) -> bool:
    return not os.path.exists(out) or any(os.path.getmtime(d) > os.path.getmtime(out) for d in deps)


def _torch_dir() -> str:
    return os.path.dirname(importlib.util.find_spec("torch").origin)


def _torch_version() -> str:
    """torch.__version__, read without importing torch."""
    spec = importlib.util.spec_from_file_location("_torch_version", os.path.join(_torch_dir(), "version.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod.__version__


def _calls_key() -> str:
    """_calls.so uses the C++ interfaces of torch and CPython: it fits the versions it was built against only."""
    return "torch %s in %s, python %s" % (_torch_version(), _torch_dir(), sysconfig.get_config_var("SOABI"))


def _calls_stale(deps) -> bool:
    if _stale(CALLS, deps) or not os.path.exists(CALLS_STAMP):
        return True
    with open(CALLS_STAMP) as f:
        return f.read() != _calls_key()


def _build_calls() -> None:
    torch_dir = _torch_dir()
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    cmd = ["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden", "-I", INCLUDE,
           '-DPA_TORCH_VERSION="%s"' % _torch_version(),
           "-isystem", sysconfig.get_path("include"), "-isystem", os.path.join(torch_dir, "include"),
           "-isystem", os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"), "-o", CALLS, os.path.join(CSRC, "calls.cpp"),
           LIB, "-L" + os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
           "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + os.path.join(torch_dir, "lib")]
    subprocess.run(cmd, check=True)
    with open(CALLS_STAMP, "w") as f:
        f.write(_calls_key())


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
    if force or _calls_stale([calls_src, header]):
        _build_calls()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
