"""Builds in-tree, with nvcc for sm_100a, liblaserkv.so (the C-ABI CUDA library) and, with the host compiler, the binding's
native call path."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblaserkv.so")
PYCALL = os.path.join(HERE, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
API = os.path.join(HERE, "..", "include", "laser_kv.h")
SOURCES = ["api.cu"]
HEADERS = ["launch_rules.h", "ptx.cuh", "theory_math.cuh", "stream_gemm.cuh", "aux_kernels.cuh", "query_proj.cuh", "decode_attn.cuh"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; the CUDA toolkit is required to build liblaserkv.so")


def _older(target: str, deps: list) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def needs_build() -> bool:
    return _older(LIB, [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [API])


def _build_pycall(force: bool) -> None:
    src = os.path.join(CSRC, "pycall.cpp")
    if not force and not _older(PYCALL, [src, API]):
        return
    cxx = os.environ.get("CXX") or shutil.which("g++") or shutil.which("c++")
    if not cxx:
        raise RuntimeError("no C++ compiler found; one is required to build the binding's native call path")
    res = subprocess.run([cxx, "-shared", "-fPIC", "-O2", "-std=c++17", "-I", sysconfig.get_paths()["include"], "-o", PYCALL, src],
                         capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("building the binding's native call path failed:\n" + res.stdout + res.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    _build_pycall(force)
    if not force and not needs_build():
        return LIB
    cmd = [_nvcc(), "-shared", "-Xcompiler", "-fPIC", "-gencode", "arch=compute_100a,code=sm_100a",
           "-lineinfo", "-O3", "-std=c++17", "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
