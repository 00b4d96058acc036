"""Builds in-tree, with nvcc for sm_100a, liblaserkv.so (the C-ABI CUDA library) and, with the host compiler, the binding's
native call path."""
from __future__ import annotations

import os
import shlex
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


def _link(cmd: list, target: str, what: str) -> str:
    """Runs a compiler that writes `target`, by way of a file of this process's own: another process that loads or builds the same
    file sees all of it or none."""
    part = f"{target}.{os.getpid()}.so"
    try:
        res = subprocess.run(cmd + ["-o", part], capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(what + " failed:\n" + res.stdout + res.stderr)
        os.replace(part, target)
    finally:
        if os.path.exists(part):
            os.remove(part)
    return res.stderr


def needs_build() -> bool:
    return _older(LIB, [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [API])


def build_pycall(force: bool = False) -> None:
    src = os.path.join(CSRC, "pycall.cpp")
    if not force and not _older(PYCALL, [src, API]):
        return
    cxx = shlex.split(os.environ.get("CXX") or "") or [c for c in ("g++", "c++") if shutil.which(c)][:1]
    if not cxx or not shutil.which(cxx[0]):
        raise RuntimeError("no C++ compiler found; one is required to build the binding's native call path")
    _link(cxx + ["-shared", "-fPIC", "-O2", "-std=c++17", "-I", sysconfig.get_paths()["include"], src], PYCALL,
          "building the binding's native call path")


def build(force: bool = False, verbose: bool = False) -> str:
    build_pycall(force)
    return build_lib(force, verbose)


def build_lib(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    cmd = [_nvcc(), "-shared", "-Xcompiler", "-fPIC", "-gencode", "arch=compute_100a,code=sm_100a",
           "-lineinfo", "-O3", "-std=c++17"] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    log = _link(cmd, LIB, "nvcc")
    if verbose:
        print(log)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
