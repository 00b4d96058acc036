"""Building the binding's two libraries, with compilers that stand in for the real ones."""
import os
import shutil
import stat
import subprocess
import sys

import pytest

from paper_2602_02199_b200 import build as B


def _compiler(path, text):
    path.write_text("#!/bin/sh\n" + text)
    path.chmod(path.stat().st_mode | stat.S_IXUSR)
    return str(path)


# writes half of its output and fails, or ends well: the output is what follows -o
HALF = 'while [ "$1" != -o ]; do shift; done; printf half > "$2"; exit 1\n'
WHOLE = 'while [ "$1" != -o ]; do shift; done; printf whole > "$2"\n'


@pytest.fixture
def targets(tmp_path, monkeypatch):
    monkeypatch.setattr(B, "LIB", str(tmp_path / "liblaserkv.so"))
    monkeypatch.setattr(B, "PYCALL", str(tmp_path / "_pycall.so"))
    for name in (B.LIB, B.PYCALL):
        with open(name, "w") as f:
            f.write("before")
    return tmp_path


@pytest.mark.parametrize("which", ["NVCC", "CXX"])
def test_a_library_is_replaced_as_a_whole_or_not_at_all(targets, tmp_path, monkeypatch, which):
    for var in ("NVCC", "CXX"):
        monkeypatch.setenv(var, _compiler(tmp_path / ("ok_" + var), WHOLE))
    monkeypatch.setenv(which, _compiler(tmp_path / "fails", HALF))
    with pytest.raises(RuntimeError):
        B.build(force=True)
    broken = B.LIB if which == "NVCC" else B.PYCALL
    assert open(broken).read() == "before"
    monkeypatch.setenv(which, _compiler(tmp_path / "works", WHOLE))
    B.build(force=True)
    assert open(B.LIB).read() == open(B.PYCALL).read() == "whole"
    assert sorted(n for n in os.listdir(targets) if n.endswith(".so")) == ["_pycall.so", "liblaserkv.so"]


LOAD = """
import sys, warnings
warnings.simplefilter("error" if sys.argv[2] == "native" else "always")
from paper_2602_02199_b200 import binding as Bn
Bn.load(build_if_missing=sys.argv[1] == "build")
assert (type(Bn._pycall).__name__ == "module") == (sys.argv[2] == "native"), Bn._pycall
st = (128, 128, 128, 1)
assert Bn._pycall.select_block(0, 0, 16, 16, 16, st, st, 1, 0) == Bn.ERR_INVALID_ARG
assert Bn._pycall.decode_attention(0, 0, 16, st, 0.0, 16, 16, 64, 0) == Bn.ERR_INVALID_ARG
assert Bn._pycall.window_scores(16, 16, st, st, 1, 4, 1, 64, 16, 2, 0.5, 256, 100, 16, 0) == Bn.ERR_CAPACITY
need = Bn.laser_kv_window_scores_scratch_bytes(1, 4, 1, 64, 16, 2)
assert f"needs {need} bytes, got 100" in Bn.load().laser_kv_last_error(None).decode()
try:
    Bn._pycall.two_stage_topk(0, 0, 1.5, 8, 1, 1, 1, 0, 0)
    assert False
except Exception as e:
    assert type(e).__name__ in ("TypeError", "ArgumentError")
"""


# the library is there and up to date, the native call path is not
@pytest.mark.parametrize("cxx,build,path", [("/nonexistent/c++", "build", "ctypes"), ("{fails}", "build", "ctypes"), ("{fails}", "no", "ctypes"),
                                            ("env -u UNSET g++", "build", "native")])
def test_the_library_loads_without_the_native_call_path(tmp_path, cxx, build, path):
    from paper_2602_02199_b200 import binding
    if path == "native" and not shutil.which("g++"):
        pytest.skip("no g++")
    root = os.path.dirname(os.path.dirname(os.path.abspath(binding.__file__)))
    binding.load()
    shutil.copytree(os.path.join(root, "paper_2602_02199_b200"), tmp_path / "paper_2602_02199_b200",
                    ignore=shutil.ignore_patterns("_pycall*", "__pycache__"))
    shutil.copytree(os.path.join(root, "include"), tmp_path / "include")
    env = dict(os.environ, CXX=cxx.format(fails=_compiler(tmp_path / "fails", HALF)), PYTHONPATH=str(tmp_path))
    subprocess.run([sys.executable, "-c", LOAD, build, path], cwd=tmp_path, env=env, check=True)
