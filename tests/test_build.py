"""Building the binding's two libraries, with compilers that stand in for the real ones."""
import os
import stat

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
