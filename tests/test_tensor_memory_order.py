"""Kernels that start beside one another on an SM and share its tensor memory, read from their sources: none waits for another
grid while it holds columns, because a CTA of that grid may still have to allocate its own."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_02199_b200", "csrc")


def _kernels():
    """(name, body without comments) of every kernel that allocates tensor memory."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\s*\(", src):
            begin = end = src.index("{", m.end())
            depth = 0
            while True:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
                if depth == 0:
                    break
            if "tmem_alloc(" in src[begin:end]:
                found.append((m.group(1), src[begin:end]))
    return found


def test_the_kernels_are_found():
    assert sorted(name for name, _ in _kernels()) == ["qsig_kernel", "stream_kernel"]


@pytest.mark.parametrize("name,body", _kernels(), ids=lambda x: x if x.endswith("_kernel") else "")
def test_no_wait_for_a_grid_while_tensor_memory_is_held(name, body):
    alloc, dealloc = body.index("tmem_alloc("), body.rindex("tmem_dealloc(")
    assert alloc < dealloc and "return" not in body[alloc:dealloc]
    assert "grid_dependency_wait(" not in body[alloc:dealloc]
