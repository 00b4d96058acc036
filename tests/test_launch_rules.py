"""The rules by which calls are cut into CTAs, compiled for the host from csrc/launch_rules.h."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_02199_b200", "csrc")
SMS = 148
SHIM = """
#include "launch_rules.h"
extern "C" int decode_splits(int sms, long long heads, long long len) { return lkv::decode_splits(sms, heads, len); }
extern "C" int decode_cluster(int sms, long long heads, int group, long long len) {
  return lkv::decode_cluster(sms, heads, group, len, lkv::decode_splits(sms, heads, len));
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    where = tmp_path_factory.mktemp("rules")
    (where / "shim.cpp").write_text(SHIM)
    lib = str(where / "rules.so")
    subprocess.run([cxx, "-shared", "-fPIC", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", lib, str(where / "shim.cpp")], check=True)
    return C.CDLL(lib)


def test_decode_splits_are_whole_tiles_and_never_empty(rules):
    for heads in (1, 3, 8, 33, 64, 400):
        for tiles in list(range(1, 200)) + [964, 4000]:
            n = rules.decode_splits(SMS, C.c_longlong(heads), C.c_longlong(64 * tiles))
            c = rules.decode_cluster(SMS, C.c_longlong(heads), 4, C.c_longlong(64 * tiles - 63))
            assert 1 <= n <= min(tiles, 512) and 0 <= c <= min(tiles, 16)


@pytest.mark.parametrize("heads", [1, 2, 3, 4, 5, 6])
def test_few_heads_give_no_cta_more_than_six_tiles_of_a_short_cache(rules, heads):
    # seven and eight tiles a CTA cost up to 12 % against splits by way of memory that have an SM each
    for group in range(1, 9):
        for tiles in range(1, 65):
            assert -(-tiles // rules.decode_cluster(SMS, C.c_longlong(heads), group, C.c_longlong(64 * tiles))) <= 6
