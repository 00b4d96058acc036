"""The rules by which calls are cut into CTAs, compiled for the host from csrc/launch_rules.h."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

import test_gpu_decode_memory as memory

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_02199_b200", "csrc")
SMS = 148
# clusters of 0 to 16 decode CTAs that such a device holds at once (9 to 15 are not used)
ROOM = [0, 0, 148, 93, 71, 56, 45, 37, 33, 0, 0, 0, 0, 0, 0, 0, 14]
SHIM = """
#include "launch_rules.h"
extern "C" int decode_splits(int sms, long long heads, long long len) { return lkv::decode_splits(sms, heads, len); }
extern "C" int decode_cluster(int sms, long long heads, int group, long long len, const int* room) {
  return lkv::decode_cluster(sms, heads, group, len, lkv::decode_splits(sms, heads, len), [=](int n) { return room[n]; });
}
extern "C" int append_beside(int sms, int nseg, long long ctas) { return lkv::append_beside(sms, nseg, ctas); }
extern "C" int lse_batch() { return lkv::kLseBatch; }
extern "C" int lse_split(int partials) { return lkv::lse_split(partials); }
extern "C" int proj_slices(int sms, int grid, long long seg_tiles, int chunks, int rows, int lse, long long qsig, int parts, int* begin, int* abreast) {
  const lkv::ProjSlices s = lkv::proj_slices(sms, grid, seg_tiles, chunks, rows, lse, qsig, parts);
  const long long tiles = seg_tiles * chunks;
  *abreast = s.abreast;
  for (int c = 0; s.w_early > 0 && c < grid; ++c) {       // as the kernel: begin and end of every CTA's slice
    const int n = grid / s.abreast;
    const long long part = tiles / s.abreast, first = part * (c % s.abreast);
    begin[2 * c] = (int)(first + lkv::weighted_begin(part, c / s.abreast, n, s));
    begin[2 * c + 1] = (int)(first + lkv::weighted_begin(part, c / s.abreast + 1, n, s));
  }
  return s.n_late;
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


def cluster(rules, heads, group, length, room=ROOM):
    return rules.decode_cluster(SMS, C.c_longlong(heads), group, C.c_longlong(length), (C.c_int * 17)(*room))


def test_decode_splits_are_whole_tiles_and_never_empty(rules):
    for heads in (1, 3, 8, 33, 64, 400):
        for tiles in list(range(1, 200)) + [964, 4000]:
            n = rules.decode_splits(SMS, C.c_longlong(heads), C.c_longlong(64 * tiles))
            c = cluster(rules, heads, 4, 64 * tiles - 63)
            assert 1 <= n <= min(tiles, 512) and 0 <= c <= min(tiles, 16)


@pytest.mark.parametrize("heads", [1, 2, 3, 4, 5, 6])
def test_few_heads_give_no_cta_more_than_six_tiles_of_a_short_cache(rules, heads):
    # seven and eight tiles a CTA cost up to 12 % against splits by way of memory that have an SM each
    for group in range(1, 9):
        for tiles in range(1, 65):
            assert -(-tiles // cluster(rules, heads, group, 64 * tiles)) <= 6


def test_the_shapes_of_the_memory_route_take_it(rules):
    for shape in memory.SHAPES:
        batch, heads, group = shape[:3]
        assert cluster(rules, batch * heads, group, memory.entries(shape)) == 0


@pytest.mark.parametrize("room", [[0] * 17, [0, 0] + [1] * 7 + [0] * 8, ROOM[:9] + [0] * 8, [n // 4 for n in ROOM]])
def test_clusters_the_device_does_not_hold_are_not_launched(rules, room):
    fewer = 0
    for heads in (1, 2, 4, 6, 8, 9, 16, 32, 40, 64, 128, 300):
        for group in (1, 4, 8):
            for tiles in (1, 2, 7, 8, 26, 48, 49, 64, 65, 100, 255, 964):
                n, usual = cluster(rules, heads, group, 64 * tiles, room), cluster(rules, heads, group, 64 * tiles)
                assert n <= 1 or heads <= room[n]
                assert n == usual or heads > room[usual]       # what fits is launched as ever
                fewer += n != usual
    assert fewer > 0


@pytest.mark.parametrize("partials", range(1, 21))
def test_normaliser_partials_are_fetched_in_one_round_trip(rules, partials):
    a_warps = -(-partials // 4) if rules.lse_split(partials) else partials
    assert a_warps <= rules.lse_batch()


def test_large_appends_of_many_segments_do_not_start_beside_the_selection(rules):
    for nseg, rows, beside in ((8, 3855, 1), (64, 1736, 1), (80, 864, 1), (128, 432, 1), (80, 1736, 0), (128, 816, 0), (149, 64, 0),
                               (128, 3855, 0)):
        assert rules.append_beside(SMS, nseg, C.c_longlong(-(-rows // 64) * nseg)) == beside
    # launched early or not, one rule for every number of segments: fewer CTAs never start later
    for nseg in range(1, 200):
        early = [rules.append_beside(SMS, nseg, C.c_longlong(ctas)) for ctas in range(1, 3000, 37)]
        assert early == sorted(early, reverse=True)


def slices(rules, seg_tiles, chunks, rows, qsig, parts=1):
    """(CTAs that start late, [begin, end) of every CTA's slice or None where they are equal, chunks abreast)."""
    lse, grid = min(SMS, seg_tiles), min(SMS, seg_tiles * chunks)
    out, abreast = (C.c_int * (2 * grid))(), C.c_int()
    late = rules.proj_slices(SMS, grid, C.c_longlong(seg_tiles), chunks, rows, lse, C.c_longlong(qsig), parts, out, C.byref(abreast))
    return late, list(zip(out[::2], out[1::2])) if late else None, abreast.value


@pytest.mark.parametrize("rows", [64, 128, 160, 192])
def test_slices_of_the_projection_pass_are_the_tiles_in_turn(rules, rows):
    weighted = 0
    for seg_tiles in list(range(1, 300, 7)) + [1024, 8192, 65536, 300000]:
        for chunks in (1, 2, 3, 4, 5, 8):
            for qsig in (1, 4, 16, 64, 147, 148, 500):
                late, cut, abreast = slices(rules, seg_tiles, chunks, rows, qsig)
                if cut is None:
                    continue
                weighted += 1
                assert 0 < late <= qsig and all(b <= e for b, e in cut)
                ends = sorted(x for x in cut if x[0] < x[1])
                assert ends[0][0] == 0 and ends[-1][1] == seg_tiles * chunks
                assert all(a[1] == b[0] for a, b in zip(ends, ends[1:]))
                if seg_tiles * 128 * 256 > 24 << 20:           # neighbours read the same keys
                    assert abreast == (chunks if SMS % chunks == 0 else 1)
                    for i in range(0, len(cut) - abreast, abreast):
                        places = [cut[i + k][0] - k * seg_tiles * chunks // abreast for k in range(abreast)]
                        assert max(places) == min(places)
    assert weighted > 100


@pytest.mark.parametrize("seg_tiles,chunks,qsig", [(48, 1, 4), (64, 1, 16), (64, 2, 4), (84, 4, 64), (96, 1, 16), (128, 1, 16), (132, 1, 16)])
def test_slices_are_equal_where_no_cta_starts_late(rules, seg_tiles, chunks, qsig):
    # every log-sum-exp CTA finds an SM without a signature CTA: a slice of two tiles beside one of none would take a tile longer
    assert slices(rules, seg_tiles, chunks, 160, qsig)[:2] == (0, None)
    assert slices(rules, SMS - qsig + 1, chunks, 160, qsig)[0] == 1
    # a window scored in parts: an ordinary launch between the parts lets every CTA start alike
    assert slices(rules, 8192, chunks, 160, qsig)[0] == qsig and slices(rules, 8192, chunks, 160, qsig, parts=2)[0] == 0
