"""The binding's native call path on the CPU: arguments reach the library as the library's own checks see them, and what is
not a call is refused."""
import numpy as np
import pytest
import torch

from paper_2602_02199_b200 import binding as Bn


@pytest.fixture(scope="module")
def native():
    Bn.load()
    return Bn._pycall


def _message():
    return (Bn.load().laser_kv_last_error(None) or b"").decode()


def test_null_handles_and_pointers_are_refused_by_the_library(native):
    st = (128, 128, 128, 1)
    for f in (native.select_block, native.select_tail):
        assert f(0, 0, 16, 16, 16, st, st, 1, 0) == Bn.ERR_INVALID_ARG and "NULL handle" in _message()
    assert native.decode_attention(0, 0, 16, st, 0.0, 16, 16, 64, 0) == Bn.ERR_INVALID_ARG and "NULL handle" in _message()
    assert native.two_stage_topk(0, 0, 1, 8, 1, 1, 1, 0, 0) == Bn.ERR_INVALID_ARG
    assert native.consensus_accumulate(0, 0, 1, 1, 1, 8, 0, 0, 0, 0) == Bn.ERR_INVALID_ARG
    assert native.window_scores(0, 0, st, st, 1, 1, 1, 64, 16, 1, 0.0, 0, 0, 0, 0) == Bn.ERR_INVALID_ARG
    assert native.collision_counts(0, 0, 0, st, st, 1, 1, 1, 64, 16, 1, 8, 8, 0, 0, 0, 0) == Bn.ERR_INVALID_ARG


def test_every_argument_reaches_its_parameter(native):
    # the entries' range ends beyond the capacity: the message repeats 64-bit values of arguments 12, 15 and 8
    big = 1 << 40
    assert native.gather_append(16, 16, 8, 8, 5, 16, 1, 7, 16, 16, 8, big + 6, 16, 8, big, 0, 16, 0) == Bn.ERR_CAPACITY
    assert f"[{big}, {big + 7})" in _message() and f"{big + 6} entries" in _message()
    assert native.two_stage_topk(16, 16, 1, 16385, 1, 1, 1, 16, 0) == Bn.ERR_UNSUPPORTED
    assert native.two_stage_topk(16, 16, 1, 10, 4, 2, 1, 16, 0) == Bn.ERR_INVALID_ARG and "exceeds the segment" in _message()
    st = (128, 128, 128, 1)
    assert native.window_scores(16, 16, st, st, 1, 4, 1, 64, 16, 2, 0.5, 256, 100, 16, 0) == Bn.ERR_CAPACITY
    need = Bn.laser_kv_window_scores_scratch_bytes(1, 4, 1, 64, 16, 2)
    assert f"needs {need} bytes, got 100" in _message()
    assert native.window_scores(16, 16, st, st, 1, 4, 1, 64, 16, 2, -0.5, 256, need, 16, 0) == Bn.ERR_INVALID_ARG
    # 32-bit parameters take integers modulo 2^32, as ctypes does
    assert native.two_stage_topk(16, 16, (1 << 32) + 1, 16385, 1, 1, 1, 16, 0) == Bn.ERR_UNSUPPORTED


class _Seven:
    def __index__(self):
        return 7


@pytest.mark.parametrize("seven", [7, np.int64(7), np.uint8(7), torch.tensor(7), _Seven()], ids=lambda x: type(x).__name__)
def test_numbers_are_whatever_ctypes_takes_for_an_integer(native, seven):
    big = 1 << 40
    assert native.gather_append(16, 16, 8, 8, 5, 16, 1, seven, 16, 16, 8, np.int64(big + 6), 16, 8, np.int64(big), 0, 16, 0) == Bn.ERR_CAPACITY
    assert f"[{big}, {big + 7})" in _message() and f"{big + 6} entries" in _message()
    lib = Bn.load()                                      # the same arguments by way of ctypes
    assert lib.laser_kv_gather_append(16, 16, 8, 8, 5, 16, 1, seven, 16, 16, 8, np.int64(big + 6), 16, 8, np.int64(big), 0, 16, 0) == Bn.ERR_CAPACITY
    st = (128, seven, np.int32(128), 1)
    assert native.window_scores(16, 16, st, st, 1, 4, 1, 64, 16, 2, 0.5, 256, 100, 16, 0) == Bn.ERR_CAPACITY


def test_what_is_not_a_call_raises(native):
    with pytest.raises(TypeError):
        native.two_stage_topk(0, 0)
    with pytest.raises(TypeError):
        native.two_stage_topk(0, 0, 1.5, 8, 1, 1, 1, 0, 0)
    with pytest.raises(TypeError):
        native.two_stage_topk(0, 0, np.float64(1), 8, 1, 1, 1, 0, 0)
    with pytest.raises(TypeError):
        native.two_stage_topk(np.int64(0), 0, 1, 8, 1, 1, 1, 0, 0)             # an address
    with pytest.raises(ValueError):
        native.decode_attention(0, 0, 16, (128,), 0.0, 16, 16, 64, 0)
    with pytest.raises(ValueError):
        native.select_block(0, 0, 16, 16, 16, [128, 128, 128, 1], (128, 128, 128, 1), 1, 0)
    with pytest.raises(TypeError):
        native.decode_attention(0, 0, 16, (128, 128, 1), "1", 16, 16, 64, 0)
    with pytest.raises(OSError):
        native.setup("/nonexistent/liblaserkv.so")
    Bn._pycall.setup(Bn.lib_path())
