"""CPU check of how the FP32 engine splits the sample axis (fp32_sample_ranges): ranges of whole 32-sample
chunks that cover the dump, and never worse -- by waves of two blocks per SM times the samples of a range
and the 24 that an item costs besides -- than the plain rule of four items per SM."""
import ctypes

import pytest

from paper_0906_1887_gb300 import build as corr_build

N_SM, CHUNK = 152, 32


@pytest.fixture(scope="module")
def ranges():
    f = ctypes.CDLL(corr_build.build())["_ZN4corr18fp32_sample_rangesEiilPiS0_"]
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p]
    f.restype = None

    def call(n_time, items):
        ts, length = ctypes.c_int(), ctypes.c_int()
        f(n_time, N_SM, items, ctypes.byref(ts), ctypes.byref(length))
        return ts.value, length.value
    return call


def _up(a, b):
    return -(-a // b)


def _plain_rule(n_time, items):
    t = max(1, min(_up(4 * N_SM, items) if items < 4 * N_SM else 1, _up(n_time, 64)))
    length = _up(_up(n_time, t), CHUNK) * CHUNK
    return _up(n_time, length), length


def _cost(items, ts, length):
    return _up(items * ts, 2 * N_SM) * (length + 24)


def test_ranges_cover_the_dump_and_fill_the_chip(ranges):
    for items in list(range(1, 40)) + [75, 152, 192, 303, 304, 305, 400, 607, 608, 5000]:
        for n_time in (1, 63, 64, 100, 500, 1000, 4096, 5000, 10000, 20000, 40000, 65536, 100000, 10 ** 6, 2 * 10 ** 9):
            ts, length = ranges(n_time, items)
            assert length % CHUNK == 0 and (ts - 1) * length < n_time <= ts * length
            assert ts == 1 or length >= 64
            assert _cost(items, ts, length) <= _cost(items, *_plain_rule(n_time, items)), (items, n_time)


def test_no_items(ranges):
    assert ranges(100, 0) == (1, 128)
