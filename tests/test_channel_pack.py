"""CPU check of the rule that packs channels of small arrays side by side in one tile (tc_channel_pack): the
tiles start where TMA can address them -- 16-byte multiples, below 2^31 in the copy's own unit (bytes of
4/8-bit samples, elements of complex floats), which is a 32-bit coordinate -- and hold whole channels."""
import ctypes

import pytest

from paper_0906_1887_gb300 import build as corr_build


@pytest.fixture(scope="module")
def pack():
    f = ctypes.CDLL(corr_build.build())["_ZN4corr15tc_channel_packEiiili"]
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int]
    f.restype = ctypes.c_int
    return f


@pytest.mark.parametrize("bps", [1, 2, 8])
def test_tiles_start_where_tma_can_address_them(pack, bps):
    for n in list(range(1, 34)) + [48, 64]:
        aligned = n * bps % 16 == 0
        for n_chan in [1, 2, 3, 7, 8, 16, 128, 1000, 4096, 2 ** 20, 2 ** 26, 2 ** 27 - 16, 2 ** 27, 2 ** 28, 2 ** 30, 2 ** 31 - 16]:
            for n_dumps, n_sm in [(1, 152), (3, 152), (1, 0)]:
                p = pack(n, bps, n_chan, n_dumps, n_sm)
                if p <= 1:
                    assert p == (1 if aligned else 0) and (p or not aligned)
                    continue
                step = p * n * (1 if bps == 8 else bps)   # from tile to tile, in the copy's unit
                assert p * n <= 64 and p <= n_chan and p * n * bps % 16 == 0 and n * bps * n_chan % 16 == 0
                last = (n_chan + p - 1) // p - 1
                assert last * step < 2 ** 31, (n, n_chan, p)


@pytest.mark.parametrize("n,bps,n_chan,n_dumps,n_sm,want", [
    (16, 2, 1300, 1, 152, 4), (8, 2, 613, 1, 152, 4), (9, 8, 512, 1, 152, 2), (31, 8, 512, 1, 152, 2), (4, 1, 2 ** 20, 1, 0, 16),
    (8, 2, 2 ** 27 - 1, 1, 152, 8), (8, 2, 2 ** 27, 1, 152, 1), (7, 2, 2 ** 28, 1, 152, 0), (2, 8, 2 ** 30 - 2, 1, 152, 32)])
def test_known_packings(pack, n, bps, n_chan, n_dumps, n_sm, want):
    assert pack(n, bps, n_chan, n_dumps, n_sm) == want
