"""Which kernel an F-stage call takes (fwide_takes), on the CPU, and that every geometry of the plain
transforms' kernel gives a frame the same bits."""
import ctypes
import math

import numpy as np
import pytest

from paper_0906_1887_gb300 import build as corr_build

C8, C4, R8 = 0, 1, 2
N_SM = 152


@pytest.fixture(scope="module")
def takes():
    f = ctypes.CDLL(corr_build.build())["_ZN4corr11fwide_takesEiiiiii"]
    f.argtypes, f.restype = [ctypes.c_int] * 6, ctypes.c_bool
    return lambda kind, log2l, n, taps, frames: f(kind, log2l, n, taps, frames, N_SM)


def test_plain_transforms_keep_one_family_of_kernels(takes):
    for kind in (C8, C4, R8):
        for lg in range(3, 13):
            for n in (1, 7, 16, 50, 64, 75, 100, 8192):
                got = {takes(kind, lg, n, 0, f) for f in (1, 3, 100, 10 ** 6)}
                words = n <= 32 or n * (2 if kind == C8 else 1) % 4 == 0 or lg not in (6, 7)
                assert got == {lg >= 8 if kind == R8 else lg >= 5 and (lg != 6 or n % 64 != 0) and words}, (kind, lg, n)


def test_filterbanks_take_the_register_window_once_they_fill_the_chip(takes):
    for kind in (C8, C4, R8):
        for lg in range(3, 13):
            for taps in range(1, 20):
                for n in (1, 3, 5, 16, 64, 65, 128, 336, 1024):
                    got = [takes(kind, lg, n, taps, f) for f in (1, 4, 16, 64, 256, 1024, 10 ** 4, 10 ** 5, 10 ** 6)]
                    assert got == sorted(got), (kind, lg, taps, n)          # from a number of frames on, or never
                    if lg < 5 or taps > 8 or lg > (11 if kind == R8 else 10):
                        assert not any(got)
                    elif taps > 4 and not (kind == R8 and lg == 5 and n <= 64) and (kind == R8 or lg < 8 or taps >= lg - 5):
                        assert got[-1] and not (got[0] and n < 65), (kind, lg, taps, n)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,log2l", [(C8, 5), (C8, 7), (C4, 8), (C8, 9), (C4, 10), (C8, 11), (C8, 12), (R8, 8), (R8, 9), (R8, 10),
                                        (R8, 11), (R8, 12)])
def test_every_row_width_gives_the_same_bits(kind, log2l):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_1887_gb300 import corr
    L, bps = 1 << log2l, 2 if kind == C8 else 1
    c = L // 2 if kind == R8 else L
    frames = max(40, (1 << 17) // L)

    def run(x, n):
        fp = corr.FPlan(n, c, kind)
        f = x.numel() // (L * n * bps)
        spec = torch.full((f * fp.n_out_chan * n * 2 + 64,), float("nan"), device="cuda")
        fp.run(x, spec, f)
        torch.cuda.synchronize()
        fp.close()
        assert torch.isnan(spec[-64:]).all()
        return spec[:-64].reshape(f, -1, n, 2)

    g = torch.Generator(device="cuda")
    g.manual_seed(log2l)
    x = torch.randint(0, 256, (frames * L, 144, bps), generator=g, device="cuda", dtype=torch.uint8)   # rows of 16, full
    whole = run(x.reshape(-1), 144)
    for n in (1, 2, 3, 4, 6, 12, 20, 75, 100):       # fewer inputs: rows of 1 and 4, odd rows, empty columns
        for f in (1, 3, frames):
            part = x[:f * L, 144 - n:].contiguous().reshape(-1)
            assert torch.equal(run(part, n), whole[:f, :, 144 - n:]), (n, f)
    assert torch.equal(run(x[L:4 * L].reshape(-1), 144), whole[1:4])
    s = x[:L].cpu().numpy()
    v = s.view(np.int8).astype(np.float64)
    z = v[..., 0] + 1j * v[..., 1] if kind == C8 else v[..., 0] if kind == R8 else (
        (s.view(np.int8)[..., 0] >> 4).astype(float) + 1j * ((s << 4).view(np.int8)[..., 0] >> 4))
    ref = np.fft.fft(z, axis=0)[:whole.shape[1]]
    got = whole[0].cpu().numpy().astype(np.float64)
    err = np.linalg.norm(got[..., 0] + 1j * got[..., 1] - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() <= 4 * 2.0 ** -24 * math.log2(L)
