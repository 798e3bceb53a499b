"""GPU parity of the paths arrays of several blocks take: CTA pairs on squares of tiles (both feeds, even
and odd block counts, the sample counts where the choice of path changes, a second exact chunk, several
dumps, accumulating), and rows that are no 16-byte multiples (repacked rows, e4m3 and fp16 planes built
from unaligned pieces), against the CPU oracle."""
import numpy as np
import pytest

import oracle
from _gpu_helpers import int_case, run_engine

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TC = 0
AUTO, PACKED, PLANES, PACKED_F8 = 0, 1, 2, 3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_1887_gb300 import corr
    corr.lib()


def _check(n, c, t, bits, feed=AUTO, n_dumps=1, accumulate=False):
    dumps = [int_case(11 * n + c + t + k, n, c, t, bits) for k in range(n_dumps)]
    refs = [oracle.xcorr_int(d, n, c, t, bits) for d in dumps]
    init = None
    if accumulate:
        init = np.random.default_rng(n).integers(-2 ** 40, 2 ** 40, size=(n_dumps,) + refs[0].shape)
    v = run_engine(np.concatenate([d.reshape(-1) for d in dumps]), n, c, t, bits, TC, n_dumps=n_dumps,
                   accumulate=accumulate, vis_init=init, operands=(feed, 0))
    for k in range(n_dumps):
        assert np.array_equal(v[k], refs[k] + (init[k] if accumulate else 0)), k


@pytest.mark.parametrize("feed", ["packed", "planes"])
@pytest.mark.parametrize("n,c,t,bits", [
    (80, 3, 128, 8), (128, 2, 129, 8), (128, 90, 192, 4), (72, 160, 256, 8), (192, 3, 257, 8), (176, 2, 320, 4),
    (256, 80, 200, 8), (256, 3, 1030, 8), (240, 2, 513, 4), (320, 2, 300, 8), (384, 30, 130, 4), (512, 3, 257, 8),
])
def test_pairs_bit_exact(feed, n, c, t, bits):
    _check(n, c, t, bits, PLANES if feed == "planes" else (PACKED if bits == 8 else PACKED_F8))


@pytest.mark.parametrize("n,c,t,bits,n_dumps", [(96, 5, 400, 8, 3), (128, 7, 1100, 8, 1), (256, 3, 600, 4, 2), (512, 2, 200, 8, 2),
                                                (192, 3, 500, 4, 1), (320, 2, 300, 4, 2), (400, 2, 260, 8, 1)])
def test_pairs_dumps_and_accumulate(n, c, t, bits, n_dumps):
    _check(n, c, t, bits, n_dumps=n_dumps)
    _check(n, c, t, bits, n_dumps=n_dumps, accumulate=True)


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n,c,t,bits", [
    (3, 7, 65, 8), (33, 5, 130, 8), (37, 3, 64, 4), (63, 160, 129, 8), (65, 9, 127, 4), (75, 33, 300, 8), (127, 3, 1030, 8),
    (129, 5, 257, 8), (131, 3, 400, 4), (191, 2, 64, 8), (250, 3, 140, 8), (255, 2, 520, 4), (301, 3, 129, 8), (450, 2, 300, 8),
])
def test_ragged_rows_bit_exact(n, c, t, bits, accumulate):
    _check(n, c, t, bits, n_dumps=2, accumulate=accumulate)


@pytest.mark.parametrize("n,c,t,bits", [(33, 3, 70, 8), (75, 4, 128, 4), (129, 2, 65, 8)])
def test_ragged_planes_hold_zero_past_the_last_input(n, c, t, bits):
    # the public planes: padded inputs and samples are zero whatever follows a row in memory
    from paper_0906_1887_gb300 import corr
    p = int_case(n, n, c, t, bits)
    plan = corr.Plan(n, c, t, bits)
    x = torch.from_numpy(np.ascontiguousarray(p).view(np.uint8).reshape(-1).copy()).cuda()
    planes = torch.full((plan.planes_size(1) // 2,), float("nan"), dtype=torch.float16, device="cuda")
    plan.unpack(x, planes, 1)
    torch.cuda.synchronize()
    nb, kp = (n + 63) // 64, (t + 63) // 64 * 64
    got = planes.cpu().numpy().reshape(c, nb * 64, 2, kp)
    re, im = oracle.unpack(p, n, c, t, bits)
    want = np.zeros((c, nb * 64, 2, kp), np.float16)
    want[:, :n, 0, :t] = np.asarray(re).reshape(t, c, n).transpose(1, 2, 0)
    want[:, :n, 1, :t] = np.asarray(im).reshape(t, c, n).transpose(1, 2, 0)
    assert np.array_equal(got, want)
    plan.close()
