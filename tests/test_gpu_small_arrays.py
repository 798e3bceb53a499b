"""GPU parity of single-block arrays (at most 64 inputs): channels packed side by side in one tile,
and the packed-run epilogue (one bulk copy or add per 16 rows), against the CPU oracle.

Sizes are the edges of the packing: 2, 3, 4 .. 64 channels per tile, tiles not full (64 mod n inputs
left over), a last tile with fewer channels, rows below 16 bytes that only packed tiles can address,
channel pairs per item, a second exact chunk, and float runs that start at odd elements.
"""
import numpy as np
import pytest

import oracle
from oracle import dump as odump
from _gpu_helpers import check_bf16x3, int_case, run_engine

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TC, BF16X3 = 0, 2


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_1887_gb300 import corr
    corr.lib()


# (n, c, t, bits): few channels keep one tile per SM, so packing needs several channels per SM (152)
CASES = [
    (1, 1216, 65, 8), (1, 640, 200, 4), (2, 1000, 64, 8), (4, 644, 70, 8), (5, 640, 33, 8), (6, 800, 130, 8),
    (7, 768, 65, 8), (8, 613, 129, 8), (10, 616, 70, 8), (12, 612, 64, 4), (16, 609, 130, 8), (16, 1300, 257, 4),
    (20, 460, 65, 8), (21, 464, 64, 8), (24, 700, 1025, 8), (31, 320, 128, 8), (32, 305, 1100, 8), (32, 1000, 65, 4),
    (33, 304, 70, 8), (40, 305, 64, 8), (48, 311, 130, 4), (63, 16, 64, 8), (64, 305, 1030, 8),
]


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n,c,t,bits", CASES)
def test_packed_channels_bit_exact(n, c, t, bits, accumulate):
    p = int_case(50 + 3 * n + c + t, n, c, t, bits)
    ref = oracle.xcorr_int(p, n, c, t, bits)
    init = None
    if accumulate:
        init = np.random.default_rng(n).integers(-2 ** 40, 2 ** 40, size=(1,) + ref.shape)
    v = run_engine(p, n, c, t, bits, TC, accumulate=accumulate, vis_init=init)[0]
    assert np.array_equal(v, ref + (init[0] if accumulate else 0))


@pytest.mark.parametrize("n,c,t,n_dumps", [(16, 311, 70, 3), (10, 320, 64, 2), (48, 153, 65, 3)])
def test_packed_channels_several_dumps(n, c, t, n_dumps):
    dumps = [int_case(70 + k + n, n, c, t, 8) for k in range(n_dumps)]
    v = run_engine(np.concatenate([d.reshape(-1) for d in dumps]), n, c, t, 8, TC, n_dumps=n_dumps)
    for k in range(n_dumps):
        assert np.array_equal(v[k], oracle.xcorr_int(dumps[k], n, c, t, 8))


# odd n (n + 1) / 2: float runs start at odd elements, so heads and tails are single elements
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n,c,t", [(2, 700, 64), (6, 460, 100), (14, 620, 65), (16, 620, 130), (30, 310, 64), (62, 5, 70)])
def test_packed_float_channels_within_bound(n, c, t, accumulate):
    x = np.random.default_rng(n + c).normal(size=(t, c, n, 2)).astype(np.float32)
    init = None
    if accumulate:
        init = np.zeros((1, c, n * (n + 1) // 2, 2), np.float32)
    v = run_engine(x, n, c, t, 32, BF16X3, accumulate=accumulate, vis_init=init)[0]
    chans = [0, 1, c // 2, c - 1]
    check_bf16x3(v[chans], x, n, c, t, chans)


@pytest.mark.parametrize("offset", [0, 1])   # the output may start at any 8-byte unit
@pytest.mark.parametrize("n,c,t,bits", [(16, 620, 100, 4), (24, 330, 64, 8), (64, 5, 300, 8), (80, 3, 100, 8)])
def test_fused_dump_packed_channels_and_output_alignment(n, c, t, bits, offset):
    from paper_0906_1887_gb300 import corr
    rng = np.random.default_rng(n)
    p = int_case(5 + n, n, c, t, bits)
    plan = corr.Plan(n, c, t, bits)
    x = torch.from_numpy(p.view(np.uint8).reshape(-1).copy()).cuda()
    buf = torch.full((c * plan.n_baselines + 2, 2), float("nan"), dtype=torch.float32, device="cuda")
    out = buf[offset:offset + c * plan.n_baselines]
    tau, nu = rng.normal(0, 2e-6, n), 1.5e8 + 1e4 * np.arange(c)
    plan.run_dump(x, out, 3, torch.from_numpy(tau).cuda(), torch.from_numpy(nu).cuda())
    torch.cuda.synchronize()
    assert plan.check_device() == 0
    got = out.cpu().numpy().astype(np.float64).reshape(c, -1, 2)
    ref = odump.dump_corrected(oracle.xcorr_int(p, n, c, t, bits), 3, tau, nu)
    err = np.hypot(*(got - ref).transpose(2, 0, 1))
    assert np.all(err <= 8 * 2.0 ** -24 * np.hypot(ref[..., 0], ref[..., 1]) + 1e-30)
    rest = buf.cpu().numpy()
    assert np.isnan(rest[:offset]).all() and np.isnan(rest[offset + c * plan.n_baselines:]).all()
    plan.close()
