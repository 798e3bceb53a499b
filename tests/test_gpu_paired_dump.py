"""GPU parity of the paths of CTA pairs that other tests leave out: the fused dump (8- and 4-bit, squares off the
diagonal, half-empty squares, odd baseline runs, outputs at an odd 8-byte unit), and float dumps added into
visibilities that are not zero."""
import numpy as np
import pytest

import oracle
from oracle import dump as odump
from _gpu_helpers import check_bf16x3, int_case, run_engine

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# pairs take even block counts above two, two blocks from 129 samples and odd counts from 257
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n,c,t,bits,n_dumps,delays", [
    (80, 3, 200, 8, 1, True), (128, 2, 1000, 8, 2, True), (256, 2, 130, 8, 1, True), (200, 3, 100, 8, 2, True), (400, 1, 300, 8, 1, True),
    (208, 2, 100, 4, 1, True), (256, 3, 500, 4, 2, True), (192, 2, 300, 8, 1, False), (320, 1, 1024, 8, 1, True), (400, 2, 260, 4, 1, True)])
def test_fused_dump_in_pairs(n, c, t, bits, n_dumps, delays, offset):
    from paper_0906_1887_gb300 import corr
    rng = np.random.default_rng(n + t)
    dumps = [int_case(40 + n + k, n, c, t, bits) for k in range(n_dumps)]
    plan = corr.Plan(n, c, t, bits)
    x = torch.from_numpy(np.concatenate([d.reshape(-1) for d in dumps]).view(np.uint8).copy()).cuda()
    size = n_dumps * c * plan.n_baselines
    buf = torch.full((size + 2, 2), float("nan"), dtype=torch.float32, device="cuda")
    tau, nu = rng.normal(0, 2e-6, n) if delays else np.zeros(n), 1.5e8 + 1e4 * np.arange(c)
    args = (torch.from_numpy(tau).cuda(), torch.from_numpy(nu).cuda()) if delays else ()
    plan.run_dump(x, buf[offset:offset + size], 3, *args, n_dumps=n_dumps)
    torch.cuda.synchronize()
    assert plan.check_device() == 0
    full = buf.cpu().numpy()
    got = full[offset:offset + size].astype(np.float64).reshape(n_dumps, c, -1, 2)
    for k in range(n_dumps):
        ref = odump.dump_corrected(oracle.xcorr_int(dumps[k], n, c, t, bits), 3, tau, nu)
        err = np.hypot(*(got[k] - ref).transpose(2, 0, 1))
        assert np.all(err <= 8 * 2.0 ** -24 * np.hypot(ref[..., 0], ref[..., 1]) + 1e-30)
    assert np.isnan(full[:offset]).all() and np.isnan(full[offset + size:]).all()
    plan.close()


# single blocks, pairs on and off the diagonal, repacked odd rows; each element is one rounded addition
@pytest.mark.parametrize("n,c,t,n_dumps", [
    (2, 700, 64, 1), (16, 620, 130, 1), (30, 311, 64, 2), (62, 5, 70, 1), (66, 3, 64, 2), (98, 90, 200, 2), (128, 160, 130, 1), (192, 3, 65, 2),
    (254, 2, 400, 1), (320, 80, 200, 1), (9, 513, 65, 2), (31, 640, 64, 1), (63, 40, 200, 1), (65, 80, 300, 2), (127, 100, 512, 1), (255, 60, 100, 1)])
def test_float_sums_add_to_what_is_there(n, c, t, n_dumps):
    rng = np.random.default_rng(n + c + t)
    x = rng.normal(size=(n_dumps, t, c, n, 2)).astype(np.float32)
    init = (rng.normal(size=(n_dumps, c, n * (n + 1) // 2, 2)) * t).astype(np.float32)
    v = run_engine(x, n, c, t, 32, 2, n_dumps=n_dumps, accumulate=True, vis_init=init)
    one = run_engine(x, n, c, t, 32, 2, n_dumps=n_dumps)
    assert np.array_equal(v, init + one)
    chans = sorted({0, c // 2, c - 1})
    check_bf16x3(one[0][chans], x[0], n, c, t, chans)
