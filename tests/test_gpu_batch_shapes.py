"""The three work-item shapes a batch can be pinned to -- single tiles, wide items, pairs of CTAs -- each run
what they name, which the number of work items shows, and give the same bits."""
import numpy as np
import pytest

import oracle
from _gpu_helpers import int_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

JOBS = [(128, 5, 300, 8), (320, 3, 200, 8), (64, 9, 130, 8), (256, 4, 1100, 8), (192, 3, 260, 4), (256, 2, 400, 4)]


def _items(n, c, shape, planes):
    nb = (n + 63) // 64
    if nb == 1:
        return (c + 1) // 2           # pairs of channels
    ng = (nb + 1) // 2
    if shape == 2:
        return c * ng * (ng + 1) // 2
    if shape == 1 and planes:
        return c * ng * ((nb + 2) // 2)
    return c * nb * (nb + 1) // 2


@pytest.mark.parametrize("plane_min_nb", [0, 2, 4])
@pytest.mark.parametrize("shape", [0, 1, 2])
def test_pinned_shapes(shape, plane_min_nb):
    from paper_0906_1887_gb300 import corr
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    jobs, refs = [], []
    for k, (n, c, t, bits) in enumerate(JOBS):
        p = int_case(900 + k, n, c, t, bits)
        refs.append(oracle.xcorr_int(p, n, c, t, bits))
        x = torch.from_numpy(np.ascontiguousarray(p).view(np.uint8).reshape(-1).copy()).cuda()
        jobs.append((n, c, t, bits, x, torch.full((c, n * (n + 1) // 2, 2), -5, dtype=torch.int64, device="cuda")))
    b = corr.Batch(jobs, flags=corr.BATCH_PLANES)
    b.set_shape(0, 2, 0, plane_min_nb, shape, 1)
    info = b.info()
    want = sum(_items(n, c, shape, plane_min_nb and (n + 63) // 64 >= plane_min_nb) for n, c, _, _ in JOBS)
    assert info["n_items"] == want and info["wide"] == (shape == 1)
    b.run()
    torch.cuda.synchronize()
    assert b.check_device() == 0
    for j, ref in zip(jobs, refs):
        assert np.array_equal(j[5].cpu().numpy(), ref), j[:4]
    with pytest.raises(corr.CorrError):
        b.set_shape(0, 2, 0, plane_min_nb, 3, 1)
    b.close()
