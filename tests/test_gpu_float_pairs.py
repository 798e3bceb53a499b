"""GPU parity of BF16x3 on float samples that the kernel splits: two 64-input blocks (CTA pairs) and odd rows, against
the hi/lo planes (the same splits and products in the same order: the same bits) and the float64 bound."""
import numpy as np
import pytest

from _gpu_helpers import check_bf16x3, run_engine

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BF16X3 = 2


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_1887_gb300 import corr
    corr.lib()


# ragged second blocks, odd baseline runs, dumps shorter than a stage and longer than the rings, more items
# than pairs, every ring depth the tuning can ask for
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n,c,t,n_dumps,op_stages", [
    (66, 1, 1, 1, 0), (66, 3, 64, 2, 0), (80, 5, 97, 1, 2), (98, 90, 200, 2, 0), (110, 2, 1000, 1, 1),
    (126, 4, 333, 3, 3), (128, 1, 65, 1, 0), (128, 160, 130, 1, 0), (128, 2, 2100, 1, 16)])
def test_float_pairs_match_planes(n, c, t, n_dumps, op_stages, accumulate):
    rng = np.random.default_rng(n + c + t)
    x = rng.normal(size=(n_dumps, t, c, n, 2)).astype(np.float32)
    init = np.zeros((n_dumps, c, n * (n + 1) // 2, 2), np.float32) if accumulate else None
    v = run_engine(x, n, c, t, 32, BF16X3, n_dumps=n_dumps, accumulate=accumulate, vis_init=init, tuning=(op_stages, 0))
    planes = run_engine(x, n, c, t, 32, BF16X3, n_dumps=n_dumps, tuning=(0, 1))
    assert np.array_equal(v, planes)
    chans = sorted({0, c // 2, c - 1})
    for d in range(n_dumps):
        check_bf16x3(v[d][chans], x[d], n, c, t, chans)


# odd counts: channels packed into tiles that start at 16-byte multiples (an even count of channels of at
# most 31 inputs), rows repacked one sample longer (the rest; accumulating dumps)
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n,c,t,n_dumps", [
    (1, 1, 1, 1), (1, 2, 70, 2), (7, 640, 64, 1), (9, 3, 65, 2), (31, 320, 130, 1), (31, 321, 64, 1), (33, 4, 100, 1),
    (41, 5, 318, 3), (63, 2, 64, 1), (65, 3, 65, 2), (75, 160, 130, 1), (127, 2, 1000, 1)])
def test_odd_float_rows_match_planes(n, c, t, n_dumps, accumulate):
    rng = np.random.default_rng(n + c + t)
    x = rng.normal(size=(n_dumps, t, c, n, 2)).astype(np.float32)
    init = np.zeros((n_dumps, c, n * (n + 1) // 2, 2), np.float32) if accumulate else None
    v = run_engine(x, n, c, t, 32, BF16X3, n_dumps=n_dumps, accumulate=accumulate, vis_init=init)
    planes = run_engine(x, n, c, t, 32, BF16X3, n_dumps=n_dumps, tuning=(0, 1))
    assert np.array_equal(v, planes)
    chans = sorted({0, c // 2, c - 1})
    for d in range(n_dumps):
        check_bf16x3(v[d][chans], x[d], n, c, t, chans)


# more than two blocks: squares off the diagonal, whose stages are two tiles; even and odd block counts
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n,c,t,n_dumps,op_stages", [
    (130, 1, 1, 1, 0), (192, 3, 65, 2, 2), (140, 90, 130, 1, 0), (254, 2, 400, 1, 16), (256, 80, 64, 1, 0),
    (129, 3, 100, 1, 0), (300, 2, 200, 2, 0), (513, 1, 130, 1, 0), (640, 2, 65, 1, 3)])
def test_float_squares_off_the_diagonal_match_planes(n, c, t, n_dumps, op_stages, accumulate):
    rng = np.random.default_rng(n + c + t)
    x = rng.normal(size=(n_dumps, t, c, n, 2)).astype(np.float32)
    init = np.zeros((n_dumps, c, n * (n + 1) // 2, 2), np.float32) if accumulate else None
    v = run_engine(x, n, c, t, 32, BF16X3, n_dumps=n_dumps, accumulate=accumulate, vis_init=init, tuning=(op_stages, 0))
    planes = run_engine(x, n, c, t, 32, BF16X3, n_dumps=n_dumps, tuning=(0, 1))
    assert np.array_equal(v, planes)
    check_bf16x3(v[0][:1], x[0], n, c, t, [0])
