"""Every operand-ring depth that the tuning call takes runs on every route of the integer tensor-core engine
that has a workspace: planes ignore a depth of one, so the calls that may leave them for packed samples must
not be refused for it."""
import numpy as np
import pytest

import oracle
from _gpu_helpers import int_case, run_engine

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# plane or packed pairs (256 and 320 inputs, 4- and 8-bit), repacked rows (75, 130), packed channels (9)
@pytest.mark.parametrize("op_stages", [1, 2, 16])
@pytest.mark.parametrize("n,c,t,bits", [(256, 3, 200, 8), (320, 2, 130, 8), (256, 2, 140, 4), (192, 3, 130, 4), (75, 4, 130, 8),
                                        (130, 2, 100, 4), (9, 16, 70, 8)])
def test_every_ring_depth_runs(n, c, t, bits, op_stages):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x = int_case(n + c + t, n, c, t, bits)
    ref = oracle.xcorr_int(x, n, c, t, bits)
    init = np.random.default_rng(n).integers(-2 ** 40, 2 ** 40, size=(1,) + ref.shape)
    for acc in (False, True):
        v = run_engine(x, n, c, t, bits, 0, accumulate=acc, vis_init=init if acc else None, tuning=(op_stages, 0))[0]
        assert np.array_equal(v, ref + (init[0] if acc else 0))
