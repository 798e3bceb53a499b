"""Which feed the tensor-core X stage takes where it has the choice (int_planes_faster, float_planes_faster), on
the CPU: planes for few items of long dumps, the conversion in the kernel where the chip is full or the dump short.
Both give the same bits, which the GPU part checks on either side of the line."""
import ctypes

import numpy as np
import pytest

from paper_0906_1887_gb300 import build as corr_build


class Plan(ctypes.Structure):   # the head of csrc/corr_internal.h's Plan
    _fields_ = [(f, ctypes.c_int) for f in ("n_inputs", "n_chan", "n_time", "sample_bits", "nb", "kp")] + [
        ("n_baselines", ctypes.c_int64), ("device", ctypes.c_int), ("n_sm", ctypes.c_int), ("d_status", ctypes.c_void_p)] + [
        (f, ctypes.c_int) for f in ("tc_op_stages", "tc_float_planes", "tc_operands", "tc_items")] + [("rest", ctypes.c_char * 256)]


@pytest.fixture(scope="module")
def rules():
    lib = ctypes.CDLL(corr_build.build())

    def rule(name, n, c, t, bits, dumps=1, acc=0):
        p = Plan(n, c, t, bits, (n + 63) // 64, (t + 63) // 64 * 64, n * (n + 1) // 2, 0, 152)
        f = lib[name]
        f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int], ctypes.c_bool
        return f(ctypes.byref(p), dumps, acc)
    return (lambda *a, **k: rule("_ZN4corr17int_planes_fasterERKNS_4PlanEii", *a, **k),
            lambda *a, **k: rule("_ZN4corr19float_planes_fasterERKNS_4PlanEii", *a, **k))


@pytest.mark.parametrize("n,c,t,acc,planes", [   # measured both ways
    (256, 1, 20000, 0, True), (256, 4, 60000, 0, True), (129, 1, 20000, 0, True), (9, 1, 20000, 1, True), (320, 16, 20000, 1, True),
    (512, 1, 60000, 1, True), (256, 16, 20000, 0, False), (75, 333, 777, 0, False), (512, 128, 2048, 0, False),
    (400, 613, 472, 1, False), (9, 256, 20000, 0, False), (256, 1, 1000, 0, False)])
def test_integer_feed(rules, n, c, t, acc, planes):
    assert rules[0](n, c, t, 8, acc=acc) == planes
    assert not rules[0](n, c, t, 4, acc=acc)


@pytest.mark.parametrize("n,c,t,acc,planes", [
    (128, 1, 4000, 0, True), (256, 4, 20000, 0, True), (512, 8, 4000, 0, True), (65, 1, 1000, 0, True), (33, 2, 20000, 0, True),
    (65, 256, 64, 1, True), (128, 16, 20000, 0, False), (64, 1, 64, 0, False), (256, 512, 512, 0, False), (1024, 64, 1024, 0, False),
    (80, 139, 1222, 0, False), (9, 512, 1000, 0, False), (255, 202, 506, 0, False), (128, 160, 130, 1, False)])
def test_float_feed(rules, n, c, t, acc, planes):
    assert rules[1](n, c, t, 32, acc=acc) == planes


def test_more_channels_never_bring_the_planes_back(rules):
    for n in (9, 33, 75, 128, 200, 256, 320, 512, 1024):
        for t in (64, 500, 2000, 20000):
            for k, bits in ((0, 8), (1, 32)):
                got = [rules[k](n, c, t, bits) for c in (300, 1000, 10000, 10 ** 6)]
                assert not any(got), (n, t, bits)


@pytest.mark.gpu
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n,c,t,bits", [(256, 2, 2100, 8), (129, 1, 2000, 8), (9, 8, 1600, 8), (75, 1, 1600, 8), (256, 1, 100, 8),
                                        (384, 2, 1000, 4), (128, 1, 2000, 32), (65, 2, 1000, 32), (66, 90, 64, 32), (31, 2, 4000, 32)])
def test_same_bits_either_way(n, c, t, bits, accumulate):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from _gpu_helpers import int_case, run_engine
    rng = np.random.default_rng(n + c + t)
    if bits == 32:
        x = rng.normal(size=(t, c, n, 2)).astype(np.float32)
        init = rng.normal(size=(1, c, n * (n + 1) // 2, 2)).astype(np.float32) * np.float32(t) if accumulate else None
        v = run_engine(x, n, c, t, 32, 2, accumulate=accumulate, vis_init=init)
        planes = run_engine(x, n, c, t, 32, 2, tuning=(0, 1))
        assert np.array_equal(v, init + planes if accumulate else planes)
        return
    x = int_case(n + c + t, n, c, t, bits)
    ref = oracle.xcorr_int(x, n, c, t, bits)
    init = rng.integers(-2 ** 40, 2 ** 40, size=(1,) + ref.shape) if accumulate else None
    for operands in ((0, 0), (2, 0)):
        v = run_engine(x, n, c, t, bits, 0, accumulate=accumulate, vis_init=init, operands=operands)[0]
        assert np.array_equal(v, ref + (init[0] if accumulate else 0))
