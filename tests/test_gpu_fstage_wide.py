"""GPU parity of the F-stage kernels for long transforms and short filterbanks (fengine_wide.cu).

Every length and kind that takes them, at the edges of their tiles: one input, inputs that are not
a multiple of the CTA's group or of the 4-input and 16-byte loads, frame counts around the batches
of 1, 2, 4 and more frames and around the runs of four, taps 2, 3, 4 (padded to 4), 5 and 8, and
samples that start off the vector alignment.  Bounds as in test_gpu_fstage.py: relative L2 error per
(frame, input) of 4 x 2^-24 log2 L, and 4 M x 2^-24 more for M taps, against complex128.
"""
import math

import numpy as np
import pytest

from oracle import fstage
from paper_0906_1887_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KIND_ID = {"c8": 0, "c4": 1, "r8": 2}
EPS = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_1887_gb300 import corr
    corr.lib()


def _samples(seed, n_samples, n_inputs, kind):
    lo, hi = (-8, 7) if kind == "c4" else (-128, 127)
    re, im = synth.uniform_ints(seed, n_samples, 1, n_inputs, lo, hi)
    if kind == "r8":
        return synth.pack_real8(re[:, 0, :])
    return synth.pack(re, im, 8 if kind == "c8" else 4)


def _run(packed, n_inputs, n_chan, n_frames, kind, n_taps=0, taps=None, offset=0):
    from paper_0906_1887_gb300 import corr
    fp = corr.FPlan(n_inputs, n_chan, KIND_ID[kind], n_taps=n_taps, taps=taps)
    raw = np.ascontiguousarray(packed).view(np.uint8).reshape(-1)
    dev = torch.zeros(raw.size + offset, dtype=torch.uint8, device="cuda")
    dev[offset:].copy_(torch.from_numpy(raw.copy()))
    guard = 64   # values past the spectra must stay as they are
    spec = torch.full((n_frames * fp.n_out_chan * n_inputs * 2 + guard,), float("nan"), device="cuda")
    fp.run(dev[offset:], spec, n_frames)
    torch.cuda.synchronize()
    out = spec.cpu().numpy()
    assert np.isnan(out[-guard:]).all()
    out = out[:-guard].reshape(n_frames, fp.n_out_chan, n_inputs, 2).astype(np.float64)
    fp.close()
    return out[..., 0] + 1j * out[..., 1]


def _check(got, ref, bound):
    err = np.linalg.norm(got - ref, axis=1)
    assert np.all(err <= bound * np.linalg.norm(ref, axis=1) + 1e-30), float(err.max())


@pytest.mark.parametrize("n_inputs,n_frames", [(1, 1), (5, 3), (16, 9), (36, 2)])
@pytest.mark.parametrize("kind,n_chan", [("c8", 512), ("c4", 512), ("c8", 1024), ("c8", 2048), ("c4", 4096),
                                         ("r8", 64), ("r8", 128), ("r8", 256), ("r8", 512), ("r8", 1024), ("r8", 2048)])
def test_long_transforms(kind, n_chan, n_inputs, n_frames):
    L = fstage.transform_length(n_chan, kind)
    p = _samples(n_chan + n_inputs, n_frames * L, n_inputs, kind)
    got = _run(p, n_inputs, n_chan, n_frames, kind)
    _check(got, fstage.fstage(p, n_inputs, n_chan, n_frames, kind), 4 * EPS * math.log2(L))
    if kind == "r8":   # DC and Nyquist of real samples are real
        assert not got[:, 0].imag.any() and not got[:, n_chan].imag.any()


@pytest.mark.parametrize("n_inputs,n_frames", [(3, 1), (12, 5), (33, 18)])
@pytest.mark.parametrize("n_taps", [2, 3, 4, 5, 8])
@pytest.mark.parametrize("kind,n_chan", [("c8", 32), ("c4", 64), ("c8", 128), ("c4", 256), ("c8", 512),
                                         ("r8", 16), ("r8", 32), ("r8", 64), ("r8", 128), ("r8", 256), ("r8", 512)])
def test_filterbank_window_in_registers(kind, n_chan, n_taps, n_inputs, n_frames):
    L = fstage.transform_length(n_chan, kind)
    p = _samples(7 * n_chan + n_inputs, (n_frames + n_taps - 1) * L, n_inputs, kind)
    taps = np.random.default_rng(n_chan + n_taps).normal(size=n_taps * L).astype(np.float32)
    got = _run(p, n_inputs, n_chan, n_frames, kind, n_taps, taps)
    ref = fstage.pfb(p, n_inputs, n_chan, n_frames, kind, taps.astype(np.float64))
    _check(got, ref, (4 * math.log2(L) + 4 * n_taps) * EPS)


@pytest.mark.parametrize("kind,n_chan,n_taps", [("c8", 512, 0), ("r8", 1024, 0), ("c8", 128, 8), ("r8", 64, 4)])
def test_samples_off_the_vector_alignment(kind, n_chan, n_taps):
    L = fstage.transform_length(n_chan, kind)
    n, f = 16, 6
    p = _samples(3 + n_chan, (f + max(0, n_taps - 1)) * L, n, kind)
    assert np.array_equal(_run(p, n, n_chan, f, kind, n_taps, offset=2), _run(p, n, n_chan, f, kind, n_taps))


# groups of inputs that are more than half of the chip, or more than all of it: several waves of runs
@pytest.mark.parametrize("kind,n_chan,n_taps,n_inputs,n_frames", [
    ("c4", 512, 4, 336, 29), ("c4", 512, 4, 1300, 9), ("r8", 512, 8, 700, 21), ("c8", 2048, 0, 680, 7)])
def test_runs_in_several_waves(kind, n_chan, n_taps, n_inputs, n_frames):
    L = fstage.transform_length(n_chan, kind)
    p = _samples(n_chan + n_inputs, (n_frames + max(0, n_taps - 1)) * L, n_inputs, kind)
    taps = np.random.default_rng(n_inputs).normal(size=n_taps * L).astype(np.float32) if n_taps else None
    got = _run(p, n_inputs, n_chan, n_frames, kind, n_taps, taps)
    ref = (fstage.pfb(p, n_inputs, n_chan, n_frames, kind, taps.astype(np.float64)) if n_taps else
           fstage.fstage(p, n_inputs, n_chan, n_frames, kind))
    _check(got, ref, (4 * math.log2(L) + 4 * n_taps) * EPS)


# CTAs with room for two inputs: a thread takes two points of each
@pytest.mark.parametrize("n_inputs,n_frames", [(1, 5), (3, 9), (34, 18)])
@pytest.mark.parametrize("n_taps", [2, 4, 5, 8])
@pytest.mark.parametrize("kind,n_chan", [("c8", 1024), ("c4", 1024), ("r8", 1024)])
def test_long_filterbank(kind, n_chan, n_taps, n_inputs, n_frames):
    L = fstage.transform_length(n_chan, kind)
    p = _samples(5 * n_chan + n_inputs, (n_frames + n_taps - 1) * L, n_inputs, kind)
    taps = np.random.default_rng(n_chan + n_taps).normal(size=n_taps * L).astype(np.float32)
    got = _run(p, n_inputs, n_chan, n_frames, kind, n_taps, taps)
    ref = fstage.pfb(p, n_inputs, n_chan, n_frames, kind, taps.astype(np.float64))
    _check(got, ref, (4 * math.log2(L) + 4 * n_taps) * EPS)
