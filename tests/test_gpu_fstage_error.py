"""Real spectra against float64: the kernels that transform real samples at half length and split the spectrum
have no more error than the transform of all points had on the same samples.  The figures are that one's relative
L2 errors, measured on these inputs with the full-length kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FULL_LENGTH = {  # (transform length, taps): relative L2 error
    (32, 1): 7.471e-8, (32, 4): 8.015e-8, (32, 8): 8.817e-8, (64, 1): 7.910e-8, (64, 4): 8.610e-8, (64, 8): 9.345e-8,
    (128, 1): 8.633e-8, (128, 4): 9.228e-8, (128, 8): 9.896e-8, (256, 1): 9.606e-8, (256, 4): 1.014e-7, (256, 8): 1.078e-7,
    (512, 1): 1.032e-7, (512, 4): 1.084e-7, (512, 8): 1.142e-7, (1024, 1): 1.086e-7, (1024, 4): 1.131e-7, (1024, 8): 1.189e-7,
    (2048, 1): 1.151e-7, (2048, 4): 1.197e-7, (2048, 8): 1.246e-7,
    (256, 0): 8.257e-8, (512, 0): 9.128e-8, (1024, 0): 9.714e-8, (2048, 0): 1.045e-7, (4096, 0): 1.144e-7}


@pytest.mark.parametrize("L,taps", sorted(FULL_LENGTH))
def test_real_spectra_no_less_exact_than_the_full_length_transform(L, taps):
    from paper_0906_1887_gb300 import corr
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, frames = 16, max(16, (1 << 18) // (16 * L))
    nf = frames + max(0, taps - 1)
    x = np.clip(np.round(np.random.default_rng(L + taps).normal(0, 16, (nf * L, n))), -127, 127).astype(np.int8)
    k = np.arange(max(1, taps) * L)
    h = (np.sinc((k - (taps * L - 1) / 2) / L) * np.hamming(max(1, taps) * L)).astype(np.float32)
    fp = corr.FPlan(n, L // 2, corr.F_REAL8, taps, h if taps else None)
    spec = fp.empty_spectra(frames)
    fp.run(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), spec, frames)
    got = spec.cpu().numpy().astype(np.float64)
    fp.close()
    z = x.astype(np.float64).reshape(nf, L, n)
    if taps:
        w = h.astype(np.float64).reshape(taps, L, 1)
        z = sum(w[m] * z[m:m + frames] for m in range(taps))
    ref = np.fft.rfft(z, axis=1)
    err = np.linalg.norm(got[..., 0] + 1j * got[..., 1] - ref) / np.linalg.norm(ref)
    assert err <= FULL_LENGTH[L, taps]
