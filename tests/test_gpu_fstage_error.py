"""Real spectra against float64: the kernels that transform real samples at half length and split the spectrum
have no more error than the transform of all points had on the same samples.  The figures are that one's relative
L2 errors, measured on these inputs, enough of them for the half-length kernels, with the full-length kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FULL_LENGTH = {   # (transform length, taps): relative L2 error
    (32, 2): 7.62121e-08, (32, 4): 8.01974e-08, (32, 8): 8.78386e-08, (64, 2): 8.23022e-08, (64, 4): 8.62521e-08,
    (64, 8): 9.33084e-08, (128, 2): 8.88388e-08, (128, 4): 9.23564e-08, (128, 8): 9.89069e-08, (256, 0): 8.2842e-08,
    (256, 2): 9.81838e-08, (256, 4): 1.01536e-07, (256, 8): 1.07544e-07, (512, 0): 9.11852e-08, (512, 2): 1.05381e-07,
    (512, 4): 1.08381e-07, (512, 8): 1.14114e-07, (1024, 0): 9.72464e-08, (1024, 2): 1.10501e-07,
    (1024, 4): 1.13496e-07, (1024, 8): 1.18858e-07, (2048, 0): 1.04366e-07, (2048, 2): 1.16925e-07,
    (2048, 4): 1.1972e-07, (2048, 8): 1.24801e-07, (4096, 0): 1.14318e-07}


@pytest.mark.parametrize("L,taps", sorted(FULL_LENGTH))
def test_real_spectra_no_less_exact_than_the_full_length_transform(L, taps):
    from paper_0906_1887_gb300 import corr
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert error(corr, L, taps) <= FULL_LENGTH[L, taps]


def error(corr, L, taps, n=128):
    frames = (1 << 23) // (n * L)
    nf = frames + max(0, taps - 1)
    x = np.clip(np.round(np.random.default_rng(L + taps).normal(0, 16, (nf * L, n))), -127, 127).astype(np.int8)
    k = np.arange(max(1, taps) * L)
    h = (np.sinc((k - (taps * L - 1) / 2) / L) * np.hamming(max(1, taps) * L)).astype(np.float32)
    fp = corr.FPlan(n, L // 2, corr.F_REAL8, taps, h if taps else None)
    x = torch.from_numpy(x).cuda()
    spec = fp.empty_spectra(frames)
    fp.run(x.view(torch.uint8).reshape(-1), spec, frames)
    torch.cuda.synchronize()
    fp.close()
    z = x.double().reshape(nf, L, n)
    if taps:
        w = torch.from_numpy(h.astype(np.float64)).cuda().reshape(taps, L, 1)
        z = sum(w[m] * z[m:m + frames] for m in range(taps))
    ref = torch.view_as_real(torch.fft.rfft(z, dim=1))
    return float((spec.double() - ref).norm() / ref.norm())
