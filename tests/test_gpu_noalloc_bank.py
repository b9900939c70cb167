"""The bank of cwt_execute_noalloc at scales whose wavelets are a few bins wide
(tens of thousands of cycles: a narrow spectral line), where the carrier lies
between two bins: both must be in it.  The expected coefficients are the closed
form of Eq. 3 on the bins, in 64 bits."""
import numpy as np
import pytest

from tests.metrics import FP32_TOL, complex_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_2506_07793_gb300 as p
    return p


@pytest.mark.parametrize("sigma", [300.0, 3e3, 2e4, 3e4, 4e4])
def test_carriers_between_two_bins(lib, sigma):
    import torch
    N, fs = 8192, 1000.0
    bins = np.array([1434.49, 1442.5, 1446.49, 1474.49, 1507.5, 1654.475, 1835.5, 2500.5])
    F = bins * fs / N
    x = np.random.default_rng(3).standard_normal(N).astype(np.float32)
    out = torch.empty((1, len(F), N), dtype=torch.complex64, device="cuda")
    lib.cwt_execute_noalloc(torch.from_numpy(x[None]).cuda(), 1, N, fs, F, np.full(len(F), sigma), complex_out=out)
    torch.cuda.synchronize()
    nu = np.arange(N) * fs / N
    W = np.exp(-0.5 * sigma ** 2 * (nu[None] / F[:, None] - 1.0) ** 2)  # kappa and aliases: below 1e-300 here
    W /= np.sqrt((W * W).sum(axis=1, keepdims=True) / N)
    ref = np.fft.ifft(np.fft.fft(x.astype(np.float64))[None] * W, axis=1)[None]
    err = complex_err(out.cpu().numpy(), ref)
    assert err.max() <= FP32_TOL, err
