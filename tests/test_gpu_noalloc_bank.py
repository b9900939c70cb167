"""The bank of cwt_execute_noalloc at scales whose wavelets are a few bins wide
(tens of thousands of cycles: a narrow spectral line), where the carrier lies
between two bins: both must be in it.  The expected coefficients are the closed
form of Eq. 3 on the bins, in 64 bits.  And its refusal inside a capture."""
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


def test_first_call_inside_a_capture_is_refused_and_leaves_it_whole(tmp_path):
    """Before the scratch's tables exist, in a process of its own: the call returns
    CWT_ECUDA, the capture goes on, and later calls work."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    prog = tmp_path / "capture.py"
    prog.write_text('''
import sys
sys.path.insert(0, %r)
import numpy as np, torch
import paper_2506_07793_gb300 as lib
x = torch.randn(2, 500, device="cuda")
out = torch.zeros(2, 1, 500, device="cuda")
y = torch.zeros(4, device="cuda")
torch.cuda.synchronize()
st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
with torch.cuda.stream(st):
    g.capture_begin()
    y += 1.0
    try:
        lib.cwt_execute_noalloc(x, 2, 500, 250.0, [10.0], [7.0], power_out=out, stream=st)
        raise SystemExit("not refused")
    except lib.CWTError as e:
        assert e.status == lib.CWT_ECUDA, e.status
    g.capture_end()
g.replay()
torch.cuda.synchronize()
assert y.tolist() == [1.0] * 4
lib.cwt_execute_noalloc(x, 2, 500, 250.0, [10.0], [7.0], power_out=out)
torch.cuda.synchronize()
assert float(out.min()) >= 0.0 and float(out.max()) > 0.0
print("capture whole")
''' % root)
    r = subprocess.run([sys.executable, str(prog)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "capture whole" in r.stdout, r.stdout + r.stderr[-2000:]
