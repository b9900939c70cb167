"""A batch of very many rows: 73728 channels of epochs of one sample each, padded to
4096 points for linear edges, 1024 scales; rows times residues of the class that
runs them pass 2^31.  Every output is the sample's square
times the wavelet's at its centre."""
import numpy as np
import pytest

from tests.metrics import FP32_TOL

pytestmark = pytest.mark.gpu


def test_seventy_five_million_short_rows():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_2506_07793_gb300 as lib
    C, E, S, fs = 8192, 9, 1024, 1000.0
    freqs, cycles = np.geomspace(15.0, 16.0, S), np.full(S, 40.0)  # support 2758 samples, bands of some 20 bins
    t = lib.CWT(C, 1, fs, freqs, cycles, outputs=("power",), edge="linear")
    try:
        assert t.info.fft_length == 4096
        epochs, n_in, n_out = lib.pack_epochs([1] * E, C, S)
        x = torch.linspace(0.5, 2.0, n_in, device="cuda")
        out = torch.full((n_out,), -1.0, device="cuda")
        lib.cwt_execute_batch(t.plan, epochs, x, power_out=out)
        one = torch.empty((C, S, 1), device="cuda")
        t(x[:C].clone(), out={"power": one})
        torch.cuda.synchronize()
        w2 = (one[:, :, 0] / x[:C, None].square()).double().mean(dim=0)  # per scale
        # two transforms, each within the bar of the truth
        for e in range(E):
            ref = x[e * C:(e + 1) * C, None].double().square() * w2
            got = out[e * C * S:(e + 1) * C * S].double().reshape(C, S)
            assert float(((got - ref).abs() / ref).max()) <= 2 * FP32_TOL
    finally:
        t.close()
