"""Scales run by output residue classes (csrc/zoom.cuh) against the FP64 oracle,
at the shapes where that path's indices meet their edges: one residue per row
and many, odd runs and odd row lengths (rows that start off a 32-byte sector),
column groups that meet several rows and the last partial one, windows that
wrap below bin 0, decimations that divide the padded length and that do not,
one- and two-stage first passes, and rows of several CTAs' worth of columns.
The bound is the FP32 bar of every transform (tests/metrics.py)."""
import numpy as np
import pytest

import oracle
from eeg_synth import eeg
from tests.metrics import FP32_TOL, complex_err, phase_err, power_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_2506_07793_gb300 as p
    return p


# samples, channels, fs, frequencies (Hz), n_cycles, outputs, decimation, pad
CASES = [
    (61, 3, 250.0, (12.0, 60.0), 7.0, ("power",), 1, "pow2"),
    (512, 5, 1000.0, (10.0, 35.0, 90.0), 7.0, ("complex", "power"), 1, "pow2"),
    (1009, 2, 1000.0, (2.0, 6.0, 25.0, 90.0, 300.0), 5.0, ("complex", "power"), 1, "pow2"),
    (1323, 3, 500.0, (1.5, 4.0, 20.0, 60.0), 6.0, ("complex", "power"), 1, "smooth"),
    (2187, 2, 500.0, (3.0, 11.0, 40.0), 7.0, ("power",), 1, "smooth"),
    (3001, 4, 1000.0, (2.0, 5.0, 15.0, 45.0, 120.0), 6.0, ("complex", "power", "phase"), 1, "smooth"),
    (4999, 2, 1000.0, (1.0, 3.0, 10.0, 30.0, 100.0), 5.0, ("complex",), 1, "smooth"),
    (6000, 3, 1000.0, (1.0, 3.0, 10.0, 30.0), 7.0, ("power",), 4, "smooth"),
    (7000, 2, 1000.0, (2.0, 8.0, 33.0), 7.0, ("power",), 3, "pow2"),
    (8190, 3, 1000.0, (2.0, 8.0, 33.0, 90.0), 7.0, ("complex", "power"), 5, "smooth"),
    (16000, 1, 1000.0, (1.0, 4.0, 16.0, 64.0), 3.0, ("complex", "power"), 1, "pow2"),
    (23000, 1, 1000.0, (1.0, 5.0, 25.0, 80.0), 6.0, ("complex", "power"), 1, "smooth"),
    (40001, 1, 2048.0, (1.0, 4.0, 16.0, 64.0, 190.0), 7.0, ("power",), 16, "pow2"),
    (70001, 1, 2048.0, (0.5, 2.0, 8.0, 32.0, 128.0), 7.0, ("power",), 1, "pow2"),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_residue_class_rows_match_the_oracle(lib, case):
    import torch
    n, C, fs, freqs, cyc, kinds, d, pad = CASES[case]
    freqs = np.array(freqs)
    cycles = np.full(len(freqs), cyc)
    x = eeg(2100 + case, C, n, fs, np.float32)
    t = lib.CWT(C, n, fs, freqs, cycles, outputs=kinds, decimation=d, pad=pad)
    try:
        out = t(torch.from_numpy(x).cuda())
        again = t(torch.from_numpy(x).cuda())
        torch.cuda.synchronize()
        rows = [(c, s) for c in range(C) for s in range(len(freqs))]
        if n > 20000:  # the oracle's direct sum: one channel's rows
            rows = rows[:len(freqs)]
        ref = oracle.cwt_rows(x.astype(np.float64), t.info.fft_length, fs, freqs, cycles, rows, decimation=d)
        for k in kinds:
            assert torch.equal(out[k], again[k])
            got = np.stack([out[k][c, s].cpu().numpy() for c, s in rows])
            err = {"complex": complex_err, "power": power_err, "phase": phase_err}[k](got, ref)
            assert err.max() <= FP32_TOL, (k, err)
    finally:
        t.close()


def test_gmw_window_and_output_guard(lib):
    """Generalized Morse scales, and nothing is written outside the outputs."""
    import torch
    C, n, fs, d = 3, 1500, 500.0, 2
    freqs, beta = np.array([4.0, 13.0, 40.0, 110.0]), np.array([17.5, 10.0, 17.5, 20.0])
    x = eeg(2200, C, n, fs, np.float32)
    t = lib.CWT(C, n, fs, freqs, beta, outputs=("power",), wavelet="gmw", decimation=d)
    try:
        no = t.info.n_out
        buf = torch.full((C * len(freqs) * no + 512,), -7.0, dtype=torch.float32, device="cuda")
        t(torch.from_numpy(x).cuda(), out={"power": buf[256:]})
        torch.cuda.synchronize()
        b = buf.cpu().numpy()
        assert (b[:256] == -7.0).all() and (b[-256:] == -7.0).all()
        ref = oracle.cwt(x.astype(np.float64), t.info.fft_length, fs, freqs, beta, wavelet="gmw", decimation=d)
        assert power_err(b[256:-256].reshape(C, len(freqs), no), ref).max() <= FP32_TOL
    finally:
        t.close()
