"""Batches whose scales all run by residue classes (csrc/batch_forward.cu): half-length forward FFTs at the edges of
every padded length, odd sample counts and offsets, a channel count that fills no CTA.  The tolerance is the library's
for float outputs (tests/metrics.py), which every other path meets."""
import numpy as np
import pytest

import oracle
from eeg_synth import eeg
from tests.metrics import FP32_TOL, power_err

pytestmark = pytest.mark.gpu

CASES = [
    # lengths, C, decimation, freqs, cycles at 500 Hz
    ([33, 64, 65, 127, 128, 255, 257, 511, 513, 1023, 1025, 2048, 2049, 4095, 4097, 8191, 8192], 3, 1, [40.0, 60.0],
     [5.0, 7.0]),
    ([8192, 8191, 5001, 4096, 3001, 2000, 1999, 700, 301, 257], 5, 4, [20.0, 30.0], [10.0, 15.0]),
    ([600, 600, 600], 33, 2, [12.0, 25.0, 40.0], [6.0, 9.0, 9.0]),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_batches_of_narrow_bands_match_the_oracle(case):
    import torch
    import paper_2506_07793_gb300 as lib
    lengths, C, d, freqs, cycles = CASES[case]
    fs, freqs, cycles = 500.0, np.array(freqs), np.array(cycles)
    o = lib.cwt_options_init()
    o.decimation = d
    plan = lib.cwt_plan_create(C, max(lengths), fs, freqs, cycles, 0, lib.CWT_OUT_POWER, o)
    try:
        ep, n_in, n_o = lib.pack_epochs(lengths, C, len(freqs), d)
        xs = [eeg(3300 + k, C, n, fs, np.float32) for k, n in enumerate(lengths)]
        x = torch.from_numpy(np.concatenate([a.reshape(-1) for a in xs])).cuda()
        pw = torch.full((n_o,), float("nan"), dtype=torch.float32, device="cuda")
        for _ in range(2):
            lib.cwt_execute_batch(plan, ep, x, None, pw, None)
        p = pw.cpu().numpy()
        for k, n in enumerate(lengths):
            n_out = -(-n // d)
            ref = oracle.cwt(xs[k].astype(np.float64), lib.cwt_fft_length(n), fs, freqs, cycles, decimation=d)
            got = p[ep[k].out_offset:ep[k].out_offset + C * len(freqs) * n_out].reshape(C, len(freqs), n_out)
            assert power_err(got, ref).max() <= FP32_TOL, n
    finally:
        lib.cwt_plan_destroy(plan)


def test_a_batch_inside_a_capture_is_refused():
    import torch
    import paper_2506_07793_gb300 as lib
    o = lib.cwt_options_init()
    o.decimation = 4
    plan = lib.cwt_plan_create(2, 1000, 500.0, np.array([20.0]), np.array([10.0]), 0, lib.CWT_OUT_POWER, o)
    try:
        ep, n_in, n_o = lib.pack_epochs([1000, 600], 2, 1, 4)
        x, p = torch.randn(n_in, device="cuda"), torch.zeros(n_o, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        lib.cwt_execute_batch(plan, ep, x, None, p, None, s.cuda_stream)  # a prepared shape
        torch.cuda.synchronize()
        want = p.clone()
        with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s):
            with pytest.raises(lib.CWTError):
                lib.cwt_execute_batch(plan, ep, x, None, p, None, s.cuda_stream)
        p.zero_()
        lib.cwt_execute_batch(plan, ep, x, None, p, None)
        assert torch.equal(p, want)
    finally:
        lib.cwt_plan_destroy(plan)
