"""The whole-row kernels -- powers of two on one CTA and on clusters, smooth lengths
on every kernel family, plan-time compiled ones, and the tensor-core stages --
against the FP64 oracle, with every scale on them (cwt_options.whole_rows): by
default most scales of a float32 plan run by residue classes instead, so that
plans of the same shapes without the option test those.  cwt_plan_routes says
which ran.  The bounds are those of the tests of each precision."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)  # also run as a program, under the bounds-checked build

import oracle  # noqa: E402
from eeg_synth import eeg  # noqa: E402
from tests.metrics import FP32_TOL, TC_TOL, complex_err, phase_err, power_err  # noqa: E402

pytestmark = pytest.mark.gpu
ALL = ("complex", "power", "phase")


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_2506_07793_gb300 as p
    return p


def _run(lib, x, fs, freqs, cycles, **kw):
    """(outputs, plan info, routes) of one transform."""
    import torch
    t = lib.CWT(x.shape[0], x.shape[1], fs, freqs, cycles, outputs=kw.pop("outputs", ALL), **kw)
    try:
        out = t(torch.from_numpy(np.ascontiguousarray(x)).cuda())
        torch.cuda.synchronize()
        return {k: v.cpu().numpy() for k, v in out.items()}, t.info, lib.cwt_plan_routes(t.plan)
    finally:
        t.close()


def _worst(res, ref):
    f = {"complex": complex_err, "power": power_err, "phase": phase_err}
    return {k: float(f[k](v, ref).max()) for k, v in res.items()}


# samples, channels, fs, frequencies, cycles, decimation, padding
ROWS = [
    (30, 3, 100.0, [9.0, 30.0], [3.0, 7.0], 1, "pow2"),
    (700, 2, 500.0, [3.0, 40.0, 230.0], [5.0, 7.0, 12.0], 1, "pow2"),
    (3000, 2, 500.0, [3.0, 40.0, 230.0], [5.0, 7.0, 12.0], 4, "pow2"),      # spectral fold
    (12000, 2, 500.0, [1.0, 40.0, 230.0], [5.0, 7.0, 3.0], 1, "pow2"),      # 32 points per thread
    (20000, 1, 1000.0, [0.8, 13.0, 480.0], [3.0, 7.0, 3.0], 1, "pow2"),     # clusters of 2
    (40000, 1, 2000.0, [3.0, 600.0, 950.0], [7.0, 5.0, 3.0], 3, "pow2"),    # of 4
    (100000, 1, 2048.0, [0.5, 30.0, 900.0], [7.0, 7.0, 5.0], 8, "pow2"),    # of 8
    (1000, 3, 500.0, [3.0, 40.0, 200.0], [5.0, 7.0, 9.0], 1, "smooth"),     # compiled in
    (10000, 1, 1000.0, [1.0, 40.0, 400.0], [5.0, 7.0, 9.0], 2, "smooth"),
    (6400, 2, 1000.0, [1.0, 40.0, 400.0], [5.0, 7.0, 9.0], 1, "smooth"),    # an inlined radix pair
    (1323, 3, 500.0, [3.0, 40.0, 200.0], [5.0, 7.0, 9.0], 1, "smooth"),     # the generic schedule
    (16400, 1, 1000.0, [1.0, 40.0, 400.0], [5.0, 7.0, 9.0], 1, "smooth"),   # 2 x 8232
    (20000, 1, 1000.0, [1.0, 40.0, 400.0], [5.0, 7.0, 9.0], 1, "smooth"),   # 2 x 10000, compiled in
]


@pytest.mark.parametrize("case", range(len(ROWS)))
def test_fp32_whole_rows_match_the_oracle(lib, case):
    n, C, fs, freqs, cycles, d, pad = ROWS[case]
    x = eeg(2500 + case, C, n, fs, np.float32)
    res, info, routes = _run(lib, x, fs, freqs, cycles, decimation=d, pad=pad, whole_rows=True)
    assert routes == (len(freqs), 0, 0)
    ref = oracle.cwt(x.astype(np.float64), info.fft_length, fs, freqs, cycles, decimation=d)
    worst = _worst(res, ref)
    assert max(worst.values()) <= FP32_TOL, worst


def test_routes_add_up_and_the_option_turns_classes_off(lib):
    """The fused workload: the default plan runs most scales by residue classes, and
    both plans agree within twice the bar (each is within one of the truth)."""
    freqs, cycles = np.geomspace(1, 100, 100), np.linspace(3, 10, 100)
    x = eeg(2550, 2, 10000, 1000.0, np.float32)
    a, _, ra = _run(lib, x, 1000.0, freqs, cycles, outputs=("power",), pad="smooth")
    b, _, rb = _run(lib, x, 1000.0, freqs, cycles, outputs=("power",), pad="smooth", whole_rows=True)
    assert sum(ra) == 100 and ra[1] + ra[2] >= 50
    assert rb == (100, 0, 0)
    peak = b["power"].max(axis=-1, keepdims=True)
    assert (np.abs(a["power"] - b["power"]) / peak).max() <= 2 * FP32_TOL


# samples (N = 16384, 32768, 65536, 131072: 1, 2, 4 and 8 CTAs per row), channels
TC = [
    (12000, 3, 1000.0, [0.7, 4.0, 13.0, 60.0, 240.0, 480.0], [3.0, 7.0, 7.0, 5.0, 12.0, 3.0], 1),
    (20000, 2, 1000.0, [0.8, 13.0, 240.0], [3.0, 7.0, 12.0], 1),
    (40000, 1, 2000.0, [3.0, 600.0, 950.0], [7.0, 5.0, 3.0], 1),
    (122880, 1, 2048.0, [0.5, 20.0, 900.0], [7.0, 7.0, 4.0], 8),
]


@pytest.mark.parametrize("precision", ["tc_fp16", "tc_bf16"])
@pytest.mark.parametrize("case", range(len(TC)))
def test_tensor_core_rows_match_the_oracle(lib, case, precision):
    """At the bars of the tensor-core tests: 2e-3, and below 131072 points what hi/lo
    operands keep."""
    n, C, fs, freqs, cycles, d = TC[case]
    x = eeg(2600 + case, C, n, fs, np.float32)
    res, info, routes = _run(lib, x, fs, freqs, cycles, decimation=d, precision=precision, whole_rows=True)
    assert routes == (len(freqs), 0, 0) and info.fft_length == 16384 << case
    worst = _worst(res, oracle.cwt(x.astype(np.float64), info.fft_length, fs, freqs, cycles, decimation=d))
    assert max(worst.values()) <= TC_TOL, worst
    if info.fft_length < 131072:
        assert worst["power"] <= (5e-5 if precision == "tc_fp16" else 2e-4), worst


def test_tensor_core_rows_are_not_the_fp32_ones(lib):
    """The BF16 stages ran: their result differs from the FP32 rows' beyond FP32."""
    x = eeg(2650, 1, 16000, 1000.0, np.float32)
    a, _, _ = _run(lib, x, 1000.0, [5.0, 60.0], [7.0, 7.0], precision="tc_bf16", whole_rows=True)
    b, _, _ = _run(lib, x, 1000.0, [5.0, 60.0], [7.0, 7.0], whole_rows=True)
    assert np.abs(a["complex"] - b["complex"]).max() > 1e-6 * np.abs(b["complex"]).max()


# one CTA per row, clusters, and the widest splits that plan-time compilation opens
SPECIAL = [
    (42, 5, 100.0, [8.0, 30.0], [3.0, 5.0], 1, None),
    (6300, 2, 1000.0, [1.0, 30.0, 400.0], [3.0, 7.0, 12.0], 1, None),
    (11025, 2, 1000.0, [0.8, 50.0, 450.0], [4.0, 7.0, 11.0], 3, None),
    (14175, 2, 1000.0, [2.0, 40.0, 300.0], [5.0, 7.0, 10.0], 1, 3),
    (19683, 1, 2000.0, [1.5, 100.0, 800.0], [20.0, 7.0, 4.0], 4, 3),
]


@pytest.mark.parametrize("case", range(len(SPECIAL)))
def test_compiled_rows_equal_the_runtime_schedule(lib, case):
    n, C, fs, freqs, cycles, d, cl = SPECIAL[case]
    x = eeg(2700 + case, C, n, fs, np.float32)
    kw = dict(decimation=d, pad="smooth", whole_rows=True)
    plain, i0, r0 = _run(lib, x, fs, freqs, cycles, **kw)
    spec, i1, r1 = _run(lib, x, fs, freqs, cycles, specialize=1, **kw)
    assert r0 == r1 == (len(freqs), 0, 0)
    assert i0.specialized == 0 and i1.specialized == 1 and i1.fixed_kernel == 1
    assert cl is None or i0.cluster == i1.cluster == cl
    for k in plain:
        assert np.array_equal(plain[k], spec[k]), k
    worst = _worst(spec, oracle.cwt(x.astype(np.float64), n, fs, freqs, cycles, decimation=d))
    assert max(worst.values()) <= FP32_TOL, worst


@pytest.mark.parametrize("n,cl", [(105000, 10), (115200, 9), (14406, 7)])
def test_compiled_wide_splits_match_the_oracle(lib, n, cl):
    fs, freqs, cycles = 1000.0, [0.8, 60.0, 450.0], [7.0, 7.0, 12.0]
    d = 8 if n > 20000 else 1
    x = eeg(2750 + cl, 1, n, fs, np.float32)
    res, info, routes = _run(lib, x, fs, freqs, cycles, decimation=d, pad="smooth", specialize=1, whole_rows=True)
    assert routes == (3, 0, 0) and info.cluster == cl and info.specialized == 1
    worst = _worst(res, oracle.cwt(x.astype(np.float64), n, fs, freqs, cycles, decimation=d))
    assert max(worst.values()) <= FP32_TOL, worst


def test_whole_rows_run_clean_under_bounds_checks(lib):
    """The same kernel families in the bounds-checked build, in a process of its own."""
    import importlib.util
    spec = importlib.util.spec_from_file_location(
        "_cwt_build", os.path.join(ROOT, "paper_2506_07793_gb300", "build.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    env = dict(os.environ, CWT_GB300_LIB=b.build(check=True))
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], capture_output=True, text=True, env=env, cwd=ROOT,
                       timeout=600)
    assert r.returncode == 0 and "whole rows clean" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]


if __name__ == "__main__":
    import paper_2506_07793_gb300 as package
    for row in ROWS:
        n_, C_, fs_, f_, c_, d_, pad_ = row
        got = _run(package, eeg(1, C_, n_, fs_, np.float32), fs_, f_, c_, decimation=d_, pad=pad_, whole_rows=True)
        assert got[2] == (len(f_), 0, 0) and all(np.isfinite(v).all() for v in got[0].values())
    for row in TC:
        n_, C_, fs_, f_, c_, d_ = row
        for prec in ("tc_fp16", "tc_bf16"):
            _run(package, eeg(2, C_, n_, fs_, np.float32), fs_, f_, c_, decimation=d_, precision=prec, whole_rows=True)
    print("whole rows clean")
