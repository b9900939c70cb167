"""Which transform each scale takes (cwt_plan_routes), and that a channel's bits
depend neither on how many channels run beside it nor on the form that a launch
of few rows takes."""
import numpy as np
import pytest

from eeg_synth import eeg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_2506_07793_gb300 as p
    return p


def _routes(lib, n, S, lo, hi, **kw):
    t = lib.CWT(2, n, 1000.0, np.geomspace(lo, hi, S), np.linspace(3, 10, S), **kw)
    try:
        return lib.cwt_plan_routes(t.plan)
    finally:
        t.close()


def test_wide_bands_of_short_rows_stay_off_the_two_kernel_form(lib):
    """Bands of 40% of the row and more leave the first of the two kernels runs of
    one or two points (64 x 6300 x 60: 340 us, 270 as whole rows; 64 x 60000 x 40,
    every 8th sample: 236 and 128)."""
    assert _routes(lib, 6300, 60, 100, 400, outputs=("complex", "power"), pad="smooth")[2] == 0
    assert _routes(lib, 60000, 40, 2, 90, decimation=8)[2] == 0


def test_compiled_rows_take_the_scales_that_classes_run_slower(lib):
    """16 x 19683 x 60 with specialize: 127 us as compiled rows alone, 172 with the
    split of a plan that compiles none."""
    kw = dict(outputs=("complex", "power"), pad="smooth")
    plain, compiled = (_routes(lib, 19683, 60, 1, 200, specialize=s, **kw) for s in (0, 1))
    assert compiled[0] > plain[0] and compiled[2] < plain[2]
    # and leave those that classes run faster
    assert _routes(lib, 6300, 60, 2, 40, specialize=1, **kw)[1] >= 50


@pytest.mark.parametrize("n,lo,hi", [(6300, 2, 40), (6300, 2, 400), (16464, 1, 60)])
def test_tuning_runs_what_the_plan_runs(lib, n, lo, hi):
    """specialize = 2 times the forward FFTs and the scales left to whole rows, which
    may be none: no scratch for outputs that nothing writes, and the oracle's values."""
    import oracle
    import torch
    from tests.metrics import FP32_TOL, power_err
    S, C = 6, 3
    f, c = np.geomspace(lo, hi, S), np.linspace(3, 10, S)
    x = eeg(2790 + hi, C, n, 1000.0, np.float32)
    t = lib.CWT(C, n, 1000.0, f, c, pad="smooth", specialize=2)
    try:
        assert t.info.specialized in (0, 2) and t.info.fixed_kernel == 1
        out = t(torch.from_numpy(x).cuda())["power"].cpu().numpy()
        ref = oracle.cwt(x.astype(np.float64), t.info.fft_length, 1000.0, f, c)
        assert power_err(out, ref).max() <= FP32_TOL
    finally:
        t.close()


def test_most_scales_of_everyday_plans_run_by_classes(lib):
    whole, one, two = _routes(lib, 10000, 100, 1, 100, outputs=("complex", "power"), pad="smooth")
    assert one + two >= 70 and whole + one + two == 100


# samples, scales, outputs, decimation, padding: launches of few rows take another
# form than those of many (column groups that meet two, four and more rows, whole
# rows by one and by several per CTA)
SHAPES = [
    (4000, 100, ("complex", "power"), 1, "pow2"), (700, 40, ("power",), 1, "pow2"), (1500, 60, ("complex",), 2, "pow2"),
    (3000, 60, ("power",), 4, "smooth"), (2500, 60, ("power",), 1, "smooth"), (3001, 61, ("complex", "power"), 1, "smooth"),
    (8000, 60, ("power",), 3, "pow2"), (394, 40, ("power",), 1, "smooth"), (9000, 20, ("complex", "power"), 1, "smooth"),
]


@pytest.mark.parametrize("case", range(len(SHAPES)))
def test_bits_of_a_channel_do_not_depend_on_the_others(lib, case):
    import torch
    n, S, outs, d, pad = SHAPES[case]
    C, lo = 48, max(2.0, 3000.0 / n)
    x = torch.from_numpy(eeg(2800 + case, C, n, 1000.0, np.float32)).cuda()
    args = (1000.0, np.geomspace(lo, 90, S), np.linspace(3, 10, S))
    kw = dict(outputs=outs, decimation=d, pad=pad)
    whole = lib.CWT(C, n, *args, **kw)
    ref = whole(x)
    for c0, c1 in ((0, 1), (7, 9), (20, 28), (47, 48)):
        part = lib.CWT(c1 - c0, n, *args, **kw)
        out = part(x[c0:c1].clone())  # aligned
        torch.cuda.synchronize()
        for k in outs:
            assert torch.equal(out[k], ref[k][c0:c1]), (k, c0)
        part.close()
    whole.close()
