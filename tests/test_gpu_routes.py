"""Which transform each scale takes (cwt_plan_routes)."""
import numpy as np
import pytest

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


def test_most_scales_of_everyday_plans_run_by_classes(lib):
    whole, one, two = _routes(lib, 10000, 100, 1, 100, outputs=("complex", "power"), pad="smooth")
    assert one + two >= 70 and whole + one + two == 100
