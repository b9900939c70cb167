"""Workspaces of residue classes where memory is short, by host-side failure
injection (CWT_FAULT_ALLOC_AT, csrc/alloc.cu): the two-kernel form's and a batch's
workspace are only as large as they can be, and the values are the same bits.  What
a plan and its batches hold is in the plan's byte count."""
import os

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


def _first_that_works(lib, tag, call):
    """call() with its k-th allocation failing, for the first k at which it returns."""
    for k in range(1, 40):
        os.environ["CWT_FAULT_ALLOC_AT"] = f"{k}:{tag}"
        try:
            return call()
        except lib.CWTError as e:
            assert e.status == lib.CWT_ENOMEM
        finally:
            os.environ.pop("CWT_FAULT_ALLOC_AT", None)
    raise AssertionError("never")


@pytest.mark.parametrize("precision", ["fp32", "tc_bf16"])
def test_two_kernel_workspace_shrinks(lib, precision):
    import torch
    C, n, S = 6, 60000, 40

    def create():
        return lib.CWT(C, n, 1000.0, np.geomspace(2, 100, S), np.linspace(3, 10, S), precision=precision)
    whole = create()
    short = _first_that_works(lib, "wide-" + precision, create)
    try:
        assert lib.cwt_plan_routes(whole.plan)[2] > 0
        assert lib.cwt_plan_routes(short.plan) == lib.cwt_plan_routes(whole.plan)
        assert short.info.workspace_bytes < whole.info.workspace_bytes
        x = torch.from_numpy(eeg(3000, C, n, 1000.0, np.float32)).cuda()
        assert torch.equal(whole(x)["power"], short(x)["power"])
    finally:
        whole.close()
        short.close()


def test_batch_workspace_shrinks_and_is_counted(lib):
    import torch
    C, S, fs = 16, 20, 1000.0
    lengths = [900, 4000, 300, 8000, 2500, 700, 1500, 6000] * 4
    args = (C, 8000, fs, np.geomspace(4, 60, S), np.linspace(3, 8, S))
    ep, n_in, n_out = lib.pack_epochs(lengths, C, S)
    x = torch.randn(n_in, device="cuda")
    a, b = lib.CWT(*args), None
    try:
        ref, got = (torch.zeros(n_out, device="cuda") for _ in range(2))

        def fresh():  # a plan of its own each time: a failed call keeps the lengths that it made
            at = os.environ.pop("CWT_FAULT_ALLOC_AT")
            t = lib.CWT(*args)
            os.environ["CWT_FAULT_ALLOC_AT"] = at
            lib.cwt_execute_batch(t.plan, ep, x, power_out=got)
            return t

        before = lib.cwt_plan_workspace_bytes(a.plan)
        lib.cwt_execute_batch(a.plan, ep, x, power_out=ref)
        assert lib.cwt_plan_workspace_bytes(a.plan) >= before + lib.cwt_plan_batch_stats(a.plan).bank_bytes + n_in
        b = _first_that_works(lib, "ws", fresh)
        torch.cuda.synchronize()
        assert lib.cwt_plan_workspace_bytes(b.plan) < lib.cwt_plan_workspace_bytes(a.plan)
        assert lib.cwt_plan_batch_stats(b.plan).graph_launches > 1
        assert torch.equal(ref, got)
    finally:
        a.close()
        if b is not None:
            b.close()
