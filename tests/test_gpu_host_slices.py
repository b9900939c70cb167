"""cwt_execute_host where outputs in pinned memory go through the staging buffers,
slices of channels at a time: bit for bit the device path's results, for plans
with whole rows, classes and two-kernel classes, channel counts that no slice
divides, outputs of which some are pageable, and new inputs on the same plan."""
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


# channels, samples, scales, outputs, those of them in pageable memory, options
CASES = [
    (11, 10000, 100, ("complex", "power"), (), dict(pad="smooth")),           # whole rows and classes, 132 MB
    (11, 10000, 100, ("complex", "power"), ("complex",), dict(pad="smooth")),
    (7, 30000, 64, ("power", "phase"), (), dict()),                           # two-kernel classes, 107 MB
    (3, 9001, 64, ("power",), (), dict()),                                    # 7 MB: one channel and two
    (1, 60000, 40, ("power",), (), dict(pad="smooth")),                       # one slice
    (5, 40000, 48, ("power",), (), dict(precision="tc_fp16", decimation=2)),
    (130, 1000, 40, ("complex", "power", "phase"), ("phase",), dict()),       # many channels per slice
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_sliced_outputs_equal_the_device_path(lib, case):
    import torch
    C, n, S, outs, pageable, kw = CASES[case]
    t = lib.CWT(C, n, 1000.0, np.geomspace(max(1.0, 3000.0 / n), 100, S), np.linspace(3, 10, S), outputs=outs, **kw)
    try:
        host = {k: torch.empty_like(v, device="cpu") for k, v in t.alloc_outputs().items()}
        host = {k: v if k in pageable else v.pin_memory() for k, v in host.items()}
        for turn in range(2):
            x = torch.from_numpy(eeg(2900 + 2 * case + turn, C, n, 1000.0, np.float32)).pin_memory()
            for v in host.values():
                v.fill_(float("nan"))
            lib.cwt_execute_host(t.plan, x, host.get("complex"), host.get("power"), host.get("phase"))
            ref = t(x.cuda())
            torch.cuda.synchronize()
            for k in outs:
                assert torch.equal(host[k], ref[k].cpu()), (k, turn)
    finally:
        t.close()
