"""The benchmark names the kernels and the arithmetic that ran, from how many
scales took which form, not from the precision that was asked for."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("_bench", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


@pytest.mark.parametrize("precision,routes,label", [
    ("fp32", (20, 80, 0), "f32"),
    ("tc_fp16", (0, 100, 28), "f32"),
    ("tc_fp16", (128, 0, 0), "f16 hi/lo, f32 accumulation"),
    ("tc_bf16", (128, 0, 0), "bf16 hi/lo, f32 accumulation"),
    ("tc_bf16", (4, 60, 64), "f32; bf16 hi/lo, f32 accumulation on 4 of 128 scales"),
])
def test_arithmetic_label(bench, precision, routes, label):
    assert bench.arithmetic(precision, routes) == label


def test_kernel_label_names_only_what_ran(bench):
    assert "rows<16>" not in bench.scale_block_kernels("rows<16>", (0, 100, 28))
    assert bench.scale_block_kernels("rows<16>", (128, 0, 0)) == "scale blocks: 128 scales on rows<16>"
    assert "zoom" in bench.scale_block_kernels("rows<16>", (3, 5, 0)) and "wide" not in bench.scale_block_kernels("r", (3, 5, 0))
