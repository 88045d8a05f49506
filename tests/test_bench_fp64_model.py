"""The bench's work model of the FP64 step's kernels: line transforms per axis and products from slices, against the
closed forms of tests/test_bench_model.py.  Host logic only (CPU)."""
import math

import pytest

from tests.test_bench_model import _problem, bench  # noqa: F401


def test_line_transforms(bench):  # noqa: F811
    p = _problem(e=16)
    assert bench.kernel_work(p, "line_z_inverse", 1, 1) == bench.kernel_work(p, "zpass_inverse", 1, 1)
    fl, by = bench.kernel_work(p, "line_rows_inverse", 1, 4)
    assert fl == pytest.approx(4 * 5 * 49 * 128 * 128 * 7)
    assert by == pytest.approx(4 * (128 * 1908 + 49 * 128 * 128) * 16)
    fl, by = bench.kernel_work(p, "line_columns", 1, 1)
    assert fl == pytest.approx(2 * 5 * 128 * 128 * 128 * math.log2(128))
    assert by == pytest.approx(2 * 49 * 128 * 128 * 16 + 128 ** 3 * 8)


def test_sliced_products(bench):  # noqa: F811
    p = _problem(nb=64, e=16)
    fl, by = bench.kernel_work(p, "sl_mma", 5, 64)
    total = 8.0 * 62759 * (256 * 64 + 2 * 64 * 64) + 8.0 * 62759 * 64 * (256 + 64)
    assert 5 * fl == pytest.approx(total)
    vals = 62759 * (256 + 64 + 2 * 64 + 64) + (62759 + 64) * (256 + 64)
    assert 5 * by == pytest.approx(36 * vals)
    assert 9 * bench.kernel_work(p, "sl_slice", 9, 64)[1] == pytest.approx(52 * vals)
    roof = bench.roofline_of({"name": "sl_mma", "achieved_tflops": 20.0, "achieved_gbs": 1.0}, "fp64",
                             {"bf16_tflops": 1889.0, "hbm_gbs": 6778.3}, {})
    assert roof["bound"] == "tensor" and roof["split_passes"] == 45
