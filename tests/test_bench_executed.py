"""The FP64 roofline's executed operations (no GPU): the kernels' own rate next to
that of the work an update stands for."""
import inspect
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("dim, ncell, step_s", [(1, 1 << 22, 1.505e-3), (2, 8192 ** 2, 48.4e-3),
                                                (3, 512 ** 3, 206e-3)])
def test_executed_is_what_the_pipe_can_do(dim, ncell, step_s):
    """A pipe busy for part of the time, with one operation in most of its slots."""
    r = bench.fp64_roofline(dim, ncell, step_s, 0.02, 1.2546)
    e = r["executed"]
    assert e["achieved"] == pytest.approx(e["flops_per_cell"] * ncell / step_s / 1e12)
    assert e["frac"] == pytest.approx(e["achieved"] / r["peak"])
    assert e["flops_per_cell"] < bench.FP64_FLOPS_PER_CELL[dim]
    assert 0.5 < e["frac"] < 0.86


def test_every_fp64_line_reports_it():
    """The lines of the benchmark that have an ALU roofline all take it from there."""
    assert inspect.getsource(bench).count('"bound": "alu"') == 1
