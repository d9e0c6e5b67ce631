"""The benchmark's rooflines count what runs on the unit that they are divided
by: a recorded run of the default arithmetic (132 x 132 cells, p = 6) stays below
the measured rates."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("p", [3, 4, 5, 6, 7, 8])
def test_fp64_part_of_the_local_factor(p):
    assert 0.3 * bench.factor_flops(p) < bench.factor_fp64_flops(p) < 0.51 * bench.factor_flops(p)


def test_fractions_of_a_recorded_run_are_fractions():
    assert bench.factor_fp64_flops(6) * 17424 / 9.6e-3 < 1054e9   # the FP64 rate of that run
    ph = [3.0, 7.9, 9.6, 7.2, 13.1, 0.24, 0.05, 40.7]
    assert bench.assembly_report(ph, 17424, 6, 60, "fp64")["frac"] < 1
