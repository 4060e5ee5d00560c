"""The FP64 roofline's denominator: the pipe's own rate where the probe's chains stay below it, so
that the product kernel's fraction is one of what the unit can do."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_fp64_peak_is_the_pipes_rate():
    peak, source = bench.fp64_peak(1.10075e12, 152, 2070.0)
    assert peak == pytest.approx(152 * 2 * 2 * 2.07e9) and "152 SMs" in source
    assert 1.133e12 / peak < 1.0  # the product kernel's rate, above the probe's


@pytest.mark.parametrize("mhz", [None, 0.0, 1000.0])
def test_fp64_peak_falls_back_to_the_probe(mhz):
    """Without a clock record, or when the probe ran faster than the record allows."""
    peak, source = bench.fp64_peak(1.1e12, 152, mhz)
    assert peak == 1.1e12 and "probe" in source
