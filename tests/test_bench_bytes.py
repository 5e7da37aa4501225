"""The byte model of the benchmark's rooflines counts what the kernels move: binning writes keys only, and the
first radix pass reads no values."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("passes,key_bytes,sort", [(4, 4, 60), (5, 8, 116), (1, 4, 12)])
def test_bytes_per_point(passes, key_bytes, sort):
    assert bench.stage_bytes("bin", 1000, 3, 10, 5, passes, key_bytes) == 1000 * (12 + key_bytes)
    assert bench.stage_bytes("sort", 1000, 3, 10, 5, passes, key_bytes) == 1000 * sort
    line = bench.sort_roofline({"key_bits": 8 * key_bytes, "sort_passes": passes}, {"sort": 1.0}, 1000, 100.0, "test", None)
    assert line["algorithmic_bytes"] * passes == pytest.approx(1000 * sort)
