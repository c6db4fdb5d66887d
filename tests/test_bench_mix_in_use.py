"""The instruction mix that the headline's roofline takes: the packed kernel's, bound by the special-function
pipe at 1608 G/s and 2070 MHz (the entry under the headline's own key is the scalar kernel's, which no run reads)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_the_headline_reads_the_packed_kernels_mix():
    key = bench.MIX_OF.get("3d-vz-100k-256cube", "3d-vz-100k-256cube")
    assert key == "3d-vz-10k-256cube"
    pipe, peak, bounds = bench.pipe_roofline(bench.PIPE_MIX[key], 2070.0)
    assert pipe == "xu" and round(peak) == 1608
    assert peak == pytest.approx(152 * 16 * 2070e6 / bench.PIPE_MIX[key]["xu"] / 1e9)
    assert all(b >= peak for b in bounds.values())
