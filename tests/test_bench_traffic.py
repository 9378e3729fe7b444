"""bench.py states measured DRAM traffic only for the kernel that ran: the figures are keyed by
layout and name the profile that holds them."""
import os

import pytest

import bench


@pytest.mark.parametrize("table", [bench.SMOOTHER_TRAFFIC, bench.SPMV_TRAFFIC])
def test_traffic_is_of_the_layout_that_ran(table, monkeypatch):
    monkeypatch.setattr(bench, "WORKLOAD", bench.P4)
    for code in (0, -1, 4, 8, 16, 104, 408, -4):  # row layouts: captured for kernels of their own
        assert bench.measured_traffic(table, code) == {"traffic": None, "traffic_note": None}
    for (name, n, layout), (got, note) in table.items():
        assert layout.startswith("interleaved slices")
        assert got > 0
        profile = os.path.join(os.path.dirname(bench.__file__), note.split()[-1])
        assert layout in " ".join(open(profile).read().split())
