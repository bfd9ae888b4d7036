"""The operator kernels and stored bytes that bench.py reports follow what the library
says its operators read, not the storage format alone."""
import pytest

import bench

NO = {"used": False, "degrid_bytes": 0, "grid_bytes": 0}
YES = {"used": True, "degrid_bytes": 700, "grid_bytes": 800}


@pytest.mark.parametrize("fmt,slices,want", [
    ("columns", YES, ("k_slice_degrid", "k_slice_grid", 700, 800)),
    ("runs", YES, ("k_slice_degrid", "k_slice_grid", 700, 800)),
    ("columns", NO, ("k_degrid", "k_grid_cells", 120, 120)),      # a short-row plan without slices
    ("runs", NO, ("k_runs_degrid", "k_runs_grid", 90, 95)),
    ("mask", NO, ("k_stream_degrid", "k_stream_grid", 95, 95)),
])
def test_operator_form(fmt, slices, want):
    assert bench.operator_form(fmt, slices, 10, 8, 90, 95) == want
