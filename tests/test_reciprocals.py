"""Error bounds of the reciprocals by Newton steps (csrc/common.cuh): the last step's
rounding, 0.5 units in the last place, and for the square root that of its residual,
another half."""
from test_row_index_range import run_host_warp


def test_error_bounds(tmp_path):
    r = run_host_warp("reciprocals", tmp_path)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
