"""Bound of the grid barrier against the longest row one warp goes through alone
while the other blocks wait (csrc/common.cuh, spin_more)."""
from test_row_index_range import run_host_warp


def test_bound_covers_the_longest_row(tmp_path):
    r = run_host_warp("spin_limit", tmp_path)
    assert r.returncode == 0, r.stdout
