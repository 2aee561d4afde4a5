"""Positions of CSR entries near the largest accepted nnz, 2^31 - 1: the row sums
of csrc/common.cuh, run on the CPU (tests/host_warp), load no entry outside the
matrix and sum every one of its own.  (-fwrapv: integers wrap as on the GPU.)"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_warp")


def run_host_warp(name, tmp_path):
    if not shutil.which("g++"):
        pytest.skip("g++ not found")
    exe = str(tmp_path / name)
    subprocess.run(["g++", "-std=c++20", "-O1", "-fwrapv", "-pthread", "-I", HERE, os.path.join(HERE, name + ".cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)
    return subprocess.run([exe], capture_output=True, text=True, timeout=300)


def test_last_rows_below_int_limit(tmp_path):
    r = run_host_warp("row_index_range", tmp_path)
    assert r.returncode == 0, r.stdout
