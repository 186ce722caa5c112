"""Index arithmetic of the column-walk iteration kernel, checked on the host.

A tap outside the staged box, a row of a TMA band the warp has not waited
for, or a pixel stored twice or never would be a fault or a race that parity
tests can miss, so the helper program goes through every phase's items for
every storage type, radius and tile edge.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2509_25924_gb300", "csrc")


def _run_check(tmp_path, name):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / name
    subprocess.check_call([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, "-gencode",
                           "arch=compute_103a,code=sm_103a", os.path.join(HERE, name + ".cu"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    return out.stdout.splitlines()


def test_walk_items_taps_and_bands(tmp_path):
    lines = _run_check(tmp_path, "walk_schedule_check")
    assert len(lines) == 3 * 20 + 1 and lines[-1] == "0 failing cases"


def test_window_sums_round_no_worse_than_the_block_form(tmp_path):
    # a sum of (2R+1)^2 products keeps the error of the block decomposition,
    # although its groups of eight outputs share a core of values
    lines = _run_check(tmp_path, "window_sum_check")
    assert len(lines) == 11 and lines[-1] == "0 failing radii"
