"""The 64-bit fixed-point line transforms (csrc/fixed.cuh) on the host, every grid size: the
error against the direct sum in units of the last place, at the top of the number range.

Bar: a transform of length N has at most ceil(log2 N) levels, each rounding a value by at most
one unit in its product and half a unit in a halving, and each later level adds at most R values
(R <= 5) of modulus <= 1: the worst case is below 1.5 (1 + 5 + 25 + ...) units over the at most
four levels above the last; observed errors are 3 to 10 units (the constants carry 61 bits: up to
one unit more at the top of the range per product).  40 units keep 55 bits of 2^61."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_lines_match_the_direct_sum(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fixed_line_check")
    src = os.path.join(ROOT, "tests", "host", "fixed_line_check.cu")
    subprocess.run([nvcc, "-std=c++17", "-O2", src, "-o", exe], check=True, capture_output=True, timeout=600)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout
    rows = [line.split() for line in out.splitlines()]
    assert [int(r[1]) for r in rows] == [12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48]
    for r in rows:
        assert max(float(v) for v in r[2:5]) <= 40.0, r
        assert float(r[5]) <= 1.0, r
