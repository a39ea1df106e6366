"""The reciprocals of the reduced eigensolver (csrc/recip.cuh) against long double over the whole
range they are used on, next to the division and 1 / sqrt(x) of the compiler.

Bars: one rounding of the last step, half a unit, and what the earlier steps leave (2^-40 of a
unit) for 1 / x; half a unit more for the rounded product in 1 / sqrt(x)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reciprocals_over_their_range(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "recip_check")
    src = os.path.join(ROOT, "tests", "device", "recip_check.cu")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", src, "-o", exe],
                   check=True, capture_output=True, timeout=300)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    rcp, div, rsqrt, root = (float(v) for v in out.split())
    assert rcp <= 0.501, out
    assert rsqrt <= 1.01, out
    assert div <= 0.501 and root <= 1.51, out   # the compiler's, in the same measure
