"""FP64 zone formulas in integers (fixed.cuh): no sum of any predictor, face or fourth-order WENO formula leaves its 64
bits, for any signs of the entered values and the largest mantissas, and driven so the formulas agree with 80-bit
arithmetic."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_no_integer_sum_overflows(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "headroom")
    subprocess.run([nvcc, "-O0", "-Xcompiler", "-O0", "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", os.path.join(HERE, "headroom.cu"), "-o", exe], check=True,
                   capture_output=True, timeout=900)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=600).stdout.splitlines()
    assert len(lines) == 10 * 2 + 1
    for text in lines:
        name, value, bound = text.split()
        assert float(value) <= float(bound), text
