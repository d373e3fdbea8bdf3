"""FP64 forms on integers: a signal far below the other values of its variable keeps its relative accuracy, and a
uniform flow has no time modes."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_small_signals_against_long_double(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "small_signals")
    subprocess.run([nvcc, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    os.path.join(HERE, "small_signals.cu"), "-o", exe], check=True, capture_output=True, timeout=900)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=600).stdout.splitlines()
    assert len(lines) == 14
    for text in lines:
        name, value, bound = text.split()
        assert float(value) <= float(bound), text
