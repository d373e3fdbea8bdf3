"""FP64 work done on integers (zone-scaled node states, WENO weights and sums): a host program over the kernels' own
headers compares it with 80-bit arithmetic, from uniform and non-finite data to the ends of the exponent range."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_integer_forms_against_long_double(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "integer_states")
    subprocess.run([nvcc, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", os.path.join(HERE, "integer_states.cu"), "-o", exe], check=True,
                   capture_output=True, timeout=900)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=600).stdout.splitlines()
    assert len(lines) == 5 * 2 * 3 + 8 + 5 * 3 * 2
    for text in lines:
        name, value, bound = text.split()
        assert float(value) <= float(bound), text
