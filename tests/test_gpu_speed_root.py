"""FP64 root of wave speeds: within a rounding of the last place around powers of two and over both parities of the
exponent, and what zero, subnormal, negative, infinite and NaN arguments give."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_speed_root(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "speed_root")
    subprocess.run([nvcc, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    os.path.join(HERE, "speed_root.cu"), "-o", exe], check=True, capture_output=True, timeout=900)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.splitlines()
    assert len(lines) == 3
    for text in lines:
        name, value, bound = text.split()
        assert float(value) <= float(bound), text
