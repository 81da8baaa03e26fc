"""The integer exponential and reciprocal on the device: the exponential the bits
of the host's code (whose error tests/test_exp_cpu.py bounds), the reciprocal
those of the division."""
import os
import subprocess

import pytest

from paper_2510_27447_gb300 import build as B

pytestmark = pytest.mark.gpu


def test_device_bits(tmp_path):
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_math_check.cu")
    exe = str(tmp_path / "t")
    subprocess.run([B.nvcc(), src, "-o", exe, "-O3", "-std=c++20", B.ARCH, "-I" + B.CSRC], check=True)
    be, br, n = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert n > 0 and be == 0 and br == 0
