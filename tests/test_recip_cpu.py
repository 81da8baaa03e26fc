"""The integer reciprocal of the FP64 membrane kernels is the division's, bit for
bit, whatever its FP32 seed returns within the documented error."""
import os
import shutil
import subprocess

import pytest

from paper_2510_27447_gb300 import build as B


def test_reciprocal_is_correctly_rounded(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "recip_check.cpp")
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-O2", "-std=c++20", "-I" + B.CSRC, src, "-o", exe], check=True)
    bad, n = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert n > 1000000 and bad == 0
