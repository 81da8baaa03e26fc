"""The FP32 Jacobi scaling is the FP64 reciprocal rounded once (not the
reciprocal of a rounded diagonal), the FP64 one the division."""
import os
import shutil
import subprocess

import pytest

from paper_2510_27447_gb300 import build as B

SRC = r"""
#include "fixexp.h"
#include <cstdio>
#include <random>
int main() {
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> u(1.0, 2.0);
  long bad = 0, differs = 0;
  for (int i = 0; i < 500000; ++i) {
    const double d = std::ldexp(u(g), int(g() % 120) - 60);
    bad += bd::jacobi_scale<float>(d) != float(1.0 / d) || bd::jacobi_scale<double>(d) != 1.0 / d;
    differs += 1.0f / float(d) != float(1.0 / d);
  }
  std::printf("%ld %ld\n", bad, differs);
}
"""


def test_rounded_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++20", "-I" + B.CSRC, str(src), "-o", str(exe)], check=True)
    bad, differs = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0 and differs > 1000   # the inputs tell the two forms apart
