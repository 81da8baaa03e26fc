"""Plan of the cluster-resident solves (which block owns, reads and sends
what), checked on the CPU by a small program over the host code itself: index
ranges, one send per halo slot, and block-wise products against plain ones."""
import os
import shutil
import subprocess

import pytest

from paper_2510_27447_gb300 import build as B


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "check")
    here = os.path.dirname(os.path.abspath(__file__))
    src = [os.path.join(here, "resident_plan_check.cpp")]
    src += [os.path.join(B.CSRC, f) for f in ("resident_plan.cpp", "amg.cpp", "assemble.cpp")]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    subprocess.run([cxx, "-O2", "-std=c++20", "-I" + inc, *src, "-o", exe, "-pthread"], check=True)
    return exe


# a mesh smaller than one slice, one that leaves blocks empty, ragged sheets on
# both sides of a row per thread, the largest sheet, rows longer than the held
# eight entries; without and with several levels
@pytest.mark.parametrize("mesh", [(5, 4, 0), (23, 21, 0), (65, 65, 0), (91, 90, 0), (130, 127, 0), (9, 8, 7), (19, 23, 11)])
@pytest.mark.parametrize("coarse_max", [20, 384])
def test_plan_products_and_sends(checker, mesh, coarse_max):
    r = subprocess.run([checker, *map(str, mesh), str(coarse_max)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
