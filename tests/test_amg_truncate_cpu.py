"""The hierarchy planned for a cluster and cut back for the grid kernels is the
one that those build by themselves."""
import os
import shutil
import subprocess

import pytest

from paper_2510_27447_gb300 import build as B


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("amg") / "check")
    here = os.path.dirname(os.path.abspath(__file__))
    src = [os.path.join(here, "amg_truncate_check.cpp")] + [os.path.join(B.CSRC, f) for f in ("amg.cpp", "assemble.cpp")]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    subprocess.run([cxx, "-O2", "-std=c++20", "-I" + inc, *src, "-o", exe, "-pthread"], check=True)
    return exe


# levels dropped, none to drop, all but one dropped, coarsest sizes that no level has
@pytest.mark.parametrize("n,fine,coarse,levels", [(61, 20, 100, 2), (41, 384, 1500, 1), (61, 20, 20, 3), (61, 20, 1500, 1),
                                                  (30, 5, 899, 1)])
def test_cut_back(check, n, fine, coarse, levels):
    out = subprocess.run([check, str(n), str(fine), str(coarse)], check=True, capture_output=True, text=True).stdout.split()
    assert out[0] == "ok" and int(out[2]) == levels, out
