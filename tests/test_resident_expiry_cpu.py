"""Waits of the cluster-resident solves that run out, on a CPU model of the
blocks' warps (tests/resident_expiry_check.cpp): whichever warps expire and
whatever arrives afterwards, every warp leaves."""
import os
import shutil
import subprocess

import pytest


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("expiry") / "check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "resident_expiry_check.cpp")
    subprocess.run([cxx, "-O2", "-std=c++20", "-pthread", src, "-o", exe], check=True)

    def run(rule, script):
        out = subprocess.run([exe, rule, script], check=True, capture_output=True, text=True, timeout=60).stdout.split()
        return out[0], int(out[1]), int(out[2])
    return run


def test_nothing_late(model):
    assert model("order", "none") == ("done", 8, 0)


@pytest.mark.parametrize("script", ["lost", "between"])
def test_late_or_lost_message(model, script):
    state, finished, late = model("order", script)
    assert state == "done" and finished == 8 and late > 0


@pytest.mark.parametrize("seed", range(1, 9))
def test_random_losses(model, seed):
    assert model("order", f"random{seed}")[:2] == ("done", 8)


def test_the_model_sees_a_block_that_splits(model):
    assert model("alone", "between")[0] == "stuck"
