"""Order of the messages of the cluster-resident solves on a CPU model with late
blocks and late messages (tests/resident_order_check.cpp): no block reads or
counts another phase's value, blocks that own nothing among them."""
import os
import shutil
import subprocess

import pytest


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("order") / "check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "resident_order_check.cpp")
    subprocess.run([cxx, "-O2", "-std=c++20", src, "-o", exe], check=True)
    return lambda *a: int(subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True).stdout)


@pytest.mark.parametrize("loop", ["jacobi", "pipelined", "amg"])
def test_dot_products_in_turn(model, loop):
    assert model(loop, "turns", 300) == 0


def test_the_model_sees_dot_products_that_share_a_buffer(model):
    assert model("jacobi", "single", 300) > 0
    assert model("pipelined", "single", 300) > 0
    assert model("amg", "single", 300) == 0   # the coarse gather lies between
