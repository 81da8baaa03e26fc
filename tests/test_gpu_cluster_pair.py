"""pair_solve = -1 on handles whose solves are cluster-resident: the two elliptic
solves of a later sweep are launches of their own, with the same bits."""
import numpy as np
import pytest

from gpu_util import gpu_sim
from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _mesh(kind):
    if kind == "bath":
        return W.bath_sheet(48, -0.25, 1.25, 0.0, 1.0, W.LR91, 0.02, 4, strip=0.1, s1_amp=80.0, s1_dur=1.0)
    return W.sheet(49, 1.0, W.LR91, 0.02, 4, strip=0.06)


@pytest.mark.parametrize("kind", ["sheet", "bath"])
@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED])
def test_one_solve_after_the_other(kind, prec):
    w = _mesh(kind)
    out = []
    for pair in (0, -1):
        sim = gpu_sim(w, precision=prec, pair_solve=pair)
        for _ in range(2):
            sim.step(w.dt, 3, 3)
        out.append((sim.fields(full=True), sim.stats()))
        sim.close()
    (a, sa), (b, sb) = out
    assert sb["kernel_launches"] == sa["kernel_launches"] + 2 * 2   # two later sweeps a step
    assert sa["cg_solves_e"] == sb["cg_solves_e"]
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED])
def test_one_solve_after_the_other_in_a_batch(prec):
    w = _mesh("sheet")
    out = []
    for pair in (0, -1):
        sims = [gpu_sim(w, precision=prec, pair_solve=pair) for _ in range(2)]
        for _ in range(2):
            binding.batch_step(sims, w.dt, 3, 2)
        out.append(([f for sim in sims for f in sim.fields(full=True)], sum(sim.stats()["kernel_launches"] for sim in sims)))
        for sim in sims:
            sim.close()
    assert out[1][1] == out[0][1] + 2        # a launch more a step
    for x, y in zip(out[0][0], out[1][0]):
        assert np.array_equal(x, y)
