"""What a handle whose solves are cluster-resident reports: that they are (its
counts differ from those of the grid kernels, which cg_block asks for), the shapes of
the hierarchy that preconditions, and its bytes in the profile."""
import pytest

from gpu_util import gpu_sim
from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _step(w, **opt):
    sim = gpu_sim(w, **opt)
    sim.step(w.dt, 3, 2)
    sim.sync()
    st, levels = sim.stats(), sim.amg_levels()
    prof = sim.profile_steps(w.dt, 3, 2, 1)
    sim.close()
    return st, levels, prof


@pytest.mark.parametrize("n", [65, 91, 113])
@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED])
def test_cluster_hierarchy_is_the_reported_one(n, prec):
    w = W.sheet(n, 1.0, W.LR91, 0.02, 4)
    st, levels, prof = _step(w, precision=prec)
    grid, _, _ = _step(w, precision=prec, cg_block=512)
    assert len(levels) == st["amg_levels"] >= 1 and levels[0]["A"][0] == w.n_nodes
    for a, b in zip(levels, levels[1:]):
        assert a["R"][0] == b["A"][0] and a["P"][0] == a["A"][0]
    assert levels[-1]["R"][0] == st["amg_coarse_rows"] <= 384
    if prec == binding.FP64:     # both solves of the later sweep in one launch
        assert st["kernel_launches"] == grid["kernel_launches"] - 1
    assert prof["vcycle_bytes"] > 0 and prof["coarse_bytes"] > 0


@pytest.mark.parametrize("n,prec,amg", [(33, binding.MIXED, True), (19, binding.MIXED, False), (33, binding.FP64, False)])
def test_small_meshes_profile_the_preconditioner_they_use(n, prec, amg):
    w = W.sheet(n, 1.0, W.LR91, 0.02, 4)
    st, levels, prof = _step(w, precision=prec)
    assert st["amg_levels"] == 0 and levels == []
    assert (prof["vcycle_bytes"] > 0) == amg and (prof["coarse_bytes"] > 0) == amg
