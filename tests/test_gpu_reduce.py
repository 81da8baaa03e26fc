"""FP64 block reductions of the persistent solvers at the block sizes where
their two stages change shape: fewer threads than the four adding warps, a
remainder of the strided stage, more than one round of it, the largest block."""
import numpy as np
import pytest

from gpu_util import gpu_sim, oracle_problem, rel
from paper_2510_27447_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("block", [32, 96, 128, 160, 544, 1024])
def test_fp64_solve_for_every_block_shape(block, precond):
    # tolerance as in the other solver tests: CG at 1e-12 against a direct solve
    w = W.sheet(47, 1.0, W.LR91, 0.02, 1)
    v = -80 + 100 * np.exp(-30 * ((w.xyz[:, 0] - 0.3) ** 2 + (w.xyz[:, 1] - 0.6) ** 2))
    for pin in (0, -1):
        ref = oracle_problem(w, pin=pin).elliptic(v)
        sim = gpu_sim(w, cg_block=block, elliptic_precond=precond, cg_tol_e=1e-12, pin_node=pin)
        u, it = sim.solve_elliptic(v)
        sim.close()
        assert it > 0 and rel(u, ref) < 1e-9, (it, rel(u, ref))
