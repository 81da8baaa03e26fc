"""A cluster solve one of whose blocks waits for a message that nobody sends ends
with BD_ERR_TIMEOUT after its bound, and the handle's results are those of one that
never met it."""
import time

import numpy as np
import pytest

from gpu_util import gpu_sim
from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec", [(9, binding.FP64), (65, binding.FP64), (9, binding.MIXED), (65, binding.MIXED)])
def test_cluster_wait_is_bounded(n, prec):
    w = W.sheet(n, 0.02 * (n - 1), W.LR91, 0.02, 3, strip=0.05)
    sims = [gpu_sim(w, precision=prec) for _ in range(2)]
    for sim in sims:
        sim.step(w.dt, 3, 2)
        sim.sync()
    t0 = time.perf_counter()
    rc = binding.lib().bd_selftest_wait_timeout(sims[0].h)
    el = time.perf_counter() - t0
    assert rc == -7 and 3.0 < el < 30.0, (rc, el)   # the device barrier's bound and the cluster's
    out = []
    for sim in sims:
        for _ in range(2):
            sim.step(w.dt, 3, 2)
        sim.sync()
        out.append(sim.fields(full=True) + (sim.stats()["cg_solves_e"],))
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
