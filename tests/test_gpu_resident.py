"""Cluster-resident solves against the grid-wide kernels (solver_tier = 1
forces those) on the same handle options, at sizes where the split over the
cluster changes shape: a mesh of less than one slice, blocks that own nothing,
one, two and three rows per thread, rows longer than the entries held in
registers, a bath (inactive rows of the parabolic solves), and the sizes next to
what the shared memory holds."""
import numpy as np
import pytest

from gpu_util import gpu_sim, rel
from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _workload(kind, n):
    if kind == "bath":
        return W.bath_sheet(n - 1, -0.25, 1.25, 0.0, 1.0, W.LR91, 0.02, 4, strip=0.1, s1_amp=80.0, s1_dur=1.0)
    if kind == "slab":
        w = W.config2(n, n, 8)
        w.dt = 0.02
        return w
    return W.sheet(n, 0.02 * (n - 1), W.LR91, 0.02, 4, strip=0.06)


CASES = [("sheet", 5), ("sheet", 23), ("sheet", 33), ("sheet", 90), ("sheet", 91), ("sheet", 115), ("sheet", 129),
         ("sheet", 150), ("bath", 49), ("slab", 17), ("slab", 31)]


@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED])
@pytest.mark.parametrize("kind,n", CASES)
def test_same_step_as_the_grid_kernels(kind, n, prec, precond):
    # both solve to the same tolerances: FP64 states agree like two solver forms
    # (1e-10, u 1e-9), mixed ones to the FP32 membrane model and increments
    w = _workload(kind, n)
    out = []
    for tier in (0, 1):
        sim = gpu_sim(w, precision=prec, solver_tier=tier, elliptic_precond=precond, cg_tol_e=1e-11, cg_tol_p=1e-11,
                      pin_node=w.pin_node if kind == "bath" else -1)
        for _ in range(3):
            sim.step(w.dt, 3, 2)
        out.append(sim.fields(full=True) + (sim.stats(),))
        sim.close()
    (v0, u0, X0, s0), (v1, u1, X1, s1) = out
    assert s0["cg_solves_e"] == s1["cg_solves_e"] and s0["cg_solves_p"] == s1["cg_solves_p"]
    tol_x, tol_u = (1e-10, 1e-9) if prec == binding.FP64 else (2e-6, 2e-6)
    assert rel(X0, X1) < tol_x and rel(u0, u1) < tol_u, (rel(X0, X1), rel(u0, u1))


@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED])
def test_decoupled_and_sweep_test_paths(prec):
    """CN-RK2 (a parabolic solve without node terms and warm start) and a closed
    sweep gate (the solve returns at once)."""
    w = W.sheet(41, 0.8, W.LR91, 0.02, 4, strip=0.06)
    got = []
    for tier in (0, 1):
        a = gpu_sim(w, precision=prec, solver_tier=tier, sweep_tol=10.0)
        b = gpu_sim(w, precision=prec, solver_tier=tier)
        for _ in range(3):
            a.step(w.dt, 3, 3)
            b.step_decoupled(0.002)
        got.append((a.fields(full=True)[2], b.fields(full=True)[2], a.stats()["cg_solves_e"]))
        a.close()
        b.close()
    tol = 1e-10 if prec == binding.FP64 else 2e-6
    assert rel(got[0][0], got[1][0]) < tol and rel(got[0][1], got[1][1]) < tol
    assert got[0][2] == got[1][2]


def test_iteration_cap_and_zero_right_hand_side():
    w = W.sheet(33, 1.0, W.LR91, 0.02, 1)
    sim = gpu_sim(w, cg_cap_e=2, cg_tol_e=1e-12)
    v = np.random.default_rng(1).uniform(-80, 20, w.n_nodes)
    with pytest.raises(binding.BdError) as e:
        sim.solve_elliptic(v)
    assert e.value.code == -4
    sim.close()
    sim = gpu_sim(w)
    u, it = sim.solve_elliptic(np.zeros(w.n_nodes))
    assert it == 0 and not np.any(u)
    sim.close()


@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED])
def test_batch_of_clusters_and_chains(prec):
    """Members of two cluster shapes and one that does not fit a cluster, in one
    captured step: each gives the bits of a batch of its own."""
    ws = [W.sheet(n, 0.02 * (n - 1), W.LR91, 0.02, 4, strip=0.06) for n in (33, 65, 129, 161)]

    def run(group):
        sims = [gpu_sim(w, precision=prec) for w in group]
        for _ in range(2):
            binding.batch_step(sims, 0.02, 3, 2)
        out = [sim.fields(full=True) for sim in sims]
        for sim in sims:
            sim.close()
        return out

    for w, f in zip(ws, run(ws)):
        for a, b in zip(f, run([w])[0]):
            assert np.array_equal(a, b)
