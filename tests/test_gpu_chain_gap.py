"""Meshes small enough to be tried for one cluster that its shared memory does not
hold: their elliptic solves follow the rule of the kernel chains like larger
meshes', and give the persistent form's fields."""
import pytest

from gpu_util import gpu_sim, rel, rest_X
from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# mesh, precision, whether the single solves become chains (the pairs do in all)
CASES = [((26, 26, 8), binding.FP64, True), ((20, 20, 16), binding.FP64, True), ((30, 30, 8), binding.FP64, True),
         ((31, 31, 8), binding.MIXED, True), ((36, 36, 9), binding.MIXED, True), ((118,), binding.FP64, False)]


@pytest.mark.parametrize("n,prec,one", CASES)
def test_gap_meshes_take_the_chains(n, prec, one):
    w = W.config2(*n) if len(n) == 3 else W.sheet(n[0], n[0] / 128.0, W.LR91, 0.02, 1)
    # tolerances of tests/test_gpu_chain.py
    opt = dict(precision=prec, cg_tol_e=1e-11)
    if prec == binding.FP64:
        opt["cg_tol_p"] = 1e-13
    for M, K in ((3, 2), (2, 1)):
        out = []
        for streaming in (0, -1):
            sim = gpu_sim(w, streaming=streaming, **opt)
            sim.set_initial(rest_X(w))
            for _ in range(2):
                sim.step(w.dt, M, K)
            out.append((sim.fields(full=True), sim.stats()))
            sim.close()
        ((_, ua, Xa), sa), ((_, ub, Xb), sb) = out
        # chains are counted launch by launch
        assert (sa["kernel_launches"] > sb["kernel_launches"]) == (one or M == 3)
        tol = 1e-8 if prec == binding.FP64 else 5e-6
        assert rel(Xa, Xb) < tol and rel(ua, ub) < tol
