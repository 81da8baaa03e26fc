"""Elliptic solves of persistent handles as kernel chains inside captured steps
(the rule on size, precision and rows): the fields of the persistent form, on
meshes on both sides of the rule, eager steps left as they are, and steps taken
into a caller's own stream capture."""
import numpy as np
import pytest

from gpu_util import gpu_sim, rel, rest_X
from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _mesh(kind, *n):
    if kind == "slab":
        return W.config2(*n)
    if kind == "bath":
        return W.bath_sheet(n[0] - 1, -0.25, 1.25, 0.0, 1.0, W.LR91_PAPER_MOD, 0.02, 1, strip=0.1, s1_amp=80.0,
                            s1_dur=1.0)
    return W.sheet(n[0], n[0] / 128.0, W.LR91, 0.02, 1)


def _run(w, M, K, steps=2, **opt):
    sim = gpu_sim(w, **opt)
    sim.set_initial(rest_X(w))
    for _ in range(steps):
        sim.step(w.dt, M, K)
    f, st = sim.fields(full=True), sim.stats()
    sim.close()
    return f, st


# mesh, precision, whether single and two-system solves become chains
CASES = [(("slab", 31, 31, 8), binding.FP64, True, True), (("slab", 41, 37, 12), binding.MIXED, True, True),
         (("sheet", 281), binding.FP64, True, True), (("bath", 281), binding.FP64, True, True),
         (("sheet", 277), binding.FP64, False, True), (("sheet", 385), binding.MIXED, False, True),
         (("sheet", 375), binding.MIXED, False, False)]


@pytest.mark.parametrize("M,K", [(3, 2), (2, 1)])
@pytest.mark.parametrize("mesh,prec,one,two", CASES)
def test_chains_give_the_persistent_fields(mesh, prec, one, two, M, K):
    w = _mesh(*mesh)
    # FP64: residuals of 1e-11 leave u within 1e-8 (as in the other cross-form
    # tests; both forms break down on the bath mesh when asked for 1e-12);
    # mixed: FP32 increments, a few units of 6e-8 a solve
    opt = dict(precision=prec, cg_tol_e=1e-11)
    if prec == binding.FP64:
        opt["cg_tol_p"] = 1e-13
    (va, ua, Xa), sa = _run(w, M, K, **opt)
    (vb, ub, Xb), sb = _run(w, M, K, streaming=-1, **opt)
    assert sa["streaming"] == 0 and sa["amg_levels"] >= 1
    # chains are counted launch by launch
    chains = one or (two and M == 3)
    assert (sa["kernel_launches"] > sb["kernel_launches"]) == chains
    tol = 1e-8 if prec == binding.FP64 else 5e-6
    assert rel(Xa, Xb) < tol and rel(ua, ub) < tol
    if not chains:
        assert np.array_equal(ua, ub) and np.array_equal(Xa, Xb)


def test_a_chain_reports_and_leaves_what_the_persistent_kernel_does():
    """A solve stopped by its iteration cap: the same error, and u keeps the
    updates made until then."""
    w = _mesh("slab", 31, 31, 8)
    out = []
    for s in (0, -1):
        sim = gpu_sim(w, streaming=s, cg_cap_e=3)
        sim.set_initial(rest_X(w))
        sim.step(w.dt, 2, 1)
        with pytest.raises(binding.BdError) as e:
            sim.sync()
        sim.clear_status()
        out.append((e.value.code, sim.fields()[1]))
        sim.close()
    assert out[0][0] == out[1][0]
    assert np.any(out[1][1]) and rel(out[0][1], out[1][1]) < 1e-9


def test_eager_steps_keep_the_persistent_form():
    w = _mesh("slab", 31, 31, 8)
    out = [_run(w, 3, 2, use_graph=0, streaming=s) for s in (0, -1)]
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    assert out[0][1]["kernel_launches"] == out[1][1]["kernel_launches"]


def test_step_in_a_callers_capture():
    torch = pytest.importorskip("torch")
    w = _mesh("slab", 31, 31, 8)
    opt = dict(cg_tol_e=1e-13, cg_tol_p=1e-13)
    ref, _ = _run(w, 3, 2, steps=4, streaming=-1, **opt)
    st = torch.cuda.Stream()
    sim = gpu_sim(w, stream=st.cuda_stream, **opt)
    sim.set_initial(rest_X(w))
    sim.step(w.dt, 3, 2)
    sim.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
        sim.step(w.dt, 3, 2)
    with torch.cuda.stream(st):
        g.replay()
        g.replay()
    sim.step(w.dt, 3, 2)
    sim.sync()
    v, u, X = sim.fields(full=True)
    sim.close()
    assert rel(X, ref[2]) < 1e-9 and rel(u, ref[1]) < 1e-9


@pytest.mark.parametrize("mesh,prec", [(("slab", 31, 31, 8), binding.FP64), (("slab", 41, 37, 12), binding.MIXED)])
def test_batches_are_untouched(mesh, prec):
    w = _mesh(*mesh)
    out = []
    for s in (0, -1):
        sims = [gpu_sim(w, precision=prec, streaming=s) for _ in range(2)]
        for k, sim in enumerate(sims):
            sim.set_initial(rest_X(w) * (1.0 + 0.001 * k))
        for _ in range(2):
            binding.batch_step(sims, w.dt, 3, 2)
        out.append([a for sim in sims for a in sim.fields(full=True)])
        for sim in sims:
            sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", [binding.FP64, binding.MIXED])
def test_footprint_holds_the_chains(prec):
    torch = pytest.importorskip("torch")
    w = W.config2(101, 101, 26)
    opts = binding.default_options(pin_node=w.pin_node, precision=prec)
    est = binding.footprint_bytes(w.xyz, w.elems, w.model, opts, w.elem_bath)
    torch.cuda.init()
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    sim = binding.simulation_from_workload(w, opts)
    sim.step(w.dt, 3, 2)
    sim.sync()
    free1, _ = torch.cuda.mem_get_info()
    sim.close()
    assert 0.9 < est / (free0 - free1) < 1.6   # the bounds of the other forms' test
