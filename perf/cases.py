"""Workloads that are timed and whose results are compared when the solver changes.

One pass advances a simulation (or a set of simulations) by one time step
through the public entry points and takes a snapshot of the fields on the
device, as a program that keeps frames of a run does.  The simulations start
from a developed state -- a wave of the membrane model's own action potential
with its front inside the tissue, plateau behind it, rest ahead of it -- so
solves, membrane kernels and stimuli meet the values of a running simulation.

`exact` restates the step from the paper's equations in 64-bit torch, with
every linear system solved to rounding; it shares nothing with the library but
the mesh arrays.

Snapshots have the type whose accuracy the handle offers: float64 on FP64
handles, float32 on mixed-precision ones (their Krylov iterations and
membrane model run in FP32).
"""
import ctypes
import functools
import math

import numpy as np
import torch

from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W

MODELS = {"lr91": W.LR91, "lr91_paper": W.LR91_PAPER_MOD, "tp06": W.TP06_EPI}
# wave speed along the fibres used to lay out the initial wave, cm/ms
# (conduction velocities of the two models on these conductivities)
SPEED = {"lr91": 0.026, "lr91_paper": 0.020, "tp06": 0.052}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    sheet = dict(kind="sheet", scheme="sdc", nodes=3, sweeps=2, dt=0.02)
    return [
        # the smallest request of the serving stream, advanced on its own: launches and barriers
        dict(sheet, name="sheet33_lr91_mixed", n=33, length=1.0, model="lr91", precision="mixed"),
        # the 65^2 LR91 parity run in the paper's precision
        dict(sheet, name="sheet65_lr91_fp64", n=65, length=1.0, model="lr91", precision="fp64"),
        # a middle request of the serving stream
        dict(sheet, name="sheet129_tp06_mixed", n=129, length=1.0, model="tp06", precision="mixed"),
        # the TP06 re-entry sheet, in both precisions: the benchmark's headline workload
        dict(sheet, name="sheet257_tp06_mixed", n=257, length=2.5, model="tp06", precision="mixed"),
        dict(sheet, name="sheet257_tp06_fp64", n=257, length=2.5, model="tp06", precision="fp64"),
        # the largest request of the serving stream
        dict(sheet, name="sheet513_lr91_mixed", n=513, length=1.0, model="lr91", precision="mixed"),
        # the paper's production mode: steps of at most 0.05 ms chosen by the embedded estimate
        dict(sheet, name="adaptive101_lr91_fp64", scheme="adaptive", n=101, length=1.0, model="lr91",
             precision="fp64", dt=0.05),
        # the decoupled reference scheme at the step it needs, 100 x 100 cells
        dict(sheet, name="decoupled101_lr91_fp64", scheme="cnrk2", n=101, length=1.0, model="lr91",
             precision="fp64", dt=0.001),
        # bidomain-bath sheet: u on tissue and bath, v on the tissue only
        dict(kind="bath", name="bath401_lr91_mixed", scheme="sdc", nodes=3, sweeps=2, dt=0.05, n=401,
             model="lr91", precision="mixed"),
        # the 3-D slab with rotating fibres, in the paper's precision and in mixed precision
        dict(kind="slab", name="slab101_tp06_fp64", scheme="sdc", nodes=3, sweeps=2, dt=0.025, nx=101, ny=101,
             nz=26, model="tp06", precision="fp64"),
        dict(kind="slab", name="slab161_tp06_mixed", scheme="sdc", nodes=3, sweeps=2, dt=0.025, nx=161, ny=161,
             nz=41, model="tp06", precision="mixed"),
        # many small requests of the serving stream advanced together, one batch per model and mesh size
        dict(kind="batch", name="batch12_mixed", scheme="sdc", nodes=3, sweeps=2, dt=0.02, small=65, large=129,
             count=12, precision="mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c = {"kind": rng.choice(["sheet", "sheet", "sheet", "bath", "slab", "slab", "batch"])}
    c["precision"] = rng.choice(["mixed", "fp64"])
    c["scheme"] = "sdc"
    c["nodes"] = rng.choice([2, 3, 3])
    c["sweeps"] = rng.choice([1, 2, 2, 3])
    c["dt"] = rng.choice([0.01, 0.02, 0.025])
    if c["kind"] == "sheet":
        c["n"] = _log_int(rng, 33, 513)
        c["length"] = rng.choice([1.0, 2.5])
        c["model"] = rng.choice(["lr91", "lr91_paper", "tp06"])
        c["scheme"] = rng.choice(["sdc", "sdc", "sdc", "adaptive", "cnrk2"])
        if c["scheme"] == "cnrk2":
            c["dt"] = 0.001
        if c["scheme"] == "adaptive":
            c["dt"], c["nodes"], c["sweeps"] = 0.05, 3, 2
    elif c["kind"] == "bath":
        c["n"] = _log_int(rng, 41, 401)
        c["model"] = rng.choice(["lr91", "tp06"])
    elif c["kind"] == "slab":
        c["nx"], c["ny"] = _log_int(rng, 31, 121), _log_int(rng, 31, 121)
        c["nz"] = _log_int(rng, 8, 41)
        c["model"] = rng.choice(["lr91", "tp06"])
        if c["precision"] == "fp64":
            c["nx"] = min(c["nx"], 101)
            c["ny"] = min(c["ny"], 101)
            c["nz"] = min(c["nz"], 26)
    else:
        c["small"], c["large"] = _log_int(rng, 25, 65), _log_int(rng, 66, 129)
        c["count"] = rng.randint(4, 12)
    if c["sweeps"] == 3 and c["kind"] != "sheet":
        c["sweeps"] = 2
    return c


# ---------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------

def _members(case):
    """(kind-specific sub-cases, group index) of the simulations of a case."""
    if case["kind"] != "batch":
        return [(case, 0)]
    out = []
    for k in range(case["count"]):
        n = case["small"] if k % 2 == 0 else case["large"]
        model = "lr91" if (k // 2) % 2 == 0 else "tp06"
        out.append((dict(case, kind="sheet", n=n, length=1.0, model=model), k % 4))
    return out


def _workload(case, rng):
    """Mesh, fibres, conductivities and stimuli; the conductivities of sheets
    are jittered by U(-20 %, 20 %), as in the serving stream."""
    model = MODELS[case["model"]]
    if case["kind"] == "sheet":
        sigma = tuple(float(s * (1.0 + rng.uniform(-0.2, 0.2))) for s in W.CONFIG0_SIGMA)
        return W.sheet(case["n"], case["length"], model, case["dt"], 0, sigma=sigma,
                       s2=(float(rng.uniform(1.0, 4.0)), 0.5 * case["length"]))
    if case["kind"] == "bath":   # the paper's square: tissue in the middle three quarters
        cells = case["n"] - 1
        return W.bath_sheet(cells, -1.0, 7.0, 0.0, 6.0, model, case["dt"], 0,
                            s2=(float(rng.uniform(1.0, 4.0)), 1.0, 3.0))
    w = W.config2(case["nx"], case["ny"], case["nz"])
    w.model = model
    w.dt = case["dt"]
    return w


def _initial(case, w, rng):
    """State X[ns, n_tissue]: a plane wave of the model's action potential
    travelling in a random direction about the x axis, its front inside the
    tissue, gates perturbed by 2 % as in the slab workload."""
    table, step = _action_potential(case["model"])
    xyz = w.xyz[:w.n_tissue]
    lo, hi = xyz.min(axis=0), xyz.max(axis=0)
    a = rng.uniform(-0.6, 0.6)
    d = xyz[:, 0] * math.cos(a) + xyz[:, 1] * math.sin(a)
    front = d.min() + rng.uniform(0.3, 0.6) * (d.max() - d.min())
    ripple = 0.02 * (hi[1] - lo[1]) * np.sin(2 * math.pi * (xyz[:, 1] - lo[1]) / (hi[1] - lo[1]) + rng.uniform(0, 6.28))
    phase = np.maximum((front + ripple - d) / SPEED[case["model"]], 0.0) / step
    k = np.minimum(phase.astype(np.int64), len(table) - 2)
    f = np.minimum(phase - k, 1.0)
    X = ((1.0 - f)[:, None] * table[k] + f[:, None] * table[k + 1]).T.copy()
    gates = range(1, 7) if X.shape[0] == 8 else range(1, 13)
    for g in gates:
        X[g] = np.clip(X[g] * (1.0 + rng.uniform(-0.02, 0.02, X.shape[1])), 0.0, 1.0)
    return X


def _inputs(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for sub, group in _members(case):
        w = _workload(sub, rng)
        out.append((sub, group, w, _initial(sub, w, rng)))
    return out


class _DeviceArray:
    """A device buffer of a handle, as torch takes it without a copy."""

    def __init__(self, ptr, shape):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f8", "data": (ptr, False), "version": 3}


@functools.lru_cache(maxsize=None)
def _stream(group):
    """The stream of a case's group of handles: one simulation steps at a time,
    the batches of different groups may overlap."""
    return torch.cuda.Stream()


class _State:
    """The handles of a case by group, each group on a stream of its own."""

    def __init__(self, case):
        self.case = case
        self.streams, self.groups, self.views = [], [], []


def _views(sim):
    X, u = ctypes.c_void_p(), ctypes.c_void_p()
    rc = binding.lib().bd_device_fields(sim.h, ctypes.byref(X), ctypes.byref(u))
    if rc != binding.BD_OK:
        raise RuntimeError("bd_device_fields: %d" % rc)
    return (torch.as_tensor(_DeviceArray(X.value, (sim.ns, sim.NT)), device="cuda"),
            torch.as_tensor(_DeviceArray(u.value, (sim.N,)), device="cuda"))


def prepare(case, seed):
    st = _State(case)
    prec = binding.MIXED if case["precision"] == "mixed" else binding.FP64
    for _, group, w, X in _inputs(case, seed):
        while group >= len(st.groups):
            st.streams.append(_stream(group))
            st.groups.append([])
            st.views.append([])
        opts = binding.default_options(precision=prec, pin_node=w.pin_node, stream=st.streams[group].cuda_stream)
        sim = binding.simulation_from_workload(w, opts)
        sim.set_initial(X)
        st.groups[group].append(sim)
        st.views[group].append(_views(sim))
    return st


def run(st):
    case = st.case
    frame = torch.float32 if case["precision"] == "mixed" else torch.float64
    out = []
    for stream, sims, views in zip(st.streams, st.groups, st.views):
        if case["kind"] == "batch":
            binding.batch_step(sims, case["dt"], case["nodes"], case["sweeps"])
        elif case["scheme"] == "cnrk2":
            sims[0].step_decoupled(case["dt"])
        elif case["scheme"] == "adaptive":
            sims[0].step_adaptive(case["dt"], 1e-2, case["nodes"], case["sweeps"])
        else:
            sims[0].step(case["dt"], case["nodes"], case["sweeps"])
        with torch.cuda.stream(stream):   # the handles' stream: after the step, before the next one
            out += [{"X": X.to(frame, copy=True), "u": u.to(frame, copy=True)} for X, u in views]
    return out


def work(case):
    """One pass: state and potential read and written, each operator and the
    lumped mass read once; arithmetic of the membrane evaluations of the
    scheme and of one operator application per linear system."""
    b = f = 0.0
    frame = 4 if case["precision"] == "mixed" else 8
    for sub, _ in _members(case):
        if sub["kind"] == "slab":
            n = nt = sub["nx"] * sub["ny"] * sub["nz"]
            nnz = 15 * n
        else:
            n = sub["n"] ** 2
            nt = n if sub["kind"] == "sheet" else int(round(0.75 * (sub["n"] - 1)) + 1) ** 2
            nnz = 7 * n
        ns, field = (19, 900.0) if sub["model"] == "tp06" else (8, 400.0)
        b += 2 * 8 * (ns * nt + n) + frame * (ns * nt + n) + (3 * 8 + 4) * nnz + 8 * nt
        if sub["scheme"] == "cnrk2":
            f += 4 * field * nt + 2 * 2 * nnz
        else:
            M, K = sub["nodes"], sub["sweeps"]
            f += K * (3 * (M - 1) + M) * field * nt + K * 4 * (M - 1) * 2 * nnz
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# membrane models, for scalars (math) and tensors (torch, also complex)
# ---------------------------------------------------------------------------

class _Scalar:
    exp, log, sqrt = math.exp, math.log, math.sqrt

    @staticmethod
    def where(c, a, b):
        return a if c else b

    @staticmethod
    def real(x):
        return x

    @staticmethod
    def exprel(z):
        return math.expm1(z) / z if z != 0.0 else 1.0


class _Tensor:
    exp, log, sqrt = torch.exp, torch.log, torch.sqrt

    @staticmethod
    def where(c, a, b):
        a = a if torch.is_tensor(a) else torch.full_like(b, a)
        b = b if torch.is_tensor(b) else torch.full_like(a, b)
        return torch.where(c, a, b)

    @staticmethod
    def real(x):
        return x.real if torch.is_complex(x) else x

    @staticmethod
    def exprel(z):
        near = _Tensor.real(z).abs() < 0.25
        s = torch.ones_like(z)
        for k in range(15, 1, -1):
            s = 1.0 + s * z / k
        zz = torch.where(near, torch.ones_like(z), z)
        return torch.where(near, s, (torch.exp(zz) - 1.0) / zz)


def _lr91(x, istim, cm, o, paper=False):
    """Luo & Rudy 1991: ([(steady state, time constant)] of the gates m h j d
    f X, [dV/dt], [dCai/dt])."""
    V, m, h, j, d, f, X, ca = x
    e = o.exp
    rtf = 8314.0 * 310.0 / 96484.6
    e_na = rtf * math.log(140.0 / 18.0)
    e_k = rtf * math.log((5.4 + 0.01833 * 140.0) / (145.0 + 0.01833 * 18.0))
    e_k1 = rtf * math.log(5.4 / 145.0)
    g_na, g_si, g_k = (4.0, 0.02, 0.423) if paper else (23.0, 0.09, 0.282)
    hi = o.real(V) >= -40.0
    rates = [
        (3.2 / o.exprel(-0.1 * (V + 47.13)), 0.08 * e(-V / 11.0)),
        (o.where(hi, 0.0, 0.135 * e(-(80.0 + V) / 6.8)),
         o.where(hi, 1.0 / (0.13 * (1.0 + e(-(V + 10.66) / 11.1))), 3.56 * e(0.079 * V) + 3.1e5 * e(0.35 * V))),
        (o.where(hi, 0.0, (-1.2714e5 * e(0.2444 * V) - 3.474e-5 * e(-0.04391 * V)) * (V + 37.78)
                 / (1.0 + e(0.311 * (V + 79.23)))),
         o.where(hi, 0.3 * e(-2.535e-7 * V) / (1.0 + e(-0.1 * (V + 32.0))),
                 0.1212 * e(-0.01052 * V) / (1.0 + e(-0.1378 * (V + 40.14))))),
        (0.095 * e(-0.01 * (V - 5.0)) / (1.0 + e(-0.072 * (V - 5.0))),
         0.07 * e(-0.017 * (V + 44.0)) / (1.0 + e(0.05 * (V + 44.0)))),
        (0.012 * e(-0.008 * (V + 28.0)) / (1.0 + e(0.15 * (V + 28.0))),
         0.0065 * e(-0.02 * (V + 30.0)) / (1.0 + e(-0.2 * (V + 30.0)))),
        (0.0005 * e(0.083 * (V + 50.0)) / (1.0 + e(0.057 * (V + 50.0))),
         0.0013 * e(-0.06 * (V + 20.0)) / (1.0 + e(-0.04 * (V + 20.0))))]
    gates = [(a / (a + b), 1.0 / (a + b)) for a, b in rates]
    i_si = g_si * d * f * (V - (7.7 - 13.0287 * o.log(ca)))
    xi = o.where(o.real(V) > -100.0, 0.11348 * o.exprel(0.04 * (V + 77.0)) * e(-0.04 * (V + 35.0)), 1.0)
    w = V - e_k1
    ak = 1.02 / (1.0 + e(0.2385 * (w - 59.215)))
    bk = (0.49124 * e(0.08032 * (w + 5.476)) + e(0.06175 * (w - 594.31))) / (1.0 + e(-0.5143 * (w + 4.753)))
    I = (g_na * m * m * m * h * j * (V - e_na) + i_si + g_k * X * xi * (V - e_k) + 0.6047 * ak / (ak + bk) * w
         + 0.0183 * w / (1.0 + e((7.488 - V) / 5.98)) + 0.03921 * (V + 59.87))
    return gates, -(I - istim) / cm, [-1e-4 * i_si + 0.07 * (1e-4 - ca)]


def _tp06(x, istim, cm, o):
    """ten Tusscher & Panfilov 2006, epicardial cell: ([(steady state, time
    constant)] of the gates m h j d f f2 s r Xr1 Xr2 Xs fCass, dV/dt,
    derivatives of Rbar Ki Nai Cai CaSR CaSS)."""
    V, m, h, j, d, f, f2, s, r, xr1, xr2, xs, fc, rb, ki, nai, cai, sr, ss = x
    e, log = o.exp, o.log
    F, rtf = 96485.3415, 8314.472 * 310.0 / 96485.3415
    vc, vsr, vss = 0.016404, 0.001094, 0.00005468

    def sig(a):
        return 1.0 / (1.0 + e(a))

    hi = o.real(V) >= -40.0
    hj = sig((V + 71.55) / 7.43) * sig((V + 71.55) / 7.43)
    ah = o.where(hi, 0.0, 0.057 * e(-(V + 80.0) / 6.8))
    bh = o.where(hi, 0.77 / 0.13 * sig(-(V + 10.66) / 11.1), 2.7 * e(0.079 * V) + 3.1e5 * e(0.3485 * V))
    aj = o.where(hi, 0.0, (-2.5428e4 * e(0.2444 * V) - 6.948e-6 * e(-0.04391 * V)) * (V + 37.78)
                 * sig(0.311 * (V + 79.23)))
    bj = o.where(hi, 0.6 * e(0.057 * V) * sig(-0.1 * (V + 32.0)),
                 0.02424 * e(-0.01052 * V) * sig(-0.1378 * (V + 40.14)))
    q = (ss / 0.05) * (ss / 0.05)
    v27, v45, v40 = V + 27.0, V + 45.0, V + 40.0
    gates = [
        (sig((-56.86 - V) / 9.03) * sig((-56.86 - V) / 9.03),
         sig((-60.0 - V) / 5.0) * (0.1 * sig((V + 35.0) / 5.0) + 0.1 * sig((V - 50.0) / 200.0))),
        (hj, 1.0 / (ah + bh)),
        (hj, 1.0 / (aj + bj)),
        (sig((-8.0 - V) / 7.5),
         (1.4 * sig((-35.0 - V) / 13.0) + 0.25) * 1.4 * sig((V + 5.0) / 5.0) + sig((50.0 - V) / 20.0)),
        (sig((V + 20.0) / 7.0),
         1102.5 * e(-v27 * v27 / 225.0) + 200.0 * sig((13.0 - V) / 10.0) + 180.0 * sig((V + 30.0) / 10.0) + 20.0),
        (0.67 * sig((V + 35.0) / 7.0) + 0.33,
         562.0 * e(-v27 * v27 / 240.0) + 31.0 * sig((25.0 - V) / 10.0) + 80.0 * sig((V + 30.0) / 10.0)),
        (sig((V + 20.0) / 5.0), 85.0 * e(-v45 * v45 / 320.0) + 5.0 * sig((V - 20.0) / 5.0) + 3.0),
        (sig((20.0 - V) / 6.0), 9.5 * e(-v40 * v40 / 1800.0) + 0.8),
        (sig((-26.0 - V) / 7.0), 450.0 * sig((-45.0 - V) / 10.0) * 6.0 * sig((V + 30.0) / 11.5)),
        (sig((V + 88.0) / 24.0), 3.0 * sig((-60.0 - V) / 20.0) * 1.12 * sig((V - 60.0) / 20.0)),
        (sig((-5.0 - V) / 14.0), 1400.0 / o.sqrt(1.0 + e((5.0 - V) / 6.0)) * sig((V - 35.0) / 15.0) + 80.0),
        (0.6 / (1.0 + q) + 0.4, 80.0 / (1.0 + q) + 2.0)]
    e_na, e_k = rtf * log(140.0 / nai), rtf * log(5.4 / ki)
    e_ks = rtf * log((5.4 + 0.03 * 140.0) / (ki + 0.03 * nai))
    e_ca = 0.5 * rtf * log(2.0 / cai)
    w = V - e_k
    ak = 0.1 * sig(0.06 * (w - 200.0))
    bk = (3.0 * e(0.0002 * (w + 100.0)) + e(0.1 * (w - 10.0))) * sig(-0.5 * w)
    i_k1, i_to, i_kr = 5.405 * ak / (ak + bk) * w, 0.294 * r * s * w, 0.153 * xr1 * xr2 * w
    i_ks = 0.392 * xs * xs * (V - e_ks)
    z = 2.0 * (V - 15.0) / rtf
    i_cal = 0.0000398 * 2.0 * F * d * f * f2 * fc * (0.25 * ss * e(z) - 2.0) / o.exprel(z)
    i_na, i_bna = 14.838 * m * m * m * h * j * (V - e_na), 0.00029 * (V - e_na)
    i_bca, i_pca = 0.000592 * (V - e_ca), 0.1238 * cai / (cai + 0.0005)
    i_nak = (2.724 * 5.4 / 6.4 * nai / (nai + 40.0)) / (1.0 + 0.1245 * e(-0.1 * V / rtf) + 0.0353 * e(-V / rtf))
    eg = e(-0.65 * V / rtf)
    i_naca = (1000.0 * (e(0.35 * V / rtf) * nai * nai * nai * 2.0 - eg * (140.0 ** 3 * 2.5) * cai)
              / ((87.5 ** 3 + 140.0 ** 3) * 3.38 * (1.0 + 0.1 * eg)))
    i_pk = 0.0146 * w * sig((25.0 - V) / 5.98)
    I = i_k1 + i_to + i_kr + i_ks + i_cal + i_na + i_bna + i_bca + i_nak + i_naca + i_pca + i_pk
    kc = 2.5 - 1.5 / (1.0 + (1.5 / sr) * (1.5 / sr))
    k1, k2 = 0.15 / kc, 0.045 * kc
    i_rel = 0.102 * (k1 * ss * ss * rb / (0.06 + k1 * ss * ss)) * (sr - ss)
    i_up = 0.006375 / (1.0 + (0.00025 / cai) * (0.00025 / cai))
    i_leak, i_xfer = 0.00036 * (sr - cai), 0.0038 * (ss - cai)
    cvf = 0.185 / (vc * F)
    bc = 1.0 / (1.0 + 0.2 * 0.001 / ((cai + 0.001) * (cai + 0.001)))
    bsr = 1.0 / (1.0 + 10.0 * 0.3 / ((sr + 0.3) * (sr + 0.3)))
    bss = 1.0 / (1.0 + 0.4 * 0.00025 / ((ss + 0.00025) * (ss + 0.00025)))
    rest = [-k2 * ss * rb + 0.005 * (1.0 - rb),
            -(i_k1 + i_to + i_kr + i_ks + i_pk - 2.0 * i_nak - istim) * cvf,
            -(i_na + i_bna + 3.0 * i_nak + 3.0 * i_naca) * cvf,
            bc * ((i_leak - i_up) * (vsr / vc) + i_xfer - (i_bca + i_pca - 2.0 * i_naca) * (0.5 * cvf)),
            bsr * (i_up - (i_rel + i_leak)),
            bss * (-i_cal * 0.185 / (2.0 * vss * F) + i_rel * (vsr / vss) - i_xfer * (vc / vss))]
    return gates, -(I - istim) / cm, rest


def _model(name):
    if name == "tp06":
        return _tp06
    return functools.partial(_lr91, paper=name == "lr91_paper")


@functools.lru_cache(maxsize=None)
def _action_potential(name):
    """(table [T, ns], sample spacing in ms): one paced cell over 300 ms, the
    gates by the exponential rule, the rest by forward Euler."""
    model, dt, every = _model(name), 0.02, 10
    x = [float(v) for v in (
        (-85.23, 0.00172, 0.7444, 0.7045, 3.373e-5, 0.7888, 0.9755, 0.999998, 2.42e-8, 0.00621, 0.4712, 0.0095,
         0.9953, 0.9073, 136.89, 8.604, 0.000126, 3.64, 0.00036) if name == "tp06" else
        (-84.3801107371, 0.00171338077730188, 0.982660523699656, 0.989108212766685, 0.00302126301779861,
         0.999967936476325, 0.0417603108167287, 0.00017948816388306))]
    rows = []
    for n in range(15000):
        if n % every == 0:
            rows.append(list(x))
        gates, dv, rest = model(x, 60.0 if n * dt < 1.0 else 0.0, 1.0, _Scalar)
        ng = len(gates)
        x = ([x[0] + dt * dv] + [g + (g - i) * math.expm1(-dt / t) for g, (i, t) in zip(x[1:1 + ng], gates)]
             + [a + dt * b for a, b in zip(x[1 + ng:], rest)])
    return np.array(rows), dt * every


# ---------------------------------------------------------------------------
# the step in 64 bits
# ---------------------------------------------------------------------------

GAMMA = 1.0 + 1.0 / math.sqrt(2.0)


class _Problem:
    """P1 operators of one workload on the GPU, and the steps of the paper
    with every linear system solved to rounding."""

    def __init__(self, w, model):
        dev = torch.device("cuda")
        self.model, self.cm, self.pin, dim = _model(model), w.cm, w.pin_node, w.xyz.shape[1]
        self.n, self.nt, self.lam = w.n_nodes, w.n_tissue, 0.25 if dim == 2 else 0.2
        xyz, el = torch.from_numpy(w.xyz).to(dev), torch.from_numpy(w.elems).to(dev).long()
        P = xyz[el]
        B = P[:, 1:] - P[:, :1]                                   # rows x_k - x_0
        meas = torch.linalg.det(B).abs() / (2.0 if dim == 2 else 6.0)
        g = torch.linalg.inv(B).transpose(1, 2)                   # gradients of the last dim basis functions
        g = torch.cat([-g.sum(1, keepdim=True), g], 1)
        fib = torch.from_numpy(w.fibers).to(dev)
        gf = (g * fib[:, None, :]).sum(2)
        iso, fibre = g @ g.transpose(1, 2), gf[:, :, None] * gf[:, None, :]
        bath = torch.zeros(len(el), dtype=torch.bool, device=dev)
        if w.elem_bath is not None:
            bath = torch.from_numpy(w.elem_bath).to(dev) != 0

        tissue = (~bath).to(torch.float64)

        def local(sl, st, sb):
            t = (sb + (st - sb) * tissue)[:, None, None] * iso + ((sl - st) * tissue)[:, None, None] * fibre
            return t * meas[:, None, None] / (w.chi * w.cm)

        sil, sit, sel, set_ = w.sigma
        k = dim + 1
        ones = torch.ones(k, k, device=dev, dtype=torch.float64)
        mass = (ones + torch.diag(ones[0])) / (k * (k + 1))
        vals = [local(sil, sit, 0.0), local(sil + sel, sit + set_, w.sbath),
                (meas * tissue)[:, None, None] * mass]
        key = (el[:, :, None] * self.n + el[:, None, :]).reshape(-1)
        uniq, inv = torch.unique(key, return_inverse=True)
        row, col = uniq // self.n, uniq % self.n
        Ai, Aie, M = (torch.zeros(len(uniq), dtype=torch.float64, device=dev).index_add_(0, inv, v.reshape(-1))
                      for v in vals)
        self.Ai_all, self.Aie = self._csr(row, col, Ai, self.n), self._csr(row, col, Aie, self.n)
        self.d_Aie = Aie[row == col]
        t = (row < self.nt) & (col < self.nt)
        self.row, self.col, self.Ai, self.M = row[t], col[t], Ai[t], M[t]
        self.A = self._csr(self.row, self.col, self.Ai, self.nt)
        self.Mc = self._csr(self.row, self.col, self.M, self.nt)
        self.ML = torch.mv(self.Mc, torch.ones(self.nt, dtype=torch.float64, device=dev))
        self.stim = [(torch.from_numpy(s.mask[:self.nt].astype(np.float64)).to(dev), s) for s in w.stimuli]

    @staticmethod
    def _csr(row, col, val, n):
        ptr = torch.zeros(n + 1, dtype=torch.int64, device=row.device)
        ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
        return torch.sparse_csr_tensor(ptr, col, val, (n, n))

    @staticmethod
    def _cg(A, invd, b, project, passes=4):
        """Jacobi-preconditioned CG, refined until the residual no longer falls."""
        x, best = torch.zeros_like(b), math.inf
        for _ in range(passes):
            r = b - torch.mv(A, x)
            if project:
                r = r - r.mean()
            rr0 = float(r.dot(r))
            if not 0.0 < rr0 < 0.25 * best:
                break
            best = rr0
            d, z = torch.zeros_like(b), invd * r
            p, rho = z.clone(), r.dot(z)
            for it in range(20000):
                q = torch.mv(A, p)
                a = rho / p.dot(q)
                d += a * p
                r = r - a * q
                if it % 8 == 7 and float(r.dot(r)) <= 1e-18 * rr0:
                    break
                z = invd * r
                new = r.dot(z)
                p = z + (new / rho) * p
                rho = new
            x = x + d
        return x

    def elliptic(self, v):
        full = torch.zeros(self.n, dtype=torch.float64, device=v.device)
        full[:self.nt] = v
        b = -torch.mv(self.Ai_all, full)
        u = self._cg(self.Aie, 1.0 / self.d_Aie, b - b.mean(), True)
        return u - u[self.pin]

    def istim(self, t, dt):
        out = torch.zeros(self.nt, dtype=torch.float64, device="cuda")
        for mask, s in self.stim:
            if t - s.t_on > -1e-9 * dt and t - s.t_on - s.duration < -1e-9 * dt:
                out += s.amplitude * mask
        return out

    def field(self, X, ist):
        gates, dv, rest = self.model(list(X), ist, self.cm, _Tensor)
        return torch.stack([dv] + [(i - X[1 + k]) / t for k, (i, t) in enumerate(gates)] + rest)

    def jacobian(self, X, ist):
        """J[r, c, node] by the complex step (exact to rounding)."""
        ns, h = X.shape[0], 1e-40
        J = torch.empty(ns, ns, X.shape[1], dtype=torch.float64, device=X.device)
        for c in range(ns):
            Z = X.to(torch.complex128)
            Z[c] += 1j * h
            J[:, c] = self.field(Z, ist.to(torch.complex128)).imag / h
        return J

    def F_v(self, X, u, f):
        return -torch.mv(self.A, X[0] + u[:self.nt]) + self.ML * f[0]

    def solve(self, alpha, J, rv, ry):
        """k of (alpha Mt - W) k = (rv, ML ry), the node states eliminated."""
        n1 = J.shape[0] - 1
        A = alpha * torch.eye(n1, dtype=torch.float64, device=J.device)[:, :, None] - J[1:, 1:]
        R = torch.stack([ry, J[1:, 0]], 1)
        for k in range(n1):
            l = A[k + 1:, k] / A[k, k]
            A[k + 1:, k:] -= l[:, None] * A[k, k:][None]
            R[k + 1:] -= l[:, None] * R[k][None]
        for k in range(n1 - 1, -1, -1):
            R[k] = (R[k] - (A[k, k + 1:, None] * R[k + 1:]).sum(0)) / A[k, k]
        z, y = R[:, 0], R[:, 1]
        s = torch.clamp(-J[0, 0] - (J[0, 1:] * y).sum(0), min=-0.9 * alpha * self.lam)
        b = rv + self.ML * (J[0, 1:] * z).sum(0)
        kv = self.shifted(alpha, self.ML * s, b)
        return torch.cat([kv[None], z + y * kv])

    def shifted(self, alpha, diag, b):
        val = alpha * self.M + self.Ai
        on = self.row == self.col
        val[on] += diag
        return self._cg(self._csr(self.row, self.col, val, self.nt), 1.0 / val[on], b, False)

    def ros2(self, X, h, u, ist):
        alpha = 1.0 / (GAMMA * h)
        J, f = self.jacobian(X, ist), self.field(X, ist)
        k1 = self.solve(alpha, J, self.F_v(X, u, f), f[1:])
        Xs, c = X + k1 / GAMMA, 2.0 / (GAMMA * h)
        f = self.field(Xs, ist)
        k2 = self.solve(alpha, J, self.F_v(Xs, u, f) - c * torch.mv(self.Mc, k1[0]), f[1:] - c * k1[1:])
        return X + (1.5 / GAMMA) * k1 + (0.5 / GAMMA) * k2, Xs

    def sdc(self, X, u_n, dt, M, K):
        """(X, u, embedded error estimate / tolerance) after one step from t = 0."""
        c = [0.0, 1.0] if M == 2 else [0.0, 0.5, 1.0]
        S = [[0.5, 0.5]] if M == 2 else [[5 / 24, 1 / 3, -1 / 24], [-1 / 24, 1 / 3, 5 / 24]]
        ist, Xk, u = self.istim(0.0, dt), [X] * M, [u_n] + [None] * (M - 1)
        for k in range(K):
            u[1:] = [self.elliptic(Xk[m][0]) for m in range(1, M)] if k else [self.elliptic(X[0])] * (M - 1)
            Xt, err = [X], 0.0
            for m in range(M - 1):
                new, hat = self.ros2(Xt[m], dt * (c[m + 1] - c[m]), u[m + 1], ist)
                err = max(err, float(((new - hat).abs() / (1.0 + new.abs())).max()))
                Xt.append(new)
            f = [self.field(x, ist) for x in Xt]
            fv = [self.F_v(Xt[m], u[m], f[m]) for m in range(M)]
            Xk = [X]
            for m in range(M - 1):
                h, D = dt * (c[m + 1] - c[m]), Xk[m] - Xt[m + 1]
                rv = torch.mv(self.Mc, D[0]) + sum(dt * S[m][q] * fv[q] for q in range(M))
                ry = D[1:] + sum(dt * S[m][q] * f[q][1:] for q in range(M))
                Xk.append(Xt[m + 1] + self.solve(1.0 / h, self.jacobian(Xt[m + 1], ist), rv / h, ry / h))
        return Xk[-1], u[-1], err

    def adaptive(self, X, u_n, dt_max, tol, M, K):
        dt = dt_max
        while True:
            Xn, un, err = self.sdc(X, u_n, dt, M, K)
            if err <= tol or dt <= dt_max * 2.0 ** -7 * (1 + 1e-12):
                return Xn, un
            want = min(0.5 * dt, dt * max(0.5, 0.9 * math.sqrt(tol / err)))
            rungs = [dt_max * 2.0 ** -k for k in range(8)]
            dt = next(d for d in rungs if d <= want * (1 + 1e-12) or d == rungs[-1])

    def cnrk2(self, X, u_n, dt):
        ist, h = self.istim(0.0, dt), 0.5 * dt

        def half(x):
            return x + h * self.field(x + 0.5 * h * self.field(x, ist), ist)

        Y = half(X)
        zero = torch.zeros(self.nt, dtype=torch.float64, device=X.device)
        Y[0] += self.shifted(2.0 / dt, zero, -2.0 * torch.mv(self.A, Y[0] + u_n[:self.nt]))
        Xn = half(Y)
        return Xn, self.elliptic(Xn[0])


def exact(case, seed):
    out = {}
    for k, (sub, group, w, X) in enumerate(_inputs(case, seed)):
        p = _Problem(w, sub["model"])
        x, u0 = torch.from_numpy(X).cuda(), torch.zeros(p.n, dtype=torch.float64, device="cuda")
        if sub["scheme"] == "cnrk2":
            xn, un = p.cnrk2(x, u0, sub["dt"])
        elif sub["scheme"] == "adaptive":
            xn, un = p.adaptive(x, u0, sub["dt"], 1e-2, sub["nodes"], sub["sweeps"])
        else:
            xn, un, _ = p.sdc(x, u0, sub["dt"], sub["nodes"], sub["sweeps"])
        out[(group, k)] = {"X": xn, "u": un}
    return [out[key] for key in sorted(out)]   # group by group, as run returns them
