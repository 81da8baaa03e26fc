"""Meshes that the elliptic preconditioner refuses, whatever solver form and
hierarchy the options lead to (the refusal comes before any device is looked
for): a mesh of two pieces (A_ie has two null vectors), no conductivity across the
fibres (one for every line of nodes), and a coarsest level too large for a dense
solve."""
import numpy as np
import pytest

from paper_2510_27447_gb300 import binding
from paper_2510_27447_gb300 import workloads as W


def _create(xyz, elems, sigma=(3.0, 0.31, 2.0, 1.35), **opt):
    """bd_create's error code, or 0; without a GPU what is accepted here ends with
    BD_ERR_CUDA."""
    try:
        sim = binding.Simulation(xyz, elems, None, sigma, 2000.0, 1.0, W.LR91, binding.default_options(**opt))
    except binding.BdError as e:
        return e.code
    sim.close()
    return 0


def _pieces(n):
    xyz, el = W.square_grid(n)
    return np.concatenate([xyz, xyz + [10.0, 0.0]]), np.concatenate([el, el + n * n]).astype(np.int32)


FORMS = [dict(precision=p, **o) for p in (binding.FP64, binding.MIXED)
         for o in (dict(), dict(cg_block=256), dict(streaming=1), dict(solver_tier=1))]


# sizes at which a hierarchy of 384 coarse rows is refused or, by rounding, not
@pytest.mark.parametrize("n", [5, 17, 21, 26])
@pytest.mark.parametrize("opt", FORMS)
def test_two_pieces(n, opt):
    xyz, el = _pieces(n)
    assert _create(xyz, el, **opt) == -1
    assert _create(xyz, el, elliptic_precond=0, **opt) != -1


@pytest.mark.parametrize("opt", FORMS)
def test_no_cross_conductivity(opt):
    xyz, el = W.square_grid(21)
    assert _create(xyz, el, sigma=(3.0, 0.0, 2.0, 0.0), **opt) == -1
    assert _create(xyz, el, **opt) != -1


@pytest.mark.parametrize("opt", FORMS)
def test_dense_level_too_large(opt):
    xyz, el = W.square_grid(66)
    assert _create(xyz, el, amg_coarse_max=5000, **opt) == -1
    assert _create(xyz, el, amg_coarse_max=1000, **opt) != -1
