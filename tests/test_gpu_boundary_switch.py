"""Boundary data given, left out (NULL: homogeneous) and given again on one
context: every sweep must be the one a fresh context makes of the same front
and data, whatever was captured before, and NULL must mean zeros.  Columns
split over a cluster and not, both precisions, Dirichlet and Neumann walls."""
import numpy as np
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu

# the sums over the facets are the same in the same order: only the zeros that
# NULL leaves out differ, so the bound is a few roundings of the path
TOL = {"fp64": 1e-14, "mixed": 1e-13}


def _case(dim, nrhs, rhs_split, precision):
    import torch
    import paper_1907_02367_gb300 as pkg
    m = inputs.mesh_square(4, 0.2, seed=6) if dim == 2 else inputs.mesh_cube(2, 0.1, seed=4)
    bnd = inputs.boundary_marker(m, lambda x: x[0] < 1e-12)   # one Neumann side
    T, kappa = 0.15, inputs.pitch_kappa(m)

    def make():
        return pkg.Solver(m.coords, m.elems, m.c, 3, T, kappa, nrhs=nrhs, rhs_split=rhs_split, precision=precision, bnd_type=bnd)

    s = make()
    x, _ = s.front_points()
    init = inputs.gaussian_pulse([0.4] * dim, 0.3)
    front = torch.tensor(np.stack([init(x) * (r + 1) for r in range(nrhs)]), dtype=torch.float64, device="cuda").contiguous()
    xt = s.boundary_points()
    g = torch.tensor(np.stack([np.sin(2.0 * xt[:, 0] + r) * (1.0 + xt[:, -1]) for r in range(nrhs)]), dtype=torch.float64,
                     device="cuda").contiguous()
    return make, s, front, g


def _sweep(s, front, g):
    s.set_state(front, g)
    s.advance()
    assert s.sync_status() == (0, 0)
    return s.get_state()[0]


CASES = [(2, 1, 1, "fp64"), (2, 3, 1, "mixed"), (2, 8, 4, "fp64"), (2, 32, 2, "mixed"), (3, 16, 2, "fp64"), (3, 32, 2, "mixed")]


@pytest.mark.parametrize("dim,nrhs,rhs_split,precision", CASES)
def test_data_and_no_data_in_turn(cuda_device, dim, nrhs, rhs_split, precision):
    import torch
    make, s, front, g = _case(dim, nrhs, rhs_split, precision)
    with_g, without = _sweep(make(), front, g), _sweep(make(), front, None)
    n = float(with_g.norm())
    assert float((with_g - without).norm()) > 1e-3 * n
    assert float((_sweep(make(), front, torch.zeros_like(g)) - without).norm()) <= TOL[precision] * n
    for data in (g, None, g, g, None):
        ref = without if data is None else with_g
        assert float((_sweep(s, front, data) - ref).norm()) <= TOL[precision] * n


@pytest.mark.parametrize("dim,nrhs,rhs_split,precision", CASES[:3])
def test_data_after_a_sweep_from_set_front(cuda_device, dim, nrhs, rhs_split, precision):
    """A context whose first sweep is captured before any set_state (set_front,
    advance) sweeps the same levels with the data of a later set_state."""
    import torch
    make, s, front, g = _case(dim, nrhs, rhs_split, precision)
    with_g, without = _sweep(make(), front, g), _sweep(make(), front, None)
    n = float(with_g.norm())
    tau0 = torch.zeros_like(s.get_state()[1])
    s.set_front(front, tau0)
    s.advance()
    assert float((s.get_state()[0] - without).norm()) <= TOL[precision] * n
    assert float((_sweep(s, front, g) - with_g).norm()) <= TOL[precision] * n
    s.set_front(front, tau0)   # the data are kept by set_front
    s.advance()
    assert float((s.get_state()[0] - with_g).norm()) <= TOL[precision] * n
