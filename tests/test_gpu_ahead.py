"""Tents assembled ahead of their wait, from tabulated front times, with the
S-point rule of the face integrals and the float-float inverse.

* Every degree with a rule of its own (2D p = 1..5, 3D p = 1..3) and 1D, one and
  five right-hand sides, both precisions, against the oracle (the bars of the
  parity tests: binary64 1e-11, 1e-10 at p = 5 on whole sweeps; mixed 1e-8).
* The inverse's register paths (up to 32, 64 and 96 unknowns): two and three
  materials at p = 3..5 in 2D, against the oracle.
* A front whose times are not the tents' own (tp_set_front): the dataflow sweep
  finds them after its wait and assembles again; the same levels launched one
  by one take the front's times from the start."""
import numpy as np
import pytest

from oracle import pitching, tdg
from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sweep(m, p, T, kappa, init, nrhs=1, precision="fp64", schedule="dataflow"):
    import torch
    import paper_1907_02367_gb300 as pkg
    s = pkg.Solver(m.coords, m.elems, m.c, p, T, kappa, nrhs=nrhs, precision=precision, schedule=schedule)
    xq, _ = s.front_points()
    f = torch.tensor(init(xq), dtype=torch.float64, device="cuda").view(1, m.n_elem, s.Q, -1)
    scale = torch.arange(1, nrhs + 1, dtype=torch.float64, device="cuda").view(-1, 1, 1, 1)
    s.set_state((f * scale).contiguous())
    s.advance()
    assert s.sync_status() == (0, 0)
    return s, (s.get_state()[0] / scale).cpu().numpy()


def _reference(m, p, T, kappa, init):
    r = pitching.pitch(m.coords, m.elems, m.c, kappa, T)
    return tdg.sweep(m.coords, m.elems, m.c, p, r, init, None)[0]


@pytest.mark.parametrize("dim,p", [(1, 1), (1, 6), (2, 1), (2, 2), (2, 3), (2, 4), (2, 5), (3, 1), (3, 2), (3, 3)])
def test_degrees_against_the_oracle(cuda_device, dim, p):
    m = {1: inputs.mesh_interval(5), 2: inputs.mesh_square(3, 0.2, seed=5), 3: inputs.mesh_cube(1, 0.0, seed=3)}[dim]
    T, kappa = {1: 0.5, 2: 0.2, 3: 0.3}[dim], inputs.pitch_kappa(m)
    init = inputs.gaussian_pulse([0.4] * dim, 0.3)
    ref = _reference(m, p, T, kappa, init)
    for precision, tol in (("fp64", 1e-10 if p >= 5 else 1e-11), ("mixed", 1e-8)):
        for nrhs in (1, 5):
            _, got = _sweep(m, p, T, kappa, init, nrhs, precision)
            for r in range(nrhs):
                rel = np.linalg.norm(got[r] - ref) / np.linalg.norm(ref)
                assert rel <= tol, (precision, nrhs, r, rel)


@pytest.mark.parametrize("p,materials", [(3, 2), (4, 2), (5, 2), (4, 3)])
def test_unknowns_of_interface_tents(cuda_device, p, materials):
    """2 x 16 = 32, 2 x 25 = 50, 2 x 36 = 72 and 3 x 25 = 75 unknowns."""
    m = inputs.mesh_square(4, 0.1, seed=9)
    cen = m.coords[m.elems].mean(axis=1)
    m.c[:] = np.where(cen[:, 0] > 0.5, 1.4, 1.0)
    if materials == 3:
        m.c[(cen[:, 0] > 0.5) & (cen[:, 1] > 0.5)] = 0.8
    T, kappa = 0.1, inputs.pitch_kappa(m)
    init = inputs.gaussian_pulse((0.45, 0.5), 0.3)
    ref = _reference(m, p, T, kappa, init)
    for precision, tol in (("fp64", 1e-10 if p >= 5 else 1e-11), ("mixed", 1e-8)):
        _, got = _sweep(m, p, T, kappa, init, 1, precision)
        rel = np.linalg.norm(got[0] - ref) / np.linalg.norm(ref)
        assert rel <= tol, (precision, rel)


@pytest.mark.parametrize("dim,precision", [(1, "fp64"), (2, "fp64"), (2, "mixed"), (3, "mixed")])
def test_front_with_other_times(cuda_device, dim, precision):
    import torch
    m = {1: inputs.mesh_interval(9), 2: inputs.mesh_square(5, 0.2, seed=4), 3: inputs.mesh_cube(2, 0.1, seed=4)}[dim]
    p, T, kappa = 3, 0.4, inputs.pitch_kappa(m)
    init = inputs.gaussian_pulse([0.4] * dim, 0.3)
    fronts, mid = [], None
    for schedule in ("dataflow", "levels"):
        s, _ = _sweep(m, p, T, kappa, init, 1, precision, schedule)
        L = s.n_levels // 2
        if mid is None:
            s.set_state(torch.tensor(init(s.front_points()[0]), dtype=torch.float64, device="cuda").view(s.front_shape()))
            s.advance(1, L + 1)
            front, tau = s.get_state()
            shift = torch.tensor(np.random.default_rng(2).uniform(0.0, 1e-3, tau.numel()), device="cuda")
            mid = (front, (tau - shift * tau.max() / s.n_levels).contiguous())   # a little below the tents' own times
        s.set_front(*mid)
        s.advance(L + 1, s.n_levels + 1)
        assert s.sync_status()[0] == 0
        fronts.append(s.get_state()[0].cpu().numpy())
        s.set_front(mid[0], tau)   # and the tents' own times: another result
        s.advance(L + 1, s.n_levels + 1)
        fronts.append(s.get_state()[0].cpu().numpy())
    n = np.linalg.norm(fronts[0])
    tol = 1e-12 if precision == "fp64" else 1e-10   # two schedules, as test_gpu_parity's dataflow_matches_levels
    assert np.linalg.norm(fronts[0] - fronts[2]) <= tol * n
    assert np.linalg.norm(fronts[1] - fronts[3]) <= tol * n
    assert np.linalg.norm(fronts[0] - fronts[1]) > 1e-7 * n
