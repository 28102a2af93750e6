"""A front whose times are not the tents' own (tp_set_front), swept by the
dataflow schedule, which finds the times after its wait and assembles again:
with right-hand sides split over a cluster (binary64, mixed with float-float
sums, mixed on the tensor cores), and on meshes with interface and Neumann
facets and boundary data.  The same levels launched one by one take the
front's times from the start."""
import numpy as np
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,walls,nrhs,rhs_split,precision,tensor_cores", [
    (1, "dirichlet", 4, 2, "fp64", True), (2, "dirichlet", 4, 2, "fp64", True), (2, "dirichlet", 32, 8, "fp64", True),
    (2, "dirichlet", 32, 2, "mixed", True), (2, "dirichlet", 8, 4, "mixed", False), (3, "dirichlet", 64, 4, "mixed", True),
    (2, "mixed walls", 1, 1, "fp64", True), (2, "mixed walls", 4, 2, "fp64", True), (2, "mixed walls", 3, 1, "mixed", True),
    (2, "mixed walls", 32, 2, "mixed", True), (3, "mixed walls", 8, 4, "fp64", True)])
def test_split_columns_from_other_times(cuda_device, dim, walls, nrhs, rhs_split, precision, tensor_cores):
    import torch
    import paper_1907_02367_gb300 as pkg
    m = {1: inputs.mesh_interval(9), 2: inputs.mesh_square(5, 0.2, seed=4), 3: inputs.mesh_cube(2, 0.1, seed=4)}[dim]
    bnd = None
    if walls == "mixed walls":   # two materials, a Neumann side, data on every wall
        m.c[m.coords[m.elems].mean(axis=1)[:, 0] > 0.5] = 1.3
        bnd = inputs.boundary_marker(m, lambda x: x[dim - 1] < 1e-12)
    p, T, kappa = 3, {1: 0.4, 2: 0.3, 3: 0.2}[dim], inputs.pitch_kappa(m)
    rng = np.random.default_rng(nrhs)
    inits = [inputs.gaussian_pulse(rng.uniform(0.3, 0.7, dim), 0.3) for _ in range(nrhs)]
    fronts, mid = [], None
    for schedule in ("dataflow", "levels"):
        s = pkg.Solver(m.coords, m.elems, m.c, p, T, kappa, nrhs=nrhs, rhs_split=rhs_split, precision=precision,
                       schedule=schedule, bnd_type=bnd, tensor_cores=tensor_cores)
        assert s.schedule()["rhs_split"] == rhs_split
        assert s.tensor_cores_used() == (precision == "mixed" and rhs_split > 1 and tensor_cores)
        x, _ = s.front_points()
        f0 = torch.tensor(np.stack([f(x) for f in inits]), dtype=torch.float64, device="cuda").contiguous()
        g = None
        if bnd is not None:
            xt = s.boundary_points()
            g = torch.tensor(np.stack([np.sin(2.0 * xt[:, 0] + r) * xt[:, -1] for r in range(nrhs)]), dtype=torch.float64,
                             device="cuda").contiguous()
        L = s.n_levels // 2
        s.set_state(f0, g)
        if mid is None:
            s.advance(1, L + 1)
            front, tau = s.get_state()
            shift = torch.tensor(np.random.default_rng(2).uniform(0.0, 1e-3, tau.numel()), device="cuda")
            mid = (front, (tau - shift * tau.max() / s.n_levels).contiguous())   # a little below the tents' own times
        for times in (mid[1], tau):
            s.set_front(front, times)
            s.advance(L + 1, s.n_levels + 1)
            assert s.sync_status() == (0, 0)
            fronts.append(s.get_state()[0])
    n = float(fronts[0].norm())
    # another order of the sums over the points (other clusters): the parity bars of whole sweeps
    tol = 1e-11 if precision == "fp64" else 1e-9
    assert float((fronts[0] - fronts[2]).norm()) <= tol * n
    assert float((fronts[1] - fronts[3]).norm()) <= tol * n
    assert float((fronts[0] - fronts[1]).norm()) > 1e-7 * n
