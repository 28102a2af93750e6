"""Sums over the functions of degree <= p - 1 alone (Grams of the derivative
terms, moments of alpha, beta and facet data, values of v and sigma): the
smallest count (p = 1: one function), counts below and above a warp and more
Gram pairs than a narrow CTA has threads (2D p = 5: 25 functions, 325 pairs),
with Dirichlet and Neumann data, right-hand sides together and split over a
cluster, against the oracle (the bars of the parity tests: binary64 1e-11,
1e-10 at p = 5 on whole sweeps; mixed 1e-8)."""
import numpy as np
import pytest

from oracle import pitching, tdg
from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,p", [(1, 1), (1, 6), (2, 1), (2, 2), (2, 5), (3, 1), (3, 2), (3, 3)])
@pytest.mark.parametrize("split", [0, 2])
def test_boundary_data(cuda_device, dim, p, split):
    import torch
    import paper_1907_02367_gb300 as pkg
    m = {1: inputs.mesh_interval(4), 2: inputs.mesh_square(3, 0.2, seed=5), 3: inputs.mesh_cube(1, 0.0, seed=3)}[dim]
    T, kappa = {1: 0.4, 2: 0.15, 3: 0.3}[dim], inputs.pitch_kappa(m)
    d = np.arange(1, dim + 1) / np.linalg.norm(np.arange(1, dim + 1))
    walls = inputs.boundary_marker(m, lambda x: x[0] < 1e-12)

    def field(x, t):   # plane wave, values (U, v, sigma)
        ph = 2.5 * (x @ d - t) + 0.3
        return np.concatenate([np.sin(ph)[:, None], -2.5 * np.cos(ph)[:, None], -2.5 * np.cos(ph)[:, None] * d], 1)

    r = pitching.pitch(m.coords, m.elems, m.c, kappa, T)
    ref = tdg.sweep(m.coords, m.elems, m.c, p, r, lambda x: field(x, np.zeros(len(x))), lambda x, t: field(x, t)[:, 1],
                    neumann=lambda x, t, n: field(x, t)[:, 2:] @ n, bnd_type=walls)[0]
    for precision, tol in (("fp64", 1e-10 if p >= 5 else 1e-11), ("mixed", 1e-8)):
        s = pkg.Solver(m.coords, m.elems, m.c, p, T, kappa, nrhs=4, precision=precision, rhs_split=split, bnd_type=walls)
        xt = s.boundary_points()
        nrm, kind = s.boundary_kinds()
        f = field(xt[:, :-1], xt[:, -1])
        g = np.where(kind == 1, (f[:, 2:] * nrm).sum(1), f[:, 1])
        xq, _ = s.front_points()
        scale = torch.arange(1, 5, dtype=torch.float64, device="cuda")
        f0 = torch.tensor(field(xq, np.zeros(len(xq))), device="cuda").view(1, m.n_elem, s.Q, -1)
        s.set_state((f0 * scale.view(-1, 1, 1, 1)).contiguous(), (torch.tensor(g, device="cuda") * scale[:, None]).contiguous())
        s.advance()
        assert s.sync_status() == (0, 0)
        got = (s.get_state()[0] / scale.view(-1, 1, 1, 1)).cpu().numpy()
        for k in range(4):
            rel = np.linalg.norm(got[k] - ref) / np.linalg.norm(ref)
            assert rel <= tol, (precision, k, rel)
