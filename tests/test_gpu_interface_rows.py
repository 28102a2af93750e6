"""The U-values of an interface facet are evaluated in rows: the + side's
points, then the - side's.  With Q > 16 points per facet taken by one CTA the
- side's rows lie in other warps than the threads that wrote their points.
The wave-speed gradient with split right-hand sides takes every facet point
in each CTA; unsplit, four CTAs share them (7 points each at p = 4).  Both
sum the same terms, in another order (1e-12 of the largest entry, as the
p = 2 comparison of test_gpu_speed_gradient)."""
import numpy as np
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_gradient_split_equals_unsplit_at_p4(cuda_device, precision):
    import torch
    import paper_1907_02367_gb300 as pkg
    m = inputs.mesh_square(6, 0.2, seed=13)
    cen = m.coords[m.elems].mean(axis=1)
    m.c[:] = np.where(np.linalg.norm(cen - 0.5, axis=1) < 0.3, 1.5, 1.0)
    p, T, kappa = 4, 0.12, inputs.pitch_kappa(m)
    tents = pkg.Tents(m.coords, m.elems, m.c, kappa, T)
    rng = np.random.default_rng(3)
    f0 = rng.standard_normal((8, m.n_elem, (p + 1) ** 2, 4))
    lam = rng.standard_normal(f0.shape)
    up = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda").contiguous()  # noqa: E731

    def grad(cols, split):
        s = pkg.Solver(m.coords, m.elems, m.c, p, T, kappa, tents=tents, nrhs=len(cols), precision=precision,
                       ckpt_stride=4, rhs_split=split)
        s.set_state(up(f0[cols]))
        g = s.speed_gradient(up(lam[cols])).cpu().numpy()
        assert s.sync_status() == (0, 0)
        return g

    g_cols = sum(grad([r], 1) for r in range(8))
    g_split = grad(list(range(8)), 4)
    tol = 1e-12 if precision == "fp64" else 1e-8   # mixed: the two forward sweeps differ in rounding (the path's bound)
    assert np.abs(g_split - g_cols).max() <= tol * np.abs(g_cols).max()
