"""Several right-hand sides in one CTA's charge (not split): which rule of the
face integrals and which cluster they take depends on their number.  Every
column is the sweep of that column alone, and 16 of them cost a few sweeps of
one (their data pass the rule's tables only where that is less work)."""
import numpy as np
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


def _solver(m, p, T, nrhs, precision, **kw):
    import paper_1907_02367_gb300 as pkg
    return pkg.Solver(m.coords, m.elems, m.c, p, T, inputs.pitch_kappa(m), nrhs=nrhs, precision=precision, rhs_split=1, **kw)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,p", [(2, 2), (2, 3), (2, 4), (2, 5), (3, 1), (3, 2), (3, 3)])
def test_columns_on_both_sides_of_the_rule(cuda_device, dim, p, precision):
    """One column to 5 and 9: the S-point rule, the front rule, kept U-values
    over other clusters; two materials in 2D."""
    import torch
    m = inputs.mesh_square(4, 0.2, seed=6) if dim == 2 else inputs.mesh_cube(2, 0.1, seed=4)
    if dim == 2:
        m.c[m.coords[m.elems].mean(axis=1)[:, 0] > 0.5] = 1.3
    T = 0.1
    one = _solver(m, p, T, 1, precision)
    x, _ = one.front_points()
    rng = np.random.default_rng(p)
    f = torch.tensor(np.stack([inputs.gaussian_pulse(rng.uniform(0.3, 0.7, dim), rng.uniform(0.2, 0.4))(x) for _ in range(9)]),
                     dtype=torch.float64, device="cuda").contiguous()
    ref = []
    for r in range(9):
        one.set_state(f[r].contiguous())
        one.advance()
        ref.append(one.get_state()[0][0])
    # other rules and orders of the sums: the parity bars of whole sweeps
    tol = {"fp64": 1e-10 if p == 5 else 1e-11, "mixed": 1e-8}[precision]
    for nrhs in (2, 3, 4, 5, 9):
        s = _solver(m, p, T, nrhs, precision)
        s.set_state(f[:nrhs].contiguous())
        s.advance()
        assert s.sync_status() == (0, 0)
        got = s.get_state()[0]
        for r in range(nrhs):
            assert float((got[r] - ref[r]).norm()) <= tol * float(ref[r].norm()), (nrhs, r)


@pytest.mark.parametrize("kind,n,p", [("square", 20, 3), ("cube", 6, 2)])
def test_sixteen_columns_cost_a_few_sweeps(cuda_device, kind, n, p):
    """The tents, their matrices and inverses are shared: 16 columns in binary64
    take at most 5.5 times one column's sweep (7 and more where every column's
    data passed the tables of the S-point rule, 3.5 and 4 without)."""
    import torch
    m = inputs.mesh_square(n, 0.2, seed=2) if kind == "square" else inputs.mesh_cube(n, 0.1, seed=4)
    ms = []
    for nrhs in (1, 16):
        s = _solver(m, p, (1.6 if kind == "square" else 0.9) / n, nrhs, "fp64")
        f = torch.tensor(inputs.gaussian_pulse([0.5] * m.dim, 0.3)(s.front_points()[0]), dtype=torch.float64, device="cuda")
        f = f.repeat(nrhs, 1, 1).contiguous()
        best = 1e9
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            s.set_state(f)
            e0.record()
            s.advance()
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        ms.append(best)
    assert ms[1] <= 5.5 * ms[0], ms
