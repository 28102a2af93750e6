"""Numbers of right-hand sides that the shared memory holds in one group, but
not together with the S-point rule's buffers: they stay in one group (every
group assembles every tent again), the wave-speed gradient (one group only)
accepts them, and the columns are those of sweeps on their own."""
import numpy as np
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


def _mesh(name):
    if name == "interval":   # two materials
        m = inputs.mesh_interval(8)
        m.c[:4] = 0.7
        return m, 0.2
    if name == "square":
        return inputs.mesh_square(4, 0.2, seed=6), 0.1
    return inputs.mesh_cube(2, 0.1, seed=4), 0.1   # one interior vertex with 24 elements


def _solver(name, p, nrhs, precision, **kw):
    import paper_1907_02367_gb300 as pkg
    m, T = _mesh(name)
    return m, pkg.Solver(m.coords, m.elems, m.c, p, T, inputs.pitch_kappa(m), nrhs=nrhs, precision=precision, **kw)


def _fronts(s, dim, nrhs):
    import torch
    x, _ = s.front_points()
    rng = np.random.default_rng(nrhs)
    return torch.tensor(np.stack([inputs.gaussian_pulse(rng.uniform(0.3, 0.7, dim), rng.uniform(0.2, 0.4))(x)
                                  for _ in range(nrhs)]), dtype=torch.float64, device="cuda").contiguous()


@pytest.mark.parametrize("name,p,nrhs,precision", [("cube", 3, 29, "fp64"), ("cube", 3, 31, "mixed"), ("cube", 3, 26, "fp64"),
                                                   ("square", 5, 37, "fp64"), ("square", 5, 41, "mixed")])
def test_columns_of_one_group(cuda_device, name, p, nrhs, precision):
    m, s = _solver(name, p, nrhs, precision)
    assert s.schedule()["rhs_groups"] == 1
    f = _fronts(s, m.dim, nrhs)
    s.set_state(f)
    s.advance()
    assert s.sync_status() == (0, 0)
    got = s.get_state()[0]
    _, one = _solver(name, p, 1, precision)
    # another rule of the face integrals, another order of the sums: the parity bars of whole sweeps
    tol = {"fp64": 1e-10 if p == 5 else 1e-11, "mixed": 1e-8}[precision]
    for r in (0, nrhs // 2, nrhs - 1):
        one.set_state(f[r].contiguous())
        one.advance()
        ref = one.get_state()[0][0]
        assert float((got[r] - ref).norm()) <= tol * float(ref.norm()), r


@pytest.mark.parametrize("name,p,nrhs,precision", [("cube", 3, 16, "fp64"), ("cube", 3, 17, "mixed"), ("cube", 3, 19, "fp64"),
                                                   ("square", 5, 19, "fp64"), ("interval", 8, 58, "mixed")])
def test_gradient_of_one_group(cuda_device, name, p, nrhs, precision):
    import torch
    m, s = _solver(name, p, nrhs, precision, ckpt_stride=4)
    assert s.schedule()["rhs_groups"] == 1
    f = _fronts(s, m.dim, nrhs)
    lam = f.flip(0).contiguous()
    s.set_state(f)
    s.advance()
    got = s.speed_gradient(lam)
    assert s.sync_status() == (0, 0)
    _, one = _solver(name, p, 1, precision, ckpt_stride=4)
    ref = torch.zeros_like(got)
    for r in range(nrhs):
        one.set_state(f[r].contiguous())
        one.advance()
        ref += one.speed_gradient(lam[r].contiguous())
    tol = {"fp64": 1e-10, "mixed": 1e-8}[precision]
    assert float((got - ref).norm()) <= tol * float(ref.norm())
