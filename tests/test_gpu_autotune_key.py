"""What tp_autotune found on one mesh is taken over only where the default
cluster of the dataflow sweep is chosen by the same things, and the default is
among its candidates."""
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


def _solver(n, T, **kw):
    import torch
    import paper_1907_02367_gb300 as pkg
    m = inputs.mesh_square(n, 0.2, seed=2)
    s = pkg.Solver(m.coords, m.elems, m.c, 2, T, inputs.pitch_kappa(m), nrhs=3, **kw)
    s.set_state(torch.tensor(inputs.gaussian_pulse((0.5, 0.5), 0.3)(s.front_points()[0]), dtype=torch.float64,
                             device="cuda").repeat(3, 1, 1).contiguous())
    return s


def test_a_wide_mesh_does_not_set_a_narrow_one(cuda_device):
    """Both meshes have five elements a star on average; the tents of a level
    of the small one leave CTAs for clusters of four, those of the large do not."""
    before = _solver(12, 0.1).schedule()
    assert before["dataflow"] and before["cluster"] == 4
    wide = _solver(22, 0.1)
    assert wide.schedule()["cluster"] == 1
    wide.autotune()
    assert _solver(12, 0.1).schedule() == before
    # nor a context whose plan serves the wave-speed gradient or tracks Neumann walls
    assert _solver(22, 0.1, ckpt_stride=4).schedule()["cluster"] == 1


def test_the_default_is_a_candidate(cuda_device):
    """The tuned sweep is no slower than the default's (25 % for the clock)."""
    import torch
    s = _solver(12, 0.2)
    assert s.schedule()["cluster"] == 4
    front, tau = s.get_state()
    best = 1e9
    for _ in range(4):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        s.set_front(front, tau)
        e0.record()
        s.advance()
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    s.set_front(front, tau)
    chosen, ms = s.autotune()
    print("default 4:", best, "ms; tuned", chosen, ms, "ms")
    assert ms <= 1.25 * best
