"""The dataflow sweep starts with rank 0 of every cluster handing the first tent
to the other CTAs through their shared memory, after a barrier by which all of
them run.  Many short sweeps, with more clusters than tents, over clusters of
every size: each the same bits."""
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,split", [(1, 2), (1, 4), (1, 8), (2, 2), (2, 8), (3, 4)])
def test_short_sweeps_repeat(cuda_device, dim, split, precision):
    import torch
    import paper_1907_02367_gb300 as pkg
    m = {1: inputs.mesh_interval(4), 2: inputs.mesh_square(2, 0.1, seed=3), 3: inputs.mesh_cube(1, 0.0, seed=3)}[dim]
    s = pkg.Solver(m.coords, m.elems, m.c, 2, 0.1, inputs.pitch_kappa(m), nrhs=16, rhs_split=split, precision=precision)
    assert s.schedule()["dataflow"] and s.schedule()["cluster"] == split
    f = torch.tensor(inputs.gaussian_pulse([0.4] * dim, 0.3)(s.front_points()[0]), dtype=torch.float64, device="cuda")
    f = f.repeat(16, 1, 1).contiguous()
    first = None
    for _ in range(40):
        s.set_state(f)
        s.advance()
        out = s.get_state()[0]
        assert s.sync_status() == (0, 0)
        first = out if first is None else first
        assert torch.equal(out, first)
