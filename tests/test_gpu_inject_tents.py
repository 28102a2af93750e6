"""tp_inject_wait holds one injection per tent: a second tent's does not
replace the first, and clearing one tent leaves the others (TP_ERR_TIMEOUT by
the bounded waits; cleared, the sweep is the one without injections)."""
import numpy as np
import pytest

from paper_1907_02367_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_injections_are_per_tent(cuda_device):
    import torch
    import paper_1907_02367_gb300 as pkg
    from paper_1907_02367_gb300 import _binding as B
    w = inputs.workload("plane1d")
    m = w.mesh
    s = pkg.Solver(m.coords, m.elems, m.c, w.p, w.T, w.kappa)
    f0 = torch.tensor(w.init(s.front_points()[0]), dtype=torch.float64, device="cuda").reshape(s.front_shape()).contiguous()
    lev = s.tents.export()["level"]
    first, second, third = (int(np.nonzero(lev == L)[0][0]) for L in (3, 4, 5))

    def status():
        s.set_state(f0)
        s.advance()
        return s.sync_status()

    assert status() == (0, 0)
    clean = s.get_state()[0]
    s.set_limits(max_polls=4096)
    s.inject_wait(first, 1000)
    s.inject_wait(second, 1000)
    s.inject_wait(second, 0)      # the first tent's stays
    st, info = status()
    assert st == B.TP_ERR_TIMEOUT and info >= first
    s.inject_wait(third, 0)       # never injected: nothing changes
    assert status()[0] == B.TP_ERR_TIMEOUT
    s.inject_wait(first, 0)
    assert status() == (0, 0)
    assert torch.equal(s.get_state()[0], clean)
