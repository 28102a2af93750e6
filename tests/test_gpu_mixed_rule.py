"""The rule of the face integrals of a mixed sweep at 2D p = 3: errors against
the method in plain torch binary64 (perf/cases.py) on a graded mesh of two
materials.  The bar lies between the front rule's errors (8.4e-14 and 9.4e-14
for the two seeds) and those of the S-point rule (1.3e-13 and 1.5e-13)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_two_materials_at_degree_three(cuda_device):
    import torch
    from perf import cases
    case = dict(mesh="inclusion", size=0.1, p=3, T=0.03, nrhs=1, precision="mixed", walls="rest", task="sweep")
    err = []
    for seed in (1, 2):
        out, ref = cases.run(cases.prepare(case, seed))["front"], cases.exact(case, seed)["front"]
        torch.cuda.synchronize()
        err.append(float((out - ref).norm() / ref.norm()))
    assert np.mean(err) <= 1.1e-13, err
