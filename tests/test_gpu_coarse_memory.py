"""Device memory of a mesh with constant coefficients: the scratch of the
coarsest inverse (as large as the inverse) is needed once, when the mesh is
made, and does not stay.  A coefficient set later is inverted all the same."""
import numpy as np
import pytest

from synth import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11370_gb300 import build as B
    B.build()
    import paper_1901_11370_gb300 as m
    return m


def test_inverse_scratch_is_given_back(mg):
    import torch
    p = W.Problem("one_level", 2, 2, 0, (78, 82, 1), (0.0,) * 3, (1.0,) * 3, (0,) * 4 + (2,) * 2, (0.0,) * 6,
                  np.zeros((0, 4), np.int32), 10000, rhs=lambda X, Y, Z: X)
    first = mg.Tree.from_problem(p)  # loads the kernels
    assert len(first.levels()) == 1
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    t = mg.Tree.from_problem(p)
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    inverse = 8 * 6396 ** 2  # 39 x 41 blocks: no coarser level
    assert free0 - free1 <= 1.25 * inverse  # fields and tables take under 2 MB; the rest is granularity
    t.fmg()
    first.fmg()
    assert torch.equal(t.get_phi(), first.get_phi())
    e = torch.full_like(first.get_phi(), 2.0)
    for q in (t, first):
        q.set_eps(e)
        q.set_phi(torch.zeros_like(e))
        q.fmg()
    assert torch.equal(t.get_phi(), first.get_phi())
    r, _ = t.residual_norm()
    assert r <= 1e-9 * np.sqrt((W.leaf_field(p, "rhs") ** 2).mean())  # u sqrt(n) kappa, kappa 4e3: 4e-11
