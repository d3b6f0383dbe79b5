"""A domain of 2358 x 6 cells in blocks of 6^2: its block counts cannot be
halved, so its coarsest level is 1179 x 3 cells, and the eigenvector solve
along the length has a table of 3 x 1179^2 values.  It takes milliseconds on the
device; one host core took seconds for it in the first solve of a mesh."""
import time

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


@pytest.mark.parametrize("ends", [0, 1, 2])
def test_first_solve_of_a_long_domain(mg, ends):
    import torch
    types = (ends, ends, 0, 1, 2, 2)
    p = W.Problem("channel", 2, 6, 0, (2358, 6, 1), (0.0,) * 3, (393.0, 1.0, 1.0), types, (0.1, -0.2, 0.3, 0.1, 0, 0),
                  np.zeros((0, 4), np.int32), 512, rhs=lambda X, Y, Z: np.cos(0.3 * X) + np.sin(5 * Y))
    t = mg.Tree.from_problem(p)
    l0 = t.levels()[0]
    assert l0["ncell"][:2] == (1179, 3)
    torch.cuda.synchronize()
    start = time.perf_counter()
    _, rel = t.solve(1e-10, 30)
    torch.cuda.synchronize()
    assert time.perf_counter() - start < 2.0
    # the same mesh through the cycles called one by one, which use the dense inverse
    u = mg.Tree.from_problem(p)
    u.fmg()
    r0, _ = mg.Tree.from_problem(p).residual_norm()
    for _ in range(30):
        if u.residual_norm()[0] <= 1e-11 * r0:
            break
        u.vcycle()
    a, b = t.get_phi(), u.get_phi()
    # both residuals are below 1e-10 of the first; Dirichlet across (one side): |A^-1| of about 0.4
    assert rel <= 1e-10 and (a - b).abs().max() <= 1e-8 * b.abs().max()
