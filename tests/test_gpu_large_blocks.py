"""Prolongation into the largest 2D blocks the cycles take (156^2 in FP64,
220^2 in FP32: the restriction's shared memory bounds them).  The first size
of each list still holds the box of parent differences beside the cells in a
CTA's 227 KB, the others do not.  FP64 blocks are compared with the oracle
after an FMG and a V-cycle at 1e-12 relative, as the other cycles; FP32 blocks
by the oracle's residual of the converged solution."""
import numpy as np
import pytest

from oracle import Oracle
from synth import workloads as W

pytestmark = pytest.mark.gpu
D, N, P = 0, 1, 2


@pytest.fixture(scope="module")
def mg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11370_gb300 import build as B
    B.build()
    import paper_1901_11370_gb300 as m
    return m


def box(n):
    return W.Problem("box", 2, n, 0, (2 * n, 2 * n, 1), (0.0,) * 3, (1.0,) * 3, (D, D, N, D, P, P),
                     (0.1, -0.2, 0.3, 0.0, 0.0, 0.0), np.zeros((0, 4), np.int32), 512,
                     rhs=lambda X, Y, Z: np.cos(3 * X) * np.sin(5 * Y))


@pytest.mark.parametrize("n", [148, 152, 156])
def test_2d_fp64_blocks_match_the_oracle(mg, n):
    p = box(n)
    t = mg.Tree.from_problem(p)
    t.fmg()
    t.vcycle()
    o = Oracle.from_problem(p)
    o.fmg()
    o.vcycle()
    ref = o.get_phi()
    assert np.abs(t.get_phi().cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("n", [212, 216, 220])
def test_2d_fp32_blocks_converge(mg, n):
    p = box(n)
    t = mg.Tree.from_problem(p)
    t.solve(1e-10, 40, precision=mg.MG_FP32_DC)
    o = Oracle.from_problem(p)
    r0, _ = o.residual_norm()
    o.set_phi(t.get_phi().cpu().numpy())
    r1, _ = o.residual_norm()
    assert r1 <= 1.05e-10 * r0
