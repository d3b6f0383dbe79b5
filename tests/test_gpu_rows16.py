"""The quarter-row FP32 sweep of 16^3 blocks (variant 0 there) pinned on every
level, against the plain-load sweep (variant 1) after the same
FP32 cycles and by the oracle's residual at convergence.  One FP32 cycle of
the two differs by rounding only: the defect correction's phi after two outer
steps agrees to 1e-5 of the second correction's size, a few hundred FP32 ulps
over some fifty dependent half-sweeps.  Constant and variable eps, refinement
faces, every boundary type, lambda, fewer blocks than stages and more than
one block per SM."""
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


def box(nblk, bc, eps=False, refine=None):
    base = tuple(16 * q for q in nblk)
    types = tuple(t for b in bc for t in (b, b))
    e = (lambda X, Y, Z: np.where((X - 0.7) ** 2 + (Y - 0.6) ** 2 + (Z - 0.5) ** 2 < 0.2, 50.0, 1.0)) if eps else None
    return W.Problem("box16", 3, 16, 0, base, (0.0,) * 3, tuple(b / 32.0 for b in base), types,
                     (0.1, -0.2, 0.3, 0.0, 0.2, -0.1), np.zeros((0, 4), np.int32) if refine is None else refine, 512,
                     rhs=lambda X, Y, Z: np.cos(2 * np.pi * X) * np.sin(2 * np.pi * Y + 0.3) + np.cos(2 * np.pi * Z), eps=e)


AMR = W.refine_spheres(3, 16, (64,) * 3, (0,) * 3, (2,) * 3, (1.0, 0.9, 1.1), (0.7,))
CASES = {
    "one_block_wide": lambda: box((2, 2, 2), (D, N, D)),
    "periodic": lambda: box((2, 4, 2), (P, P, D)),
    "vareps": lambda: box((4, 2, 2), (N, D, P), eps=True),
    "many_blocks": lambda: box((8, 6, 8), (D, D, N)),
    "amr": lambda: box((4, 4, 4), (D, N, D), refine=AMR),
    "amr_vareps": lambda: box((4, 4, 4), (D, N, D), eps=True, refine=AMR),
}


def outer(mg, p, variant, n, **kw):
    t = mg.Tree.from_problem(p)
    t.set_sweep_variant(variant, precision=mg.MG_FP32_DC)
    assert any(t.sweep_variant(l, mg.MG_FP32_DC) == variant for l in range(len(t.levels())))
    t.solve(1e-13, n, precision=mg.MG_FP32_DC, raise_on_fail=False, **kw)
    return t.get_phi().cpu().numpy()


@pytest.mark.parametrize("name", sorted(CASES))
def test_equals_the_plain_sweep_and_converges(mg, name):
    p = CASES[name]()
    a, b, one = outer(mg, p, 0, 2), outer(mg, p, 1, 2), outer(mg, p, 1, 1)
    assert np.abs(a - b).max() <= 1e-5 * np.abs(b - one).max() + 1e-7 * np.abs(one).max()
    res = {}
    for variant in (1, 0):  # whether the V-cycle contracts on a mesh is the method's matter: both alike
        t = mg.Tree.from_problem(p)
        t.set_sweep_variant(variant, precision=mg.MG_FP32_DC)
        res[variant] = t.solve(1e-10, 60, precision=mg.MG_FP32_DC, raise_on_fail=False)
    assert (res[0][1] <= 1e-10) == (res[1][1] <= 1e-10), res
    assert abs(res[0][0] - res[1][0]) <= 1, res
    if res[0][1] > 1e-10:
        return
    o = Oracle.from_problem(p)
    r0, _ = o.residual_norm()
    o.set_phi(t.get_phi().cpu().numpy())
    r1, _ = o.residual_norm()
    assert r1 <= 1.05e-10 * r0


def test_an_expired_wait_reports_timeout(mg):
    p = CASES["many_blocks"]()
    t = mg.Tree.from_problem(p)
    t.set_sweep_variant(0, precision=mg.MG_FP32_DC)
    t.set_wait_limit(0)
    with pytest.raises(mg.MGError) as e:
        t.solve(1e-10, 2, precision=mg.MG_FP32_DC)
    assert e.value.code == -6


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp32_cycles_contract_like_fp64_cycles(mg, name):
    """The FP32 sweeps and transfers of 16^3 blocks inside the defect
    correction against plain FP64 cycles: while the residual is far above
    FP32 rounding (two outer steps of one cycle from a reduction of about 0.1
    a cycle), the defect after each is the FP64 cycle's to 1 %.  A wrong
    neighbour, weight or ghost in a transfer changes the contraction."""
    p = CASES[name]()
    rel = {}
    for prec in (mg.MG_FP64, mg.MG_FP32_DC):
        t = mg.Tree.from_problem(p)
        _, rel[prec] = t.solve(1e-14, 2, fmg_first=False, precision=prec, raise_on_fail=False)
    if len(p.refine):  # refinement ghosts of the correction cycle lag differently
        assert rel[mg.MG_FP32_DC] <= 2 * rel[mg.MG_FP64]
    else:
        assert abs(rel[mg.MG_FP32_DC] - rel[mg.MG_FP64]) <= 0.01 * rel[mg.MG_FP64]
