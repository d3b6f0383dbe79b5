"""Small coarsest levels: which inversion they take (up to 80 cells the host's),
and that both give the oracle's solve, at 1e-12 relative (condition numbers
below 1e3): one level, where an FMG cycle is the exact coarsest solve, and
meshes of several levels, whose coarsest coefficients lie before the others
(FMG and a V-cycle)."""
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


def problem(n, cells):
    return W.Problem("small", 2, n, 0, cells + (1,), (0.0,) * 3, (cells[0] / 10.0, cells[1] / 10.0, 1.0),
                     (D, N, D, D, P, P), (0.1, 0.2, 0.3, 0.4, 0, 0), np.zeros((0, 4), np.int32), 64 if n == 8 else 4000,
                     rhs=lambda X, Y, Z: np.cos(3 * X) + np.sin(5 * Y))


@pytest.mark.parametrize("n, cells, nc", [(2, (2, 2), 4), (2, (6, 10), 60), (2, (2, 38), 76), (2, (6, 14), 84),
                                          (2, (10, 10), 100), (8, (64, 64), 64), (8, (96, 32), 48), (8, (80, 64), 20),
                                          (8, (72, 88), 99)])
def test_small_coarsest_levels(mg, n, cells, nc):
    import torch
    p = problem(n, cells)
    t, o = mg.Tree.from_problem(p), Oracle.from_problem(p)
    l0 = t.levels()[0]
    assert l0["nb"] * l0["n"] ** 2 == nc
    rng = np.random.default_rng(2)
    for eps in (False, True, True):
        if eps:
            e = 1.0 + 9.0 * rng.random(t.n_leaf)
            t.set_eps(torch.from_numpy(e).cuda())
            t.set_phi(torch.zeros(t.n_leaf, dtype=torch.float64, device="cuda"))
            o.set_eps(e)
            o.set_phi(np.zeros(t.n_leaf))
        t.fmg()
        o.fmg()
        if len(t.levels()) > 1:
            t.vcycle()
            o.vcycle()
        ref = o.get_phi()
        assert np.abs(t.get_phi().cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


def test_the_device_inversion_starts_above_80_cells(mg):
    """set_eps on one level: beside what every mesh launches, the rows, two
    kernels a pivot block of 32 rows and the store."""
    import torch
    n = {}
    for cells in ((2, 2), (6, 10), (2, 38), (6, 14), (10, 10)):
        t = mg.Tree.from_problem(problem(2, cells))
        assert len(t.levels()) == 1
        e = torch.ones(t.n_leaf, dtype=torch.float64, device="cuda")
        t.set_eps(e)
        n0 = t.launch_count()
        t.set_eps(e)
        n[cells[0] * cells[1]] = t.launch_count() - n0
    assert n[60] == n[76] == n[4] and n[84] == n[4] + 8 and n[100] == n[4] + 10, n
