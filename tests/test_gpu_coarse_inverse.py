"""The device inverse of the coarsest level (mg_coarse.cu), alone: meshes of
one level, where an FMG cycle is the exact coarsest solve, against the
oracle's dense solve.  The cell counts sit around the 32-row pivot blocks and
tiles (below one, one, ragged, several, more than a thousand), with every
boundary type, without a Dirichlet face (the shifted form), in cylindrical
form, with lambda and with variable eps.  Tolerance 1e-12 relative: the
condition numbers are below 1e3, rounding 1.1e-16 times a few.  A coefficient
that is not positive is inverted on the host with pivoting, as before: its
solve is compared with numpy's."""
import numpy as np
import pytest

from oracle import Oracle
from synth import workloads as W

pytestmark = pytest.mark.gpu
D, N, P, A = 0, 1, 2, 3


@pytest.fixture(scope="module")
def mg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11370_gb300 import build as B
    B.build()
    import paper_1901_11370_gb300 as m
    return m


def problem(dim, cells, bc, geom=0, eps=False):
    base = tuple(cells) + ((1,) if dim == 2 else ())
    types = tuple(t for b in bc for t in (b if isinstance(b, tuple) else (b, b))) + ((P, P) if dim == 2 else ())
    hi = tuple(c / 10.0 for c in cells) + ((1.0,) if dim == 2 else ())

    def rhs(X, Y, Z):
        return np.cos(3 * X) + np.sin(5 * Y) * np.cos(2 * Z)
    e = (lambda X, Y, Z: 1.0 + 9.0 * (np.sin(4 * X) * np.cos(3 * Y) > 0.2)) if eps else None
    return W.Problem("one_level", dim, 2, geom, base, (0.0,) * 3, hi, types, (0.0,) * 6, np.zeros((0, 4), np.int32),
                     4000, rhs=rhs, eps=e)


CASES = {
    "2x2": lambda: problem(2, (2, 2), (D, D)),
    "30_cells": lambda: problem(2, (6, 10), (D, N)),
    "32_cells_odd": lambda: problem(2, (2, 30), (D, D)),
    "196_cells_eps": lambda: problem(2, (14, 14), (N, D), eps=True),
    "360_cells_periodic": lambda: problem(3, (6, 6, 10), (P, D, N), eps=True),
    "1000_cells": lambda: problem(3, (10, 10, 10), (D, D, N)),
    "singular_neumann": lambda: problem(2, (10, 14), (N, N), eps=True),
    "singular_periodic": lambda: problem(3, (6, 10, 6), (P, P, P)),
    "cylinder": lambda: problem(2, (10, 14), ((A, D), D), geom=1, eps=True),
    "cylinder_singular": lambda: problem(2, (14, 10), ((A, N), N), geom=1),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_one_level_solve_matches_oracle(mg, name):
    p = CASES[name]()
    t = mg.Tree.from_problem(p)
    assert len(t.levels()) == 1
    t.fmg()
    o = Oracle.from_problem(p)
    o.fmg()
    phi, ref = t.get_phi().cpu().numpy(), o.get_phi()
    assert np.abs(phi - ref).max() <= 1e-12 * np.abs(ref).max()


def test_new_coefficients_replace_the_inverse(mg):
    import torch
    p = CASES["196_cells_eps"]()
    t = mg.Tree.from_problem(p)
    t.fmg()
    e = 1.0 + 1.0 / W.leaf_field(p, "eps")
    t.set_eps(torch.from_numpy(e).cuda())
    t.set_phi(torch.zeros(t.n_leaf, dtype=torch.float64, device="cuda"))
    t.fmg()
    o = Oracle.from_problem(p)
    o.set_eps(e)
    o.fmg()
    ref = o.get_phi()
    assert np.abs(t.get_phi().cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


def test_coefficients_of_both_signs_keep_the_pivoting_inverse(mg):
    import torch
    p = problem(2, (6, 6), (D, D))
    t = mg.Tree.from_problem(p)
    e = np.where(np.arange(t.n_leaf) < t.n_leaf // 2, 1.0, -3.0)
    t.set_eps(torch.from_numpy(e).cuda())
    t.fmg()
    r, _ = t.residual_norm()
    f = W.leaf_field(p, "rhs")
    assert r <= 1e-12 * np.sqrt((f * f).mean())
