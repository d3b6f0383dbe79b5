"""The device inverse of a coarsest level without Dirichlet faces, over the
size of the coefficient: one level, where an FMG cycle is the exact coarsest
solve, so the residual it leaves is rounding.  An explicit inverse leaves at
most a few u sqrt(n) kappa of the right-hand side (u = 1.1e-16, n at most 840
cells, condition numbers below 1e3, rounding errors that add up like a random
walk): 1e-11.  A solve that is exact at eps of order one is as
exact at 1e-16 or 1e16 of it: the operator is only scaled."""
import numpy as np
import pytest

from synth import workloads as W

pytestmark = pytest.mark.gpu
N, P, A = 1, 2, 3


@pytest.fixture(scope="module")
def mg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11370_gb300 import build as B
    B.build()
    import paper_1901_11370_gb300 as m
    return m


def problem(dim, cells, bc, geom=0):
    base = tuple(cells) + ((1,) if dim == 2 else ())
    types = tuple(t for b in bc for t in (b if isinstance(b, tuple) else (b, b))) + ((P, P) if dim == 2 else ())
    hi = tuple(c / 10.0 for c in cells) + ((1.0,) if dim == 2 else ())
    return W.Problem("one_level", dim, 2, geom, base, (0.0,) * 3, hi, types, (0.0,) * 6, np.zeros((0, 4), np.int32), 4000)


MESHES = {
    "3d_neumann": lambda: problem(3, (6, 10, 14), (N, N, N)),
    "2d_periodic_neumann": lambda: problem(2, (10, 14), (P, N)),
    "cylinder": lambda: problem(2, (14, 10), ((A, N), N), geom=1),
}


@pytest.mark.parametrize("scale", [1e-16, 8.85e-12, 1e-8, 1.0, 1e8, 1e12, 1e16])
@pytest.mark.parametrize("mesh", sorted(MESHES))
def test_singular_solve_is_exact_at_every_scale(mg, mesh, scale):
    import torch
    p = MESHES[mesh]()
    X = W.leaf_cell_centres(p)[0]
    vol = X if p.geom else np.ones_like(X)  # 2 pi r dr dz up to a factor
    rng = np.random.default_rng(7)
    f = rng.standard_normal(len(X))
    f -= (vol * f).sum() / vol.sum()
    t = mg.Tree.from_problem(p)
    assert len(t.levels()) == 1
    t.set_eps(torch.from_numpy(scale * rng.uniform(1.0, 10.0, len(X))).cuda())
    t.set_rhs(torch.from_numpy(f).cuda())
    t.fmg()
    r, _ = t.residual_norm()
    assert r <= 1e-11 * np.sqrt((vol * f * f).sum() / vol.sum())
    phi = t.get_phi().cpu().numpy()
    assert abs((vol * phi).sum()) <= 1e-11 * (vol * np.abs(phi)).sum()
