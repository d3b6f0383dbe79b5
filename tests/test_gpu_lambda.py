"""lambda > 0 (the Helmholtz term) in the solves' cluster kernel and in the
device inverse of the coarsest level, against the oracle: after the same
cycles at 1e-12 relative, as for lambda = 0 (the term adds one product a
cell; it lowers the condition number).  Both coarsest solves of the kernel (by
eigenvectors from 400 cells on, by the dense inverse below), constant and
variable eps, and the meshes that are singular without lambda."""
import numpy as np
import pytest

from oracle import Oracle
from synth import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12
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


def box(dim, nblk, n, bc, eps=False, coarse_max=512, refine=None):
    base = tuple(q * n for q in nblk) + ((1,) if dim == 2 else ())
    hi = tuple(b / 16.0 for b in base[:dim]) + ((1.0,) if dim == 2 else ())
    types = tuple(t for b in bc for t in (b, b)) + ((P, P) if dim == 2 else ())

    def rhs(X, Y, Z):
        return np.cos(2 * np.pi * X) * np.sin(2 * np.pi * Y + 0.3) + (np.cos(2 * np.pi * Z) if dim == 3 else 0.0)
    e = (lambda X, Y, Z: 1.5 + np.sin(2 * np.pi * X) * np.cos(2 * np.pi * Y)) if eps else None
    return W.Problem("box", dim, n, 0, base, (0.0,) * 3, hi, types, (0.1, -0.2, 0.3, 0.0, 0.2, -0.1),
                     np.zeros((0, 4), np.int32) if refine is None else refine, coarse_max, rhs=rhs, eps=e)


SPHERE = W.refine_spheres(3, 8, (32,) * 3, (0,) * 3, (2,) * 3, (1.0,) * 3, (0.6,))
CASES = {  # problem, lambda, cells of the coarsest level
    "2d_eigenvectors": (lambda: box(2, (5, 7), 8, (D, N), coarse_max=600), 7.0, 560),
    "2d_dense": (lambda: box(2, (5, 7), 8, (D, N)), 7.0, 140),
    "2d_neumann": (lambda: box(2, (6, 4), 8, (N, N)), 40.0, 384),
    "2d_periodic_eigenvectors": (lambda: box(2, (10, 14), 8, (P, P), coarse_max=600), 0.5, 560),
    "2d_vareps": (lambda: box(2, (6, 4), 8, (N, N), eps=True), 40.0, 384),
    "3d_eigenvectors": (lambda: box(3, (7, 5, 5), 8, (D, N, D), coarse_max=1500), 7.0, 1400),
    "3d_dense_periodic": (lambda: box(3, (2, 2, 8), 4, (P, P, P), coarse_max=64), 3.0, 32),
    "3d_amr": (lambda: box(3, (4, 4, 4), 8, (N, N, N), refine=SPHERE), 20.0, 512),
    "3d_amr_vareps": (lambda: box(3, (4, 4, 4), 8, (D, N, N), eps=True, refine=SPHERE), 20.0, 512),
}


def both(mg, p, helm):
    import torch
    args = (p.dim, p.N, p.geom, p.bc_type, p.bc_val, p.base, p.lo, p.hi, p.refine, p.coarse_max)
    t, o = mg.Tree(*args, helm=helm), Oracle(*args, helm=helm)
    f = W.leaf_field(p, "rhs")
    if p.eps is not None:
        e = W.leaf_field(p, "eps")
        t.set_eps(torch.from_numpy(e).cuda())
        o.set_eps(e)
    t.set_rhs(torch.from_numpy(f).cuda())
    o.set_rhs(f)
    return t, o


@pytest.mark.parametrize("jacobi", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_cycles_match_the_oracle(mg, name, jacobi):
    make, helm, nc = CASES[name]
    t, o = both(mg, make(), helm)
    l0 = t.levels()[0]
    assert l0["nb"] * l0["n"] ** t.dim == nc and len(t.levels()) > 1
    t.solve(1e-14, 3, raise_on_fail=False, smoother=jacobi)
    o.set_smoother(jacobi)
    o.residual_norm()
    o.fmg()
    for _ in range(2):
        o.residual_norm()
        o.vcycle(1)
    ref = o.get_phi()
    assert np.abs(t.get_phi().cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("name", sorted(CASES))
def test_mixed_precision_reaches_tolerance(mg, name):
    make, helm, _ = CASES[name]
    t, o = both(mg, make(), helm)
    t.solve(1e-10, 60, precision=mg.MG_FP32_DC, inner_cycles=2)
    r0, _ = o.residual_norm()
    o.set_phi(t.get_phi().cpu().numpy())
    r1, _ = o.residual_norm()
    assert r1 <= 1.05e-10 * r0


@pytest.mark.parametrize("eps", [False, True])
@pytest.mark.parametrize("bc", [(D, N), (N, N), (P, P)])
def test_one_level_solve_matches_the_oracle(mg, bc, eps):
    p = box(2, (5, 7), 2, bc, eps=eps)
    t, o = both(mg, p, 7.0)
    assert len(t.levels()) == 1
    t.fmg()
    o.fmg()
    ref = o.get_phi()
    assert np.abs(t.get_phi().cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()
