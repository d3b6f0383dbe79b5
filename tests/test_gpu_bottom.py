"""The cluster kernel that runs the lower levels of a cycle inside the solves
(mg_solve, the adjoint): FMG and V-cycles through it against the FP64 oracle
after the same number of cycles, at 1e-12 relative as for the
launch-by-launch cycle (the arithmetic is the same up to rounding order).
The meshes vary what the kernel's cut depends on: 2D and 3D, cubes and long
boxes, odd block counts, every boundary type (periodic along and across the
cut), refinement above the base grid, variable eps, lambda > 0, the Jacobi
smoother, a per-level schedule, one level above the coarsest."""
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


def box(dim, nblk, n, bc, vals=(0.1, -0.2, 0.3, 0.0, 0.2, -0.1), eps=False, coarse_max=512, refine=None):
    base = tuple(q * n for q in nblk) + ((1,) if dim == 2 else ())
    hi = tuple(b / 16.0 for b in base[:dim]) + ((1.0,) if dim == 2 else ())
    types = tuple(t for b in bc for t in (b, b)) + ((P, P) if dim == 2 else ())

    def rhs(X, Y, Z):
        return np.cos(2 * np.pi * X) * np.sin(2 * np.pi * Y + 0.3) + (np.cos(2 * np.pi * Z) if dim == 3 else 0.0)
    e = (lambda X, Y, Z: 1.5 + np.sin(2 * np.pi * X) * np.cos(2 * np.pi * Y)) if eps else None
    return W.Problem("box", dim, n, 0, base, (0.0,) * 3, hi, types, vals,
                     np.zeros((0, 4), np.int32) if refine is None else refine, coarse_max, rhs=rhs, eps=e)


CASES = {
    "poisson2d_64": (lambda: W.cfg1_poisson2d(n=64, N=8), {}),
    "2d_long_mixed": (lambda: box(2, (12, 2), 8, (D, N)), {}),
    "2d_odd_blocks_periodic_y": (lambda: box(2, (9, 6), 8, (D, P), coarse_max=64), {}),
    "2d_periodic_x": (lambda: box(2, (4, 8), 8, (P, D)), {}),
    "3d_odd_blocks": (lambda: box(3, (5, 3, 3), 8, (D, N, D)), {}),
    "3d_long_z_periodic_z": (lambda: box(3, (2, 2, 8), 4, (D, N, P), coarse_max=64), {}),
    "3d_periodic_xy": (lambda: box(3, (4, 2, 2), 8, (P, P, D)), {}),
    "3d_all_periodic": (lambda: box(3, (2, 4, 2), 8, (P, P, P)), {}),
    "3d_amr": (lambda: W.cfg2_gauss3d(base=32, N=8, radii=(0.3, 0.15), sigma=0.05), {}),
    "3d_16_blocks": (lambda: box(3, (2, 2, 2), 16, (D, D, N)), {}),
    "2d_vareps": (lambda: box(2, (6, 4), 8, (N, D), eps=True), {}),
    "3d_vareps_periodic": (lambda: W.cfg3_varcoef3d(n=32, N=16, seed=2, contrast=10.0), {}),
    "3d_vareps_amr": (lambda: box(3, (4, 4, 4), 8, (D, D, N), eps=True,
                                  refine=W.refine_spheres(3, 8, (32,) * 3, (0,) * 3, (2,) * 3, (1.0,) * 3, (0.6,))), {}),
    "2d_jacobi": (lambda: box(2, (6, 4), 8, (N, D)), dict(smoother=1)),
    "3d_jacobi_vareps": (lambda: box(3, (4, 2, 2), 8, (D, N, P), eps=True), dict(smoother=1)),
}


def rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def cycles(mg, p, n, smoother=0, schedule=None):
    """phi after FMG and n - 1 V-cycles of the solve loop, and the launches they took."""
    t = mg.Tree.from_problem(p)
    if schedule:
        t.set_schedule(*schedule)
    n0 = t.launch_count()
    t.solve(1e-14, n, raise_on_fail=False, smoother=smoother)
    return t, t.get_phi().cpu().numpy(), t.launch_count() - n0


def oracle_cycles(o, n):
    """The solve loop: FMG, then V-cycles, the composite residual (which resets covered cells) before each."""
    o.residual_norm()
    o.fmg()
    for _ in range(n - 1):
        o.residual_norm()
        o.vcycle(1)


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_cycles_match_oracle(mg, name):
    make, kw = CASES[name]
    p = make()
    t, phi, launches = cycles(mg, p, 3, **kw)
    o = Oracle.from_problem(p)
    if kw.get("smoother"):
        o.set_smoother(1)
    oracle_cycles(o, 3)
    ref = o.get_phi()
    if D not in p.bc_type[:2 * p.dim]:  # defined up to a constant
        phi, ref = phi - phi.mean(), ref - ref.mean()
    assert rel(phi, ref) <= TOL
    # the lower levels ran in one launch per leg: fewer than the same cycles one by one
    u = mg.Tree.from_problem(p)
    n0 = u.launch_count()
    u.fmg(**kw)
    u.vcycle(2, **kw)
    assert launches < u.launch_count() - n0


@pytest.mark.parametrize("name", ["2d_odd_blocks_periodic_y", "3d_odd_blocks", "3d_amr", "3d_vareps_periodic", "2d_jacobi"])
def test_mixed_precision_reaches_tolerance(mg, name):
    make, kw = CASES[name]
    p = make()
    t = mg.Tree.from_problem(p)
    cyc, r = t.solve(1e-10, 60, precision=mg.MG_FP32_DC, inner_cycles=2, **kw)
    o = Oracle.from_problem(p)
    r0, _ = o.residual_norm()
    o.set_phi(t.get_phi().cpu().numpy())
    r1, _ = o.residual_norm()
    assert r <= 1e-10 and r1 <= 1.05e-10 * r0, (cyc, r, r1 / r0)


def test_schedule_applies_to_the_lower_levels(mg):
    p = box(2, (8, 8), 8, (D, D))
    nl = len(mg.Tree.from_problem(p, finalize=False).levels())
    down, up = [(l + 1) % 3 for l in range(nl)], [(2 * l + 1) % 4 for l in range(nl)]
    _, phi, _ = cycles(mg, p, 3, schedule=(down, up))
    o = Oracle.from_problem(p)
    o.set_schedule(down, up)
    oracle_cycles(o, 3)
    assert rel(phi, o.get_phi()) <= TOL


def test_new_coefficients_reach_the_kernel(mg):
    """A later set_eps rebuilds the dense coefficients: the solve equals a fresh tree's."""
    import torch
    p = CASES["2d_vareps"][0]()
    t, _, _ = cycles(mg, p, 2)
    e = torch.from_numpy(1.0 + W.leaf_field(p, "eps") ** 2).cuda()
    u = mg.Tree.from_problem(p)
    for q in (t, u):
        q.set_eps(e)
        q.set_phi(torch.zeros_like(e))
        q.solve(1e-14, 3, raise_on_fail=False)
    assert torch.equal(t.get_phi(), u.get_phi())
