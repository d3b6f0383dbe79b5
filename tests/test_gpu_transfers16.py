"""One FP32 correction cycle of 16^3 blocks against the oracle's FP64 cycle,
field by field.  From phi = 0 a defect-correction step is phi = e with e the
FP32 V-cycle of the residual; the V-cycle is affine, so the oracle's V-cycle
from phi = 0 with the boundary values gives the same field up to FP32
rounding (the oracle's two forms agree to 1e-15).  With few smoothing steps a
wrong neighbour, weight or ghost of the restriction or the prolongation, at a
refinement face too, is not smoothed away: it shows at the size of the jumps
across a cell, 1e-2 and more.  Bound: u = 6e-8 of the largest value, some
three roundings a half-sweep or transfer, on five levels of up to 12 such
steps: 1e-5.  The sweep variant of 16^3 blocks is pinned, so that every level
goes through these kernels and not through the cluster kernel."""
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
CASES = {  # problem, lambda
    "one_block_wide": (lambda: box((2, 2, 2), (D, N, D)), 0.0),
    "periodic": (lambda: box((2, 4, 2), (P, P, D)), 0.0),
    "many_blocks": (lambda: box((8, 6, 8), (D, D, N)), 0.0),
    "vareps": (lambda: box((4, 2, 2), (N, D, P), eps=True), 0.0),
    "amr": (lambda: box((4, 4, 4), (D, N, D), refine=AMR), 0.0),
    "amr_vareps": (lambda: box((4, 4, 4), (D, N, D), eps=True, refine=AMR), 0.0),
    "lambda": (lambda: box((4, 2, 4), (N, N, P)), 30.0),
    "lambda_amr_vareps": (lambda: box((4, 4, 4), (N, N, N), eps=True, refine=AMR), 30.0),
}


def both(mg, p, helm):
    """GPU tree and oracle of a problem with constant boundary values."""
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


@pytest.mark.parametrize("steps", [(1, 0, 1), (0, 1, 1), (1, 1, 1), (1, 1, 2)])  # down, up, cycles
@pytest.mark.parametrize("name", sorted(CASES))
def test_one_correction_matches_the_oracle(mg, name, steps):
    make, helm = CASES[name]
    t, o = both(mg, make(), helm)
    down, up, inner = steps
    t.set_sweep_variant(0, precision=mg.MG_FP32_DC)
    t.solve(1e-30, 1, fmg_first=False, precision=mg.MG_FP32_DC, inner_cycles=inner, n_down=down, n_up=up, raise_on_fail=False)
    o.set_cycle(down, up)
    o.vcycle(inner)
    ref = o.get_phi()
    assert np.abs(t.get_phi().cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("name", ["lambda", "lambda_amr_vareps"])
@pytest.mark.parametrize("variant", [0, 1])
def test_lambda_converges(mg, name, variant):
    make, helm = CASES[name]
    t, o = both(mg, make(), helm)
    t.set_sweep_variant(variant, precision=mg.MG_FP32_DC)
    t.solve(1e-10, 60, precision=mg.MG_FP32_DC)
    r0, _ = o.residual_norm()
    o.set_phi(t.get_phi().cpu().numpy())
    r1, _ = o.residual_norm()
    assert r1 <= 1.05e-10 * r0
