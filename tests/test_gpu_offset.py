"""FP64 cycles of a solution with a large offset: x = 1e4 (and 1e4 plus a
linear part) with Dirichlet values of x and f = 0, the exact discrete
solution on a uniform mesh.  A cycle's rounding may follow the differences of
x in its residuals and x itself only where a cell is updated: a few u x per
half-sweep (u = 1.1e-16), b = 3, the same sign in the worst case, over the
upward half-sweeps of every level (the coarse correction removes those of the
downward ones): 4 b u x a level, at most 8 levels here: 100 u x.  A residual
whose rounding follows w |x|, alike in like cells, shows as that times
1 / (h^2 lambda_min), 1e3 and more."""
import numpy as np
import pytest

from synth import workloads as W

pytestmark = pytest.mark.gpu
CASES = {  # dim, block size, base cells
    "2d_8_blocks": (2, 8, 512),
    "2d_16_blocks": (2, 16, 1024),
    "2d_cluster_kernel_alone": (2, 8, 128),
    "3d_8_blocks": (3, 8, 128),
    "3d_16_blocks": (3, 16, 128),
    "3d_cluster_kernel_alone": (3, 4, 32),
}


@pytest.fixture(scope="module")
def mg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11370_gb300 import build as B
    B.build()
    import paper_1901_11370_gb300 as m
    return m


@pytest.mark.parametrize("slope", [0.0, 0.1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_error_of_an_offset_solution(mg, name, slope):
    import torch
    dim, n, cells = CASES[name]

    def x(X, Y, Z):
        return 1e4 + slope * (X + 2 * Y + (Z if dim == 3 else 0.0))
    p = W.Problem("offset", dim, n, 0, (cells,) * dim + (1,) * (3 - dim), (0.0,) * 3, (3.7,) * 3,
                  (0,) * (2 * dim) + (2,) * (6 - 2 * dim), (0.0,) * 6, np.zeros((0, 4), np.int32), 512,
                  rhs=lambda X, Y, Z: 0.0 * X, bc=lambda face, X, Y, Z: x(X, Y, Z))
    X, Y, Z, _ = W.leaf_cell_centres(p)
    exact = np.broadcast_to(x(X, Y, Z), X.shape)
    t = mg.Tree.from_problem(p)
    for solve in (True, False):  # through the solve loop and by the cycles called one by one
        t.set_phi(torch.zeros(t.n_leaf, dtype=torch.float64, device="cuda"))
        if solve:
            t.solve(0.0, 16, raise_on_fail=False)
        else:
            t.fmg()
            t.vcycle(15)
        err = np.abs(t.get_phi().cpu().numpy() - exact).max()
        assert err <= 100 * 2.0 ** -53 * exact.max(), solve
