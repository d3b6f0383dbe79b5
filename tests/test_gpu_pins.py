"""Pinned sweep variants and the solves' cluster kernel: a pin on a level
above the kernel's levels leaves it on, one on its levels turns it off, and
taking the pin back restores it, level by level or all at once; an adapted
mesh keeps the pins.  Counted by launches: the launch-by-launch cycle takes more of them."""
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


@pytest.mark.parametrize("precision", [0, 1])
def test_pins_and_the_cluster_kernel(mg, precision):
    import torch
    p = W.cfg2_gauss3d(base=64, N=8, radii=(0.3,), sigma=0.05)
    t = mg.Tree.from_problem(p)
    top = len(t.levels()) - 1
    zero = torch.zeros(t.n_leaf, dtype=torch.float64, device="cuda")

    def launches(t=t, zero=zero):
        t.set_phi(zero)
        n0 = t.launch_count()
        t.solve(1e-30, 2, precision=precision, raise_on_fail=False)
        return t.launch_count() - n0
    launches()
    free = launches()
    t.set_sweep_variant(0, level=top, precision=precision)
    assert launches() == free
    t.set_sweep_variant(-1, level=top, precision=precision)
    t.set_sweep_variant(0, level=2, precision=precision)
    assert launches() > free
    t.set_sweep_variant(-1, level=2, precision=precision)
    assert launches() == free
    t.set_sweep_variant(0, precision=precision)
    assert launches() > free
    t.set_sweep_variant(-1, precision=precision)
    assert launches() == free
    # an adapted mesh takes the pins along
    add = [(0, 0, 0, 0)]
    a = t.adapt(add=add)
    za = torch.zeros(a.n_leaf, dtype=torch.float64, device="cuda")
    a.set_rhs(za + 1.0)
    launches(a, za)
    free = launches(a, za)
    t.set_sweep_variant(0, level=2, precision=precision)
    b = t.adapt(add=add)
    b.set_rhs(za + 1.0)
    launches(b, za)
    assert launches(b, za) > free


@pytest.mark.parametrize("cells, eps, cluster", [((200, 120), True, True), ((248, 216), True, False),
                                                 ((248, 216), False, False), ((200, 280), False, True)])
def test_a_large_coarsest_solve_stays_with_the_whole_chip(mg, cells, eps, cluster):
    """Coarsest levels of 1500 and 3348 cells with the dense inverse (the
    second cannot take eigenvectors), of 3500 with eigenvectors: whether the
    solves take the cluster kernel, by what a pin on its levels changes."""
    import torch
    p = W.Problem("box", 2, 4, 0, cells + (1,), (0.0,) * 3, (1.0,) * 3, (0, 1, 0, 1, 2, 2), (0.0,) * 6,
                  np.zeros((0, 4), np.int32), 4000)
    t = mg.Tree.from_problem(p)
    assert t.levels()[0]["ncell"][:2] == (cells[0] // 4, cells[1] // 4)
    one = torch.ones(t.n_leaf, dtype=torch.float64, device="cuda")
    t.set_rhs(one)
    if eps:
        t.set_eps(2 * one)
    n = []
    for pin in (False, True):
        if pin:
            t.set_sweep_variant(1, level=1)
        for _ in range(2):
            t.set_phi(0 * one)
            n0 = t.launch_count()
            t.solve(1e-30, 2, raise_on_fail=False)
        n.append(t.launch_count() - n0)
    assert (n[0] < n[1]) == cluster, n
