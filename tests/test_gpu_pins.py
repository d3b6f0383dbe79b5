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
