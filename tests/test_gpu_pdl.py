"""Programmatic dependent launch (MG_PDL=1, read once per process) against the
default launches, each in its own process: set_eps with the coarsest inverse,
the cluster kernel's coefficients and a solve behind each, an adapted mesh, a
batch with parallel branches.  Without the timed choice of sweep kernels both
processes run the same arithmetic in the same order: the results are equal bit
for bit.  (The adjoint adds its ghosts with atomics and differs between any
two runs: not here.)  A batch keeps its timed choice, whose kernels differ in
rounding order: 1e-12 relative after three cycles, as between the variants."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
import numpy as np
import torch
from synth import workloads as W
import paper_1901_11370_gb300 as mg
rng = np.random.default_rng(3)
out = {}
types = {2: (0, 1, 0, 0, 2, 2), 3: (1, 0, 2, 2, 0, 1)}
for dim, n, base in ((2, 8, (96, 48, 1)), (3, 8, (64, 64, 32))):
    p = W.Problem("box", dim, n, 0, base, (0.0,) * 3, (1.0,) * 3, types[dim], (0.1, 0.2, 0.3, 0.4, 0.5, 0.6),
                  np.zeros((0, 4), np.int32), 512, rhs=lambda X, Y, Z: np.cos(3 * X) * np.sin(5 * Y) + Z)
    t = mg.Tree.from_problem(p)
    for prec in (mg.MG_FP64, mg.MG_FP32_DC):
        t.set_sweep_variant(-1, precision=prec)  # drops the timed choice: the same sweeps in every process
    for k in range(3):
        t.set_eps(torch.from_numpy(rng.uniform(1.0, 10.0, t.n_leaf)).cuda())
        for prec in (mg.MG_FP64, mg.MG_FP32_DC):
            t.set_phi(torch.zeros(t.n_leaf, dtype=torch.float64, device="cuda"))
            t.solve(1e-9, 4, precision=prec, raise_on_fail=False)
            out["solve%d_%d_%d" % (dim, k, prec)] = t.get_phi().cpu().numpy()
    a = t.adapt(add=[(0, 1, 1, 0), (0, 2, 1, 0)])
    out["adapt%d" % dim] = a.get_phi().cpu().numpy()
trees = [mg.Tree.from_problem(W.cyl_ring_tree(s, N=16, kmin=2, kmax=4), finalize=False) for s in range(6)]
b = mg.Batch(trees)
b.set_rhs(torch.from_numpy(np.random.default_rng(1).standard_normal(b.n_leaf)).cuda())
b.vcycle(3)
out["batch"] = b.get_phi().cpu().numpy()
np.savez(sys.argv[1], **out)
"""


def test_programmatic_launches_give_the_same_results(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11370_gb300 import build as B
    B.build()
    got = []
    for mode in ("0", "1"):
        f = str(tmp_path / ("pdl%s.npz" % mode))
        env = dict(os.environ, MG_PDL=mode, PYTHONPATH=ROOT)
        r = subprocess.run([sys.executable, "-c", PROGRAM, f], cwd=ROOT, env=env, timeout=300, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
        got.append(np.load(f))
    assert sorted(got[0].files) == sorted(got[1].files)
    for k in got[0].files:
        assert np.isfinite(got[0][k]).all() and np.abs(got[0][k]).max() > 0, k
        if k == "batch":
            assert np.abs(got[0][k] - got[1][k]).max() <= 1e-12 * np.abs(got[0][k]).max()
        else:
            assert np.array_equal(got[0][k], got[1][k]), k
