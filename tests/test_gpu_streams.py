"""A mesh on a stream that does not block on the default stream (torch's own
streams are of that kind), while the default stream is busy: zero fills of new
arrays and table uploads must follow the mesh's stream, or they land after the
values that the caller has set.  The results are those of the same calls on
the default stream, bit for bit (timed sweep choices dropped)."""
import os
import re

import numpy as np
import pytest

from synth import workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_11370_gb300", "csrc")


def test_no_fill_or_upload_on_the_default_stream():
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cpp", ".h", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        assert not re.search(r"\bcudaMemset\(", src), name
        assert not re.search(r"\bcudaMemcpy\([^;]*cudaMemcpyHostToDevice", src), name


def results(mg, p, seed):
    import torch
    rng = np.random.default_rng(seed)
    t = mg.Tree.from_problem(p)
    out = []
    for prec in (mg.MG_FP64, mg.MG_FP32_DC):
        t.set_sweep_variant(-1, precision=prec)
    for eps in (False, True):
        if eps:
            t.set_eps(torch.from_numpy(rng.uniform(1.0, 5.0, t.n_leaf)).cuda())
        for prec in (mg.MG_FP64, mg.MG_FP32_DC):
            for smoother in (mg.MG_SMOOTH_RBGS, mg.MG_SMOOTH_JACOBI):
                t.set_phi(torch.zeros(t.n_leaf, dtype=torch.float64, device="cuda"))
                t.solve(1e-30, 2, precision=prec, smoother=smoother, raise_on_fail=False)
                out.append(t.get_phi())
    return out


@pytest.mark.gpu
def test_calls_on_a_non_blocking_stream_ignore_the_default_stream():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11370_gb300 import build as B
    B.build()
    import paper_1901_11370_gb300 as mg
    p = W.cfg2_gauss3d(base=64, N=8, radii=(0.3,), sigma=0.05)
    want = results(mg, p, 5)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(1000)  # loads the kernel
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)  # about 0.2 s on the default stream
    with torch.cuda.stream(s):
        got = results(mg, p, 5)
    torch.cuda.synchronize()
    for a, b in zip(want, got):
        assert torch.isfinite(a).all() and torch.equal(a, b)
