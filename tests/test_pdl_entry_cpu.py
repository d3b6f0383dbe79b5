"""Kernels launched with the programmatic-serialization attribute (launch_k,
when MG_PDL=1) may start before the grid they depend on has finished: stream
order is kept by pdl_entry(), which waits for it, as each one's first
statement.  Read off the sources: a kernel without it reads memory that the
previous kernel may still be writing, on some runs only."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_11370_gb300", "csrc")
# launched without the attribute, by the named helper
PLAIN = {"k_bottom": "launch_cluster", "k_tail": "launch_coop"}


def kernels(src):
    """(name, body) of every kernel, comments removed."""
    src = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
    for g in re.finditer(r"__global__", src):
        m = re.compile(r"\b(k_\w+)\s*\(").search(src, g.end())
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        yield m.group(1), src[src.index("{", i) + 1:].lstrip()


@pytest.mark.parametrize("name", ["mg_kernels.cu", "mg_adjoint.cu", "mg_bottom.cu", "mg_coarse.cu"])
def test_every_kernel_waits_for_its_stream_first(name):
    src = open(os.path.join(CSRC, name)).read()
    found = list(kernels(src))
    assert found
    bad = [k for k, body in found if not body.startswith("pdl_entry();")]
    for k in bad:
        assert k in PLAIN and PLAIN[k] + "(" in src, k
        assert not re.search(r"launch_k\(%s\b" % k, src), k
