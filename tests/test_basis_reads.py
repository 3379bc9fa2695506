"""The basis is rewritten by every update, and with programmatic launch the
next pass's blocks may already be resident while an update still runs.  The
non-coherent load path (__ldg) is for data that stay constant over a kernel's
whole lifetime, so no kernel may take the basis, its 16-bit operands, the
projections or the lists through it: those may be read through __ldg only
that are constant over a run -- the points, their norms, the lengths."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_03425_gb300", "csrc")
CONSTANT = re.compile(r"^(a\.(X|nu|w|xn) \+|w32t \+|p\)?$)")


def test_only_constant_data_take_the_noncoherent_path():
    seen = 0
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__ldg\(([^()]*)", src):
            seen += 1
            assert CONSTANT.match(m.group(1)), "%s: __ldg(%s" % (f, m.group(1))
        # the helper that wraps it is instantiated with the points' type only
        for m in re.finditer(r"ld_fp64<(\w+), RO>\(([^)]*)\)", src):
            assert m.group(1) == "TX" and m.group(2).startswith(("xi", "xj")), "%s: %s" % (f, m.group(0))
    assert seen > 0


@pytest.mark.gpu
@pytest.mark.parametrize("n,k", [(100, 5), (224, 10), (200, 16)])
def test_overlapped_launches_give_the_same_bits(n, k):
    """Iterations whose kernels overlap (programmatic launch) against the same
    iterations one kernel after another: histories, pairs and bases bitwise
    equal, over two hundred iterations."""
    import numpy as np

    import paper_1807_03425_gb300 as P
    import workloads as W
    X = W.hyperspectral(1500, 3, W.endmembers(4, n), noise=0.02, bf16=False)
    U = W.random_basis(n, k, 5)
    out = []
    for pdl in (0, 1):
        with P.Sap(X) as s:
            s.set_basis(U)
            s.set_tuning(refine_tier=5, programmatic_launch=pdl)
            h, am = s.run(0.01, 200)
            out.append((h, am, s.get_basis()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
