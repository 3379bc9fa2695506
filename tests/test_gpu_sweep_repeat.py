"""Dimension sweeps called again on one handle: the replayed graphs must not
race with what the call writes before them (the bases' upload, the product's
buffers), so every repetition of a small sweep returns the same bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_repeated_small_sweeps_agree_bitwise():
    import paper_1807_03425_gb300 as P
    E = W.endmembers(3, 40)
    X = W.hyperspectral(300, 5, E, noise=0.01, bf16=False)
    U0 = W.random_basis(40, 6, 7)
    with P.Sap(X) as s:
        first = s.estimate_dim(U0, 3, 0.01, 0.1)
        pairs = [s.sweep_history(k, 4)[1] for k in range(1, 7)]
        for _ in range(60):
            k, r = s.estimate_dim(U0, 3, 0.01, 0.1)
            assert k == first[0] and np.array_equal(r, first[1])
        for k in range(1, 7):
            assert np.array_equal(s.sweep_history(k, 4)[1], pairs[k - 1])
