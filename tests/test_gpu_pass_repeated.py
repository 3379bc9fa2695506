"""The all-pairs pass over and over on data whose filter flags many columns,
while other warps (and, in a sweep, other bases' passes) lower the bound: the
lanes of a warp may see different values of it, and none of what they do
together may depend on that.  Every repetition returns the same bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_repeated_image_sweeps():
    import paper_1807_03425_gb300 as P
    g = W.rng(3)
    side, N = 40, 1000
    c = side / 4 + side / 2 * g.random((N, 2))
    u = np.arange(side)
    gx, gy = (np.exp(-((u - c[:, q:q + 1]) ** 2) / (2 * (side / 16) ** 2)) for q in (0, 1))
    X = (gy[:, :, None] * gx[:, None, :]).reshape(N, side * side).astype(np.float32)
    U0 = W.random_basis(side * side, 12, 5)
    for tier in (-1, 5):
        with P.Sap(X) as s:
            s.set_basis(U0)
            s.set_tuning(refine_tier=tier)
            _, first = s.estimate_dim(U0, 6, 0.01, 0.1)
            for _ in range(80):
                _, r = s.estimate_dim(U0, 6, 0.01, 0.1)
                assert np.array_equal(r, first)


@pytest.mark.parametrize("N,n,k", [(1500, 60, 5), (1500, 60, 20), (1500, 300, 6)])
@pytest.mark.parametrize("far", [1e3, 1e4])
def test_repeated_runs_with_a_far_point(N, n, k, far):
    import paper_1807_03425_gb300 as P
    X = W.moment_curve(N, n // 2, 3, np.float32, noise=0.02, noise_seed=4)
    X[N // 3] *= np.float32(far)
    U = W.random_basis(n, k, 5)
    with P.Sap(X) as s:
        s.set_basis(U)
        first = s.run(0.005, 100)
        for _ in range(8):
            s.set_basis(U)
            h, am = s.run(0.005, 100)
            assert np.array_equal(h, first[0]) and np.array_equal(am, first[1])
