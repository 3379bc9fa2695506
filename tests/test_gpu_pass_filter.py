"""The all-pairs pass's tensor-core filter (a certified lower bound of every
pair's ratio) and what follows it, at the sizes where they can go wrong: one
to a few tiles with ragged edges, every operand width (1 to 7 MMA steps),
rows of Y staged and not, data far from unit scale and far from the origin,
tight clusters (near pairs), pass bounds from a long to an empty near list.
The argmin is decided in FP64, so the pair must be the FP64 oracle's (or tied
with it within 1e-6, the bar of the other tests)."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import check_pair

pytestmark = pytest.mark.gpu


def judge(X, k, tier=-1, bound=5e-4, seed=5):
    import paper_1807_03425_gb300 as P
    U = W.random_basis(X.shape[1], k, seed)
    X64 = X.astype(np.float64)
    m = O.min_secant(X64, U)
    with P.Sap(X) as s:
        s.set_basis(U)
        s.set_tuning(refine_tier=tier, pass_bound=bound)
        for _ in range(2):  # the second evaluation starts from the first's bound
            check_pair(X64, U, m, *s.min_secant())
        return s.stats()


@pytest.mark.parametrize("N,n,k", [(2, 3, 1), (3, 40, 20), (127, 9, 4), (128, 10, 5), (129, 24, 8), (200, 24, 9),
                                   (255, 30, 12), (256, 30, 13), (257, 40, 16), (300, 40, 17), (385, 60, 20),
                                   (300, 60, 21), (300, 60, 25), (300, 70, 32)])
@pytest.mark.parametrize("tier", [0, 5])
def test_filter_every_width(N, n, k, tier):
    judge(W.hyperspectral(N, N + k, W.endmembers(k, n), noise=0.1, bf16=False), k, tier)


@pytest.mark.parametrize("scale", [1e-9, 1e-3, 1e4, 1e9])
@pytest.mark.parametrize("k", [1, 5, 11])
def test_filter_data_scale(scale, k):
    X = W.moment_curve(400, 12, 3, np.float32) * np.float32(scale)
    judge(X, k)


@pytest.mark.parametrize("k", [2, 7])
def test_filter_far_from_origin(k):
    X = W.moment_curve(300, 8, 4, np.float32) + np.float32(1000.0)
    judge(X, k)


@pytest.mark.parametrize("bound", [1e-6, 5e-4, 0.25])
@pytest.mark.parametrize("tier", [-1, 1])
def test_filter_clusters(bound, tier):
    g = W.rng(8)
    c = g.standard_normal((40, 20))
    X = (np.repeat(c, 9, axis=0) + 1e-4 * g.standard_normal((360, 20))).astype(np.float32)
    X[7] = X[3]  # a duplicate
    st = judge(X, 3, tier, bound)
    assert bound > 1e-6 or st["n_near"] == st["n_pairs"] - st["n_excluded"]
