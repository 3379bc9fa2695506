"""The forms of the PCA start: the eigensolver as one cluster launch (n <=
256) and as launches per round (n > 256) at the boundary, odd and even n, few
points; FP32 data's lengths and Laplacian in FP32 pairs with the short secants
in FP64: tight clusters (all secants short or all long relative to the
spread), a threshold met exactly (d == eps is kept), data far from the
origin.  Against the FP64 oracle at the tolerances of the other PCA tests
(1e-10 on the singular values, 1e-8 on the vectors where the spectrum has
gaps)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def decaying(N, n, seed):
    g = np.random.default_rng(seed)
    return (g.standard_normal((N, n)) * (3.0 * 0.9 ** np.arange(n)) + 1.5).astype(np.float32)


def check(X, k, eps=0.0, vectors=True):
    import paper_1807_03425_gb300 as P
    with P.Sap(X) as s:
        if eps:
            s.set_min_secant_length(eps)
        U, sv = s.secant_pca(k)
    Uo, svo = O.secant_pca(X.astype(np.float64), k, eps)
    assert np.allclose(sv, svo, rtol=1e-10, atol=0)
    assert np.abs(U @ U.T - np.eye(k)).max() < 1e-12
    if vectors:
        assert np.abs(U - Uo).max() < 1e-8


@pytest.mark.parametrize("N,n,k", [(3, 2, 1), (40, 3, 2), (130, 31, 4), (64, 128, 3), (90, 255, 3), (90, 256, 3),
                                   (90, 257, 3), (70, 300, 2)])
def test_eigensolver_forms(N, n, k):
    check(decaying(N, n, N + n), k)


@pytest.mark.parametrize("spread", [1e-6, 1e-2, 1.0])
def test_clusters(spread):
    g = np.random.default_rng(4)
    c = g.standard_normal((6, 12)) * (3.0 * 0.7 ** np.arange(12))
    X = (np.repeat(c, 30, axis=0) + spread * g.standard_normal((180, 12)) * 0.8 ** np.arange(12)).astype(np.float32)
    check(X, 3)


@pytest.mark.parametrize("eps", [1.0, 2.0, 5.0])
def test_threshold_met_exactly(eps):
    """Integer points: many squared lengths equal eps^2 exactly and are kept."""
    g = np.random.default_rng(6)
    X = g.integers(0, 6, size=(150, 4)).astype(np.float32) * np.array([1, 1, 2, 3], np.float32)
    check(X, 2, eps)


def test_far_from_origin():
    check(decaying(200, 10, 8) + np.float32(512.0), 2)
