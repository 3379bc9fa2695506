"""The PCA start of FP32 data at every scale that FP32 holds: S S^T does not
depend on the unit of length, so neither may its accuracy.  Where the squares
of the coordinates or their residuals leave FP32's range the lengths have to
come from FP64.  Against the FP64 oracle at the bars of the other PCA tests
(1e-10 on the singular values, 1e-8 on the vectors)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def check(X, k, eps=0.0):
    import paper_1807_03425_gb300 as P
    with P.Sap(X) as s:
        if eps:
            s.set_min_secant_length(eps)
        U, sv = s.secant_pca(k)
    # the same problem near unit scale (a power of two: nothing is rounded)
    unit = 2.0 ** np.floor(np.log2(float(np.abs(X).max())))
    Uo, svo = O.secant_pca(X.astype(np.float64) / unit, k, eps / unit)
    assert np.allclose(sv, svo, rtol=1e-10, atol=0), np.abs(sv / svo - 1).max()
    assert np.abs(U - Uo).max() < 1e-8, np.abs(U - Uo).max()


@pytest.mark.parametrize("scale", [1e-30, 1e-23, 1e-21, 1e-20, 1e-18, 1e-15, 1e-12, 1e-3, 1e6, 1e12, 1e17])
def test_scales(scale):
    g = np.random.default_rng(11)
    X = g.standard_normal((400, 60)) * (3.0 * 0.9 ** np.arange(60)) + 0.5
    check((X * scale).astype(np.float32), 4)


@pytest.mark.parametrize("e", [-66, -40, 0, 40])
@pytest.mark.parametrize("eps", [1.0, 2.0, 5.0])
def test_threshold_met_exactly(e, eps):
    """Integer points times a power of two: many lengths equal the threshold
    exactly and are kept."""
    g = np.random.default_rng(6)
    X = g.integers(0, 6, size=(150, 4)) * np.array([1, 1, 2, 3])
    check(np.ldexp(X, e).astype(np.float32), 2, float(np.ldexp(eps, e)))
