"""The double-float tier (n > 256) with few and with very many near pairs: up
to a share of them the pass judges the near pairs itself and what is left is
evaluated pair by pair, beyond it every near pair goes through the
double-float rows of Y.  Both sides of that line, one basis and several, against
the FP64 oracle; and a set whose pairs are mostly near may not take many
times what a spread-out one takes."""
import time

import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import check_pair

pytestmark = pytest.mark.gpu


def clusters(N, n, m, seed, spread=0.02):
    g = W.rng(seed)
    return (g.standard_normal((m, n))[g.integers(0, m, N)] + spread * g.standard_normal((N, n))).astype(np.float32)


@pytest.mark.parametrize("N,n,m", [(300, 300, 100), (300, 300, 4), (300, 300, 2), (700, 260, 30), (520, 1030, 1), (200, 500, 3)])
@pytest.mark.parametrize("k", [3, 13, 25])
def test_argmin(N, n, m, k):
    import paper_1807_03425_gb300 as P
    X = clusters(N, n, m, N + m)
    X64 = X.astype(np.float64)
    U = W.random_basis(n, k, 5)
    with P.Sap(X) as s:
        s.set_basis(U)
        for _ in range(2):
            U0 = s.get_basis()
            m_ = O.min_secant(X64, U0)
            check_pair(X64, U0, m_, *s.min_secant())
            check_pair(X64, U0, m_, *s.step(0.02))


@pytest.mark.parametrize("m", [2, 60])
def test_sweep(m):
    import paper_1807_03425_gb300 as P
    X = clusters(400, 300, m, 3)
    U0 = W.random_basis(300, 6, 7)
    with P.Sap(X) as s:
        _, ratios = s.estimate_dim(U0, 0, 0.01, 0.1)
    for k in range(1, 7):
        want = O.min_secant(X.astype(np.float64), U0[:k])["r"]
        assert abs(ratios[k - 1] - want) <= 1e-5 * want + 1e-13


def test_many_near_pairs_cost_little():
    """All judged in the pass in vain, two clusters took 4.5 times as long as
    spread-out points; 1.8 times now."""
    import paper_1807_03425_gb300 as P
    best = []
    for X in (W.moment_curve(3000, 150, 3, np.float32), clusters(3000, 300, 2, 4)):
        with P.Sap(X) as s:
            U = W.random_basis(300, 6, 5)
            t = []
            for _ in range(8):
                s.set_basis(U)
                t0 = time.perf_counter()
                s.run(0.005, 16)
                t.append(time.perf_counter() - t0)
        best.append(min(t[1:]))
    assert best[1] < 3.0 * best[0], best
