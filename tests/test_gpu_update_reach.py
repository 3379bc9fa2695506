"""The cluster update and the soft-min step where the other tests do not take
them: through the split over ranks (its records form the list that the recheck
before the update reads), at the largest numbers of coordinates (blocks near
the limit of shared memory), and a soft-min step so long that the first
Cholesky pass leaves more than rounding (the factorisation is repeated)."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import check_basis

pytestmark = pytest.mark.gpu


def orthonormality(U):
    U = U.astype(np.longdouble)
    return float(np.abs(U @ U.T - np.eye(len(U))).max())


@pytest.mark.parametrize("n,k,world", [(40, 12, 2), (224, 10, 3), (300, 9, 2), (130, 4, 2)])
def test_split_equals_unsplit_bitwise(n, k, world):
    import paper_1807_03425_gb300 as P
    X = W.hyperspectral(900, 3, W.endmembers(4, n), noise=0.02, bf16=False)
    U0, alpha, T = W.random_basis(n, k, 5), 0.01, 6
    with P.Sap(X) as s:
        s.set_basis(U0)
        hist, am = s.run(alpha, T)
        U = s.get_basis()
    ranks = [P.ShardSap(X, world, r) for r in range(world)]
    try:
        for s in ranks:
            s.set_basis(U0)
        for _ in range(T):
            recs = [s.min_record() for s in ranks]
            for s in ranks:
                s.step_records(alpha, recs)
        for s in ranks:
            h, a = s.get_history(T)
            assert np.array_equal(h, hist[:T]) and np.array_equal(a, am[:T]) and np.array_equal(s.get_basis(), U)
    finally:
        for s in ranks:
            s.close()


@pytest.mark.parametrize("n,k", [(8192, 24), (16384, 5), (16384, 9), (16384, 32)])
def test_largest_dimensions(n, k):
    import paper_1807_03425_gb300 as P
    X = W.rng(n + k).standard_normal((40, n)).astype(np.float32)
    X64 = X.astype(np.float64)
    with P.Sap(X) as s:
        s.set_basis(W.random_basis(n, k, 5))
        for _ in range(2):
            U0 = s.get_basis()
            i, j, r = s.step(0.02)
            assert abs(r - O.ratio(X64, U0, i, j)) <= 1e-12
            Ug = s.get_basis()
            check_basis(Ug, O.update(X64, U0, i, j, 0.02, O.MODE_LITERAL)[0])
            assert orthonormality(Ug) <= (4 * n + 64) * 2.0 ** -53


@pytest.mark.parametrize("k", [2, 5, 8])
@pytest.mark.parametrize("eta", [0.5, 30.0, 1e4, 1e5])
def test_long_softmin_steps(k, eta):
    """One pair dominates at this tau, so U + eta G_R / |G_R| has a condition
    of about eta; from 3000 on the first pass leaves more than 1e-9."""
    import paper_1807_03425_gb300 as P
    X = W.moment_curve(300, 15, 7, np.float32)
    U = W.random_basis(30, k, 8)
    tau = 1e-3
    with P.Sap(X) as s:
        s.set_basis(U)
        s.softmin_ascent(tau, eta, 1)
        Ug = s.get_basis()
    assert orthonormality(Ug) <= (4 * 30 + 64) * 2.0 ** -53
    if eta <= 30.0:
        # the span moves by at most eta times the gradient's relative error
        Uo, _, _ = O.softmin_ascent_step(X.astype(np.float64), U, tau, eta)
        assert np.abs(Ug.T @ Ug - Uo.T @ Uo).max() <= 1e-4 * eta
