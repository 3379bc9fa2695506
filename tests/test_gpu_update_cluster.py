"""The basis update by a thread-block cluster (FP32/BF16 data, k > 8 or
n > 128) at the sizes where its split can go wrong: row counts around the
blocks' shares, one to sixteen blocks, compute widths with pad columns, a
direction that vanishes, both readings of the rotation.  Against the FP64
oracle's update for the pair the GPU chose: the rotated basis is formed in
FP32, so entries agree to a few FP32 roundings of the k-term sums (1e-5, the
bar of the other update tests); the re-orthonormalisation is FP64, so
|U U^T - I| stays below 4 n 2^-53 + 64 * 2^-53."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import check_basis

pytestmark = pytest.mark.gpu


def points(N, n, seed):
    return W.hyperspectral(N, seed, W.endmembers(seed + 1, n), noise=0.05, bf16=False)


def orthonormality(U):
    U = U.astype(np.longdouble)
    return float(np.abs(U @ U.T - np.eye(len(U))).max())


@pytest.mark.parametrize("n,k", [(9, 9), (33, 12), (64, 13), (65, 17), (128, 32), (129, 1), (129, 8), (256, 5),
                                 (257, 10), (512, 24), (513, 25), (1024, 2), (1031, 16), (2050, 9)])
@pytest.mark.parametrize("path", ["restructured", "plain"])
def test_cluster_update_matches_oracle(n, k, path):
    import paper_1807_03425_gb300 as P
    if path == "plain" and k > 8:
        pytest.skip("the FP32 plain form has k <= 8")
    X = points(150, n, 3)
    U = W.random_basis(n, k, 5)
    for mode, om in (("literal", O.MODE_LITERAL), ("angle", O.MODE_ANGLE)):
        if mode == "angle" and k == n:
            continue  # s lies in the span: e = s - P P^T s is zero, e/|e| undefined
        with P.Sap(X) as s:
            s.set_path(path)
            s.set_update_mode(mode)
            s.set_basis(U)
            for _ in range(3):
                U0 = s.get_basis()
                i, j, r = s.step(0.02)
                assert abs(r - O.ratio(X.astype(np.float64), U0, i, j)) <= 1e-12
                Ug = s.get_basis()
                Uo, _ = O.update(X.astype(np.float64), U0, i, j, 0.02, om)
                check_basis(Ug, Uo)
                assert orthonormality(Ug) <= (4 * n + 64) * 2.0 ** -53


def test_cluster_update_vanishing_direction():
    """alpha = 1 with the argmin secant in the span: the rotated direction is
    zero up to rounding and the old first direction is kept."""
    import paper_1807_03425_gb300 as P
    n, k = 160, 10
    X = np.zeros((2, n), np.float32)
    X[1, 0] = 1.0
    U = np.eye(n)[:k]
    with P.Sap(X) as s:
        s.set_basis(U)
        i, j, r = s.step(1.0)
        Ug = s.get_basis()
    assert (i, j) == (0, 1) and abs(r - 1.0) < 1e-12
    Uo, _ = O.update(X.astype(np.float64), U, 0, 1, 1.0, O.MODE_LITERAL)
    assert orthonormality(Ug) <= (4 * n + 64) * 2.0 ** -53
    assert np.abs(Ug.T @ Ug - Uo.T @ Uo).max() <= 1e-5
