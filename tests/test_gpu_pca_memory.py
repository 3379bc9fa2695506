"""The work memory of the PCA start: 8 B per pair, 8 N n for the Laplacian's
rows and four n x n FP64 matrices; partial Gram matrices beside them only
while n is small.  Accuracy where the rows are cut into one, some and all of
the bands, with fewer rows than bands."""
import threading

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def points(N, n, seed):
    g = np.random.default_rng(seed)
    return (g.standard_normal((N, n)) * (3.0 * 0.97 ** np.arange(n)) + 1.5).astype(np.float32)


def test_work_memory_of_many_coordinates():
    torch = pytest.importorskip("torch")
    import paper_1807_03425_gb300 as P
    N, n = 300, 2048
    with P.Sap(points(N, n, 1)) as s:
        s.secant_pca(2)  # the basis's own buffers exist from here on
        torch.cuda.synchronize()
        before, low, stop = torch.cuda.mem_get_info()[0], [], threading.Event()

        def watch():
            while not stop.is_set():
                low.append(torch.cuda.mem_get_info()[0])
        t = threading.Thread(target=watch)
        t.start()
        s.secant_pca(2)
        stop.set()
        t.join()
    used = before - min(low)
    need = 8 * N * N + 8 * N * n + 32 * n * n
    assert len(low) > 10 and used >= 32 * n * n, "the call was not observed"
    assert used <= need + (64 << 20), (used, need)


@pytest.mark.parametrize("N,n,k", [(20, 40, 2), (33, 20, 2), (400, 100, 3), (515, 100, 3), (513, 260, 3), (90, 570, 2)])
def test_bands(N, n, k):
    import paper_1807_03425_gb300 as P
    X = points(N, n, N)
    with P.Sap(X) as s:
        U, sv = s.secant_pca(k)
    Uo, svo = O.secant_pca(X.astype(np.float64), k)
    assert np.allclose(sv, svo, rtol=1e-10, atol=0)
    assert np.abs(U @ U.T - np.eye(k)).max() < 1e-12
    assert np.abs(U.T @ (U @ Uo.T) - Uo.T).max() < 1e-8
