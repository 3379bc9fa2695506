"""A batch in which one dataset has no secant at all: the call reports it, and
the histories and pairs of the datasets before it are delivered.  The next
call on the same batch starts clean."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [0, 1, 2])
def test_results_before_the_failing_dataset_are_delivered(bad):
    import paper_1807_03425_gb300 as P
    lib = P.load_library()
    T, n, k = 5, 12, 3
    Xs = [W.moment_curve(90 + 40 * b, n // 2, b, np.float32) for b in range(3)]
    alone = []
    for b in range(3):
        with P.Sap(Xs[b]) as s:
            s.set_basis(W.random_basis(n, k, b))
            alone.append(s.run(0.01, T))
    Xs[bad] = np.ones_like(Xs[bad])  # duplicates only
    with P.SapBatch(Xs) as s:
        for b in range(3):
            s.set_basis(b, W.random_basis(n, k, b))
        hist = np.full((3, T + 1), -7.0)
        am = np.full((3, T + 1, 2), -7, np.int64)
        code = lib.sap_run_batch(s.h, 0.01, T, hist.ctypes.data_as(ctypes.c_void_p), am.ctypes.data_as(ctypes.c_void_p))
        assert P.capi.sap_status_str(code) == "SAP_E_NO_SECANT"
        for b in range(3):
            if b < bad:
                assert np.array_equal(hist[b], alone[b][0]) and np.array_equal(am[b], alone[b][1])
            else:
                assert (hist[b] == -7.0).all() and (am[b] == -7).all()
        with pytest.raises(P.SapError) as e:  # the same again, not an error left over
            s.run(0.01, T)
        assert "dataset %d" % bad in str(e.value)
        good = 0 if bad else 1
        s.set_basis(good, W.random_basis(n, k, good))  # the run moved it
        i, j, r = s.min_secant(good)
        assert (i, j) == tuple(alone[good][1][0]) and r == alone[good][0][0]


def test_reading_a_history_allocates_nothing():
    torch = pytest.importorskip("torch")
    import paper_1807_03425_gb300 as P
    T = 200000
    with P.Sap(W.moment_curve(40, 4, 1, np.float32)) as s:
        s.set_basis(W.random_basis(8, 2, 2))
        s.run(0.001, T, history=False)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        h, am = s.get_history(T + 1)
        assert torch.cuda.mem_get_info()[0] == free
        assert h.shape == (T + 1,) and np.isfinite(h).all()
