"""A basis handed over by sap_set_basis: the call copies its input, so what
the caller (or the allocator) does with host memory right after it must not
reach the device.  Wide bases of many coordinates, each followed by
allocations of the same size that overwrite freed memory."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(40, 3), (4096, 20), (16384, 32)])
def test_upload_survives_reuse_of_host_memory(n, k):
    import paper_1807_03425_gb300 as P
    X = W.rng(1).standard_normal((64, n)).astype(np.float32)
    bases = [W.random_basis(n, k, s) for s in (2, 3)]
    with P.Sap(X) as s:
        for it in range(20):
            U = bases[it % 2]
            mine = U.copy()
            s.set_basis(mine)
            mine[:] = np.nan
            junk = [np.full((k, n), 1e300) for _ in range(3)]
            assert np.array_equal(s.get_basis(), U)
            del junk
