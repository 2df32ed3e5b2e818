"""x-panel products whose copies stop coming: every kernel instance gives up
within its bound, says so in the status word, and leaves the device usable."""
import time

import numpy as np
import pytest

import gen
import oracle
from helpers import rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,q,nvec", [(65521, 1, 1), (65521, 2, 4), (3, 1, 1), (2**31 - 1, 2, 2), (2**32 - 5, 4, 1)])
def test_products_without_their_copies_end_within_the_bound(lib, m, q, nvec):
    A = gen.powerlaw_matrix(seed=8, n=150_001, lmax=10_000, m=m)
    opts = dict(priority_format=lib.FMT.PANEL, panel_cluster=q, transpose_mode=lib.TRANSPOSE.NONE)
    # hook 2: stages from the second on are never issued; hook 4: one pass for all the vectors
    M = lib.Matrix.from_csr(A, test_hooks=2 | 4, **opts)
    x = rand_block(5, A.ncols, nvec, m)
    xd, yd = to_dev(x), to_dev(np.zeros((A.nrows, nvec), dtype=np.uint32))
    assert M.launches(False, nvec) == 1     # (builds the layout of a wide pass)
    t = time.perf_counter()
    M.apply(xd, yd)
    with pytest.raises(lib.FFSPMVError) as e:
        M.check_status()
    # 0.7 s for the first wait, 0.05 s for copies in flight
    assert e.value.status == 6 and time.perf_counter() - t < 2.0
    N = lib.Matrix.from_csr(A, test_hooks=4, **opts)
    N.apply(xd, yd)
    N.check_status()
    assert np.array_equal(to_host(yd), oracle.csr_spmv(A, x).reshape(A.nrows, nvec))
