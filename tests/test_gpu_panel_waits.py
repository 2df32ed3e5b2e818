"""What the CTAs of an x-panel product wait for: copies that stop coming (every
kernel instance gives up within its bound, says so in the status word, and
leaves the device usable), and each other's row sums."""
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


@pytest.mark.parametrize("m,q,n", [(65521, 2, 4_000_000), (2**31 - 1, 2, 2_000_000), (2**31 - 1, 4, 1_200_000)])
def test_ctas_of_a_cluster_with_uneven_work(lib, m, q, n):
    """More row groups than fit the GPU at once (x staged by a launch before, so
    no grid barrier), and rows whose entries lie in one column group but for one
    in a hundred: one CTA of a cluster is done long before the others and adds
    its few terms into their row sums."""
    nc = 200_000
    rng = np.random.default_rng(q)
    # rows in q bands, each with the columns of one q-th
    lo = np.arange(n) * q // n * (nc // q)
    cols = lo[:, None] + rng.integers(0, nc // q, (n, 3))
    far = rng.random(n) < 0.01
    cols[far, 0] = rng.integers(0, nc, int(far.sum()))
    A = gen.CSR(n, nc, np.arange(n + 1, dtype=np.int64) * 3, np.sort(cols, axis=1).reshape(-1).astype(np.int32),
                rng.integers(0, m, 3 * n, dtype=np.uint64).astype(np.uint32), m)
    M = lib.Matrix.from_csr(A, priority_format=lib.FMT.PANEL, panel_cluster=q, transpose_mode=lib.TRANSPOSE.NONE)
    assert M.launches(False, 1) == 2     # staging, product
    for k in range(3):
        x = rand_block(k, nc, 1, m)
        xd = to_dev(x)
        ys = [M.apply(xd) for _ in range(4)]
        M.check_status()
        want = oracle.csr_spmv(A, x)
        for y in ys:
            assert np.array_equal(to_host(y).reshape(want.shape), want)


def test_batch_without_a_layout_reports_a_wait_that_ran_out(lib):
    # no memory for the block layout (hook 16), so the x-panel plan runs, without its copies (hook 2)
    A = gen.powerlaw_matrix(seed=8, n=150_001, lmax=10_000, m=65521)
    M = lib.Matrix.from_csr(A, priority_format=lib.FMT.PANEL, transpose_mode=lib.TRANSPOSE.NONE, test_hooks=2 | 16)
    x, y = to_dev(rand_block(5, A.ncols, 1, 65521)), to_dev(np.zeros(A.nrows, dtype=np.uint32))
    lib.spmv_batch_apply([M.handle], [x], [y], [1])
    with pytest.raises(lib.FFSPMVError) as e:
        M.check_status()
    assert e.value.status == 6
    lib.spmv_batch_apply([M.handle], [x], [y], [1])     # on its layout now
    M.check_status()
    assert np.array_equal(to_host(y), oracle.csr_spmv(A, to_host(x)))
