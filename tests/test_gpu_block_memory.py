"""Device memory of block layouts: what the packed rows of X take for the widths
in use, widths that grow, layouts that find no memory at first, and which blocks
run on the layout at all."""
import numpy as np
import pytest

import gen
import oracle
from helpers import rand_block, to_dev, to_host
from test_gpu_spmv import check_apply

pytestmark = pytest.mark.gpu


def _wide(m, rows=2000, cols=1_000_000):
    lengths = np.full(rows, 600)
    return gen.uniform_matrix(11, rows, cols, lengths, m, pm_fraction=0.1)


def _staged(M):
    return [int(line.split(" values, ")[1].split()[0]) for line in M.describe().splitlines() if "blocks:" in line]


def test_staging_is_as_wide_as_the_blocks(lib):
    import torch
    m = 2**31 - 1
    A = _wide(m)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    x = [to_dev(rand_block(1, A.ncols, v, m)) for v in (2, 3, 7)]
    y = [torch.empty((A.nrows, v), dtype=torch.int32, device="cuda") for v in (2, 3, 7)]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        M.apply(x[0], y[0])
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    # 1.2M entries of 8 bytes, 16 MB of packed rows; not 32 vectors' 128 MB
    assert _staged(M) == [16 * A.ncols] and used < 64 << 20, used
    M.apply(x[1], y[1])
    assert _staged(M) == [16 * A.ncols]
    for k in (2, 0, 1):
        M.apply(x[k], y[k])
        assert np.array_equal(to_host(y[k]), oracle.csr_spmv(A, to_host(x[k])))
    assert _staged(M) == [48 * A.ncols]


def test_captured_width_outlives_a_wider_block(lib):
    """A graph captured with narrow blocks keeps its buffer when wider blocks
    come, and a width that has no buffer yet is captured by the plan's path."""
    import torch
    m = 65521
    A = gen.uniform_matrix(3, 3000, 2500, np.full(3000, 9), m)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    X = {v: rand_block(v, A.ncols, v, m) for v in (3, 16, 32)}
    x = {v: to_dev(X[v]) for v in X}
    y = {v: torch.zeros((A.nrows, v), dtype=torch.int32, device="cuda") for v in X}
    M.launches(False, 3)
    M.apply(x[3], y[3])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graphs = []
    for v in (3, 32):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lib.spmv_apply(M.handle, x[v], v, y[v], v, v)
        graphs.append(g)
    for v in (16, 32):
        M.apply(x[v], y[v])
    for v in (3, 32):
        y[v].zero_()
    for g in graphs:
        g.replay()
    torch.cuda.synchronize()
    for v in X:
        assert np.array_equal(to_host(y[v]), oracle.csr_spmv(A, X[v])), v


@pytest.mark.parametrize("m", [65521, 2**31 - 1])
def test_no_memory_at_first(lib, m):
    # test hook 16: the first attempt at each layout fails
    A = gen.uniform_matrix(4, 3000, 2500, np.full(3000, 9), m)
    M = lib.Matrix.from_csr(A, test_hooks=16)
    B = lib.Matrix.from_csr(A, test_hooks=16, transpose_mode=lib.TRANSPOSE.NONE)
    for k in range(4):
        for transpose in (False, True):
            check_apply(lib, M, A, nvec=9, alpha=3, beta=2, seed=k, transpose=transpose)
        x, y = rand_block(k, A.ncols, 5, m), to_dev(np.zeros((A.nrows, 5), dtype=np.uint32))
        lib.spmv_batch_apply([B.handle], [to_dev(x)], [y], [5])
        assert np.array_equal(to_host(y), oracle.csr_spmv(A, x))
        if k == 0:
            assert not _staged(M) and not _staged(B)
    assert len(_staged(M)) == 2 and len(_staged(B)) == 1


@pytest.mark.parametrize("m", [251, 65521, 2**31 - 1, 2**32 - 5])
@pytest.mark.parametrize("nvec", [2, 4, 8, 16, 33])
def test_which_blocks_run_on_the_layout(lib, m, nvec):
    """Large enough that a binned plan's blocks of every width go to the layout,
    from the second on, in both directions; the result is the plan's."""
    n = 2**21 // (2 * 11) + 1000
    A = gen.uniform_matrix(nvec, n, n + 17, np.full(n, 11), m, pm_fraction=0.2)
    M = lib.Matrix.from_csr(A)
    assert "panels" not in M.describe()
    for transpose in (False, True):
        check_apply(lib, M, A, nvec=nvec, seed=1, transpose=transpose)
        before = len(_staged(M))
        check_apply(lib, M, A, nvec=nvec, alpha=5, beta=m - 1, seed=2, transpose=transpose)
        assert len(_staged(M)) == before + 1 == 1 + int(transpose)
