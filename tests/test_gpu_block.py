"""GPU parity of blocks on the block layout (FFSPMV_FMT_AUTO handles) against
the CPU oracle, bit-exact: row lengths at the edges of every length class and
of the chunks of long rows, moduli on both sides of the 16-bit, 31-bit and
32-bit limits, block widths around the pieces and passes, strided and
unaligned blocks, the largest values, and the calls that keep the plan's own
path (few small products, a block captured before the layout exists)."""
import numpy as np
import pytest

import gen
import oracle
from helpers import rand_block, to_dev, to_host
from test_gpu_spmv import check_apply

pytestmark = pytest.mark.gpu

# around quads (4), classes (4, 8, 16, 32, 64), one chunk (512) and several
EDGES = [0, 1, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 511, 512, 513, 1024, 1025, 2600]


def edge_matrix(m, ncols=3001, copies=3, largest=False):
    rng = np.random.default_rng(m % 1000)
    lengths = np.array(EDGES * copies)
    rng.shuffle(lengths)
    A = gen.uniform_matrix(5, lengths.size, ncols, lengths, m, pm_fraction=0.2)
    if largest:
        A.val[:] = m - 1
    return A


@pytest.mark.parametrize("m", [2, 251, 65521, 65536, 65537, 2**31 - 1, 2**31, 2**31 + 11, 4294967291])
def test_row_lengths_and_widths(lib, m):
    A = edge_matrix(m)
    M = lib.Matrix.from_csr(A)
    for nvec in (2, 3, 4, 5, 7, 8, 9, 12, 15, 16, 17, 24, 25, 31, 32, 33, 65):
        assert M.launches(False, nvec) <= 2 * -(-nvec // 32), M.describe()   # the block layout
        check_apply(lib, M, A, nvec=nvec, alpha=(m - 2) % m, beta=5 % m, seed=nvec)
        check_apply(lib, M, A, nvec=nvec, transpose=True, seed=nvec + 1)


@pytest.mark.parametrize("m", [65521, 65536, 2**31, 4294967291])
def test_largest_sums(lib, m):
    A = edge_matrix(m, largest=True)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    assert M.launches(False, 32) <= 2    # builds the layout
    for nvec in (3, 16, 32):
        X = np.full((A.ncols, nvec), m - 1, dtype=np.uint32)
        assert np.array_equal(to_host(M.apply(to_dev(X))), oracle.csr_spmv(A, X))


@pytest.mark.parametrize("m", [65521, 2**31 - 1])
def test_strided_and_unaligned_blocks(lib, m):
    import torch
    A = edge_matrix(m)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    assert M.launches(False, 32) <= 2    # builds the layout
    for nvec, ldx, ldy, ox, oy in ((8, 8, 8, 1, 0), (8, 8, 8, 0, 1), (8, 12, 16, 0, 0), (7, 9, 11, 3, 2), (16, 20, 17, 0, 0)):
        x = rand_block(nvec, A.ncols, ldx, m)
        y0 = rand_block(nvec + 1, A.nrows, ldy, m)
        xb = torch.zeros(x.size + 8, dtype=torch.int32, device="cuda")
        yb = torch.zeros(y0.size + 8, dtype=torch.int32, device="cuda")
        xb[ox:ox + x.size] = to_dev(x).reshape(-1)
        yb[oy:oy + y0.size] = to_dev(y0).reshape(-1)
        lib.spmv_apply(M.handle, xb[ox:], ldx, yb[oy:], ldy, nvec, 3, 4)
        got = to_host(yb)
        want = y0.copy()
        want[:, :nvec] = oracle.csr_spmv(A, np.ascontiguousarray(x[:, :nvec]), y=np.ascontiguousarray(y0[:, :nvec]),
                                         alpha=3, beta=4)
        assert np.array_equal(got[oy:oy + y0.size].reshape(y0.shape), want)   # columns past nvec untouched
        assert not got[:oy].any() and not got[oy + y0.size:].any()


def test_repeated_calls_and_both_directions(lib):
    # the sums of long rows are cleared by the call that used them
    A = edge_matrix(65521)
    M = lib.Matrix.from_csr(A)
    for k in range(3):
        for nvec in (16, 3):
            check_apply(lib, M, A, nvec=nvec, seed=k)
            check_apply(lib, M, A, nvec=nvec, transpose=True, seed=k + 9)


@pytest.mark.parametrize("m,nvec", [(251, 4), (65521, 3), (65521, 16), (2**31 - 1, 2)])
def test_blocks_of_a_panel_handle(lib, m, nvec):
    n = 40_000
    A = gen.powerlaw_matrix(seed=8, n=n, mean=56.0, lmax=9000, m=m)   # more than 2^21 entries
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    assert "panels" in M.describe() and A.nnz >= 1 << 21
    check_apply(lib, M, A, nvec=nvec, alpha=7, beta=m - 1, seed=nvec)
    assert M.launches(False, nvec) <= 2


def test_captured_before_the_layout_exists(lib):
    import torch
    A = gen.tiny_matrix()
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    X = rand_block(4, A.ncols, 7, A.modulus)
    x, y = to_dev(X), torch.zeros((A.nrows, 7), dtype=torch.int32, device="cuda")
    lib.spmv_apply(M.handle, x, 7, y, 7, 1)           # one vector: the kernels are loaded, no layout is built
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    for _ in range(2):                                # captured without the layout, then with it
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lib.spmv_apply(M.handle, x, 7, y, 7, 7)
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(to_host(y), oracle.csr_spmv(A, X))
        assert np.array_equal(to_host(M.apply(x)), oracle.csr_spmv(A, X))
