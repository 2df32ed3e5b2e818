"""Batches in which a handle appears many times, against the CPU oracle: packed
and in-place blocks mixed, more pieces and more vectors than fit beside each
other, rows of several chunks (whose sums share words of the handle), repeated
calls, and a capture before and after the buffers are there."""
import numpy as np
import pytest

import gen
import oracle
from helpers import rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


def _matrix(m, long_rows, n=700):
    lengths = np.random.default_rng(m % 1000).integers(0, 30, n)
    if long_rows:
        lengths[3], lengths[9] = 1700, 513
    return gen.uniform_matrix(m % 91, n, 2103, lengths, m, pm_fraction=0.2)


def _run(lib, mats, hs, picks, widths, seed):
    import torch
    xs = [rand_block(seed + i, mats[j].ncols, s, mats[j].modulus) for i, (j, s) in enumerate(zip(picks, widths))]
    ys = [torch.full((mats[j].nrows, s), -1, dtype=torch.int32, device="cuda") for j, s in zip(picks, widths)]
    lib.spmv_batch_apply([hs[j].handle for j in picks], [to_dev(x) for x in xs], ys, widths)
    for i, (j, s) in enumerate(zip(picks, widths)):
        want = oracle.csr_spmv(mats[j], xs[i])
        assert np.array_equal(to_host(ys[i]).reshape(want.shape), want), (i, j, s)


@pytest.mark.parametrize("long_rows", [False, True])
@pytest.mark.parametrize("m", [251, 65521, 65537, 2**31 - 1, 2**32 - 5])
def test_one_handle_many_times(lib, m, long_rows):
    A = _matrix(m, long_rows)
    rng = np.random.default_rng(m % 77)
    for count in (2, 17, 90):
        M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
        for k in range(2):
            _run(lib, [A], [M], [0] * count, [int(v) for v in rng.integers(1, 33, count)], 1000 * k + count)
        _run(lib, [A], [M], [0] * count, [16] * count, 5000 + count)


def test_handles_repeated_unevenly(lib):
    mats = [_matrix(m, k % 2 == 1) for k, m in enumerate((3, 65536, 2**31 - 1, 2**31, 65521))]
    hs = [lib.Matrix.from_csr(a, transpose_mode=lib.TRANSPOSE.NONE) for a in mats]
    rng = np.random.default_rng(8)
    for k in range(4):
        picks = [int(j) for j in rng.choice(5, 60, p=[0.5, 0.3, 0.1, 0.05, 0.05])]
        _run(lib, mats, hs, picks, [int(v) for v in rng.integers(1, 33, 60)], 100 * k)


def test_captured_repeats(lib):
    import torch
    A = _matrix(65521, True)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    B = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    xs = [rand_block(k, A.ncols, 7, A.modulus) for k in range(6)]
    xd, ys = [to_dev(x) for x in xs], [torch.zeros((A.nrows, 7), dtype=torch.int32, device="cuda") for _ in xs]
    lib.spmv_batch_apply([B.handle] * 6, xd, ys, [7] * 6)       # the kernels are loaded
    lib.spmv_batch_apply([M.handle], xd[:1], ys[:1], [7])       # the layout, with room for one block
    s = torch.cuda.Stream()
    for _ in range(2):                                          # without room for six, then with it
        s.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lib.spmv_batch_apply([M.handle] * 6, xd, ys, [7] * 6)
        for y in ys:
            y.zero_()
        g.replay()
        torch.cuda.synchronize()
        for x, y in zip(xs, ys):
            assert np.array_equal(to_host(y), oracle.csr_spmv(A, x))
        lib.spmv_batch_apply([M.handle] * 6, xd, ys, [7] * 6)
