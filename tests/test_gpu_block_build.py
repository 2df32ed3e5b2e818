"""Building a block layout: the caller's stream is not waited for, a capture that
goes on elsewhere is not disturbed, and the layout is right for matrices whose
arrays go up together or apart, empty ones among them."""
import time

import numpy as np
import pytest

import gen
import oracle
from helpers import rand_block, to_dev, to_host
from test_gpu_spmv import check_apply

pytestmark = pytest.mark.gpu


def _matrix(n=60_000, m=65521):
    return gen.uniform_matrix(6, n, n + 5, np.full(n, 23), m, pm_fraction=0.2)


def test_building_does_not_wait_for_the_stream(lib):
    import torch
    A = _matrix()
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    X = [rand_block(k, A.ncols, 16, A.modulus) for k in range(3)]
    x = [to_dev(v) for v in X]
    y = [torch.zeros((A.nrows, 16), dtype=torch.int32, device="cuda") for _ in X]
    G = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    for k in range(2):
        G.apply(x[k], y[k])                    # the kernels are loaded
    assert "blocks:" in G.describe()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(s):
        M.apply(x[0], y[0])
        torch.cuda._sleep(2_000_000_000)       # about a second
        t = time.perf_counter()
        M.apply(x[1], y[1])                    # the second block builds the layout
        M.apply(x[2], y[2])
        spent = time.perf_counter() - t
        done.record()
        assert not done.query() and spent < 0.3, spent
    assert "blocks:" in M.describe()
    torch.cuda.synchronize()
    for a, b in zip(X, y):
        assert np.array_equal(to_host(b), oracle.csr_spmv(A, a))


def test_building_while_another_stream_is_captured(lib):
    import torch
    A = _matrix()
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    B = _matrix(3000)
    N = lib.Matrix.from_csr(B, transpose_mode=lib.TRANSPOSE.NONE)
    x, xb = rand_block(1, A.ncols, 16, A.modulus), rand_block(2, B.ncols, 1, B.modulus)
    xd, yd = to_dev(x), torch.zeros((A.nrows, 16), dtype=torch.int32, device="cuda")
    xbd, ybd = to_dev(xb), torch.zeros(B.nrows, dtype=torch.int32, device="cuda")
    M.apply(xd, yd)
    N.apply(xbd, ybd)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):                  # captured with cudaStreamCaptureModeGlobal
        N.apply(xbd, ybd)
        # a block product on a stream that is not captured; this one builds its layout
        lib.spmv_apply(M.handle, xd, 16, yd, 16, 16, stream=side)
    assert "blocks:" in M.describe()
    ybd.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(to_host(ybd), oracle.csr_spmv(B, xb).reshape(-1))
    assert np.array_equal(to_host(yd), oracle.csr_spmv(A, x))


@pytest.mark.parametrize("m", [251, 2**31 - 1])
@pytest.mark.parametrize("rows,cols,mean", [(1, 1, 0), (7, 3, 2), (3, 4000, 1300), (33_000, 900, 5), (900, 70_000, 200), (9000, 9000, 40)])
def test_layouts_of_many_shapes(lib, m, rows, cols, mean):
    rng = np.random.default_rng(rows)
    lengths = rng.integers(0, min(cols, 2 * mean) + 1, rows)
    A = gen.uniform_matrix(rows, rows, cols, lengths, m, pm_fraction=0.1)
    M = lib.Matrix.from_csr(A)
    for k in range(2):
        for nvec in (5, 32):
            M.launches(False, nvec)
            check_apply(lib, M, A, nvec=nvec, seed=k)
            check_apply(lib, M, A, nvec=nvec, alpha=3, beta=4, seed=k + 5, transpose=True)


@pytest.mark.parametrize("even", [0, 1, 1000])
@pytest.mark.parametrize("n,mean", [(300, 7), (40_000, 60)])
def test_patterns_with_and_without_even_values(lib, n, mean, even):
    """GF(2) patterns whose values are all odd go up without them; one even
    value, or many, and they go up too.  Arrays below and above the upload's
    slots (2 MB)."""
    from oracle import gf2
    A = gen.uniform_matrix(n + even, n, n + 9, np.full(n, mean), 2)
    A.val[:] = 1
    A.val[:even] = 0
    A.val[-1] = 0 if even else 1
    M = lib.Matrix.from_csr(A)
    for transpose in (False, True):
        x = gen.uniform_block(4, n if transpose else n + 9, 4, 2**32 - 1).view(np.uint64)
        y = M.apply_gf2(x, transpose=transpose).cpu().numpy().view(np.uint64)
        assert np.array_equal(y, gf2.csr_gf2(A, x, transpose))


def test_layouts_of_a_batch_are_built_together(lib):
    """Handles with and without a layout, empty ones, one that finds no memory at
    first, moduli and widths mixed, more than one build's temporary memory (64
    MB), and then the same again with what is there."""
    import torch
    shapes = [(0, 5, 0), (40, 0, 0), (300, 200, 9)] + [(50_000 + k, 40_000, 20) for k in range(9)] + [(17, 90_000, 1500)]
    mats, hs = [], []
    for k, (rows, cols, mean) in enumerate(shapes):
        m = (65521, 2**31 - 1, 251, 2**32 - 5)[k % 4]
        mats.append(gen.uniform_matrix(k, rows, cols, np.full(rows, mean), m, pm_fraction=0.1))
        hs.append(lib.Matrix.from_csr(mats[-1], transpose_mode=lib.TRANSPOSE.NONE, test_hooks=16 if k == 5 else 0))
    hs[3].launches(False, 32)       # (its layout may be there already)
    for k in range(4):
        nv = [1 + (7 * j + 3 * k) % 32 for j in range(len(hs))]
        xs = [rand_block(k * 100 + j, A.ncols, v, A.modulus).reshape(A.ncols, v) for j, (A, v) in enumerate(zip(mats, nv))]
        ys = [torch.full((A.nrows, v), -1, dtype=torch.int32, device="cuda") for A, v in zip(mats, nv)]
        lib.spmv_batch_apply([h.handle for h in hs], [to_dev(x) for x in xs], ys, nv)
        for j, A in enumerate(mats):
            if A.nrows:
                want = oracle.csr_spmv(A, xs[j]).reshape(A.nrows, nv[j]) if A.ncols else np.zeros((A.nrows, nv[j]), np.uint32)
                assert np.array_equal(to_host(ys[j]), want), (k, j)
    assert all("blocks:" in h.describe() for h, A in zip(hs, mats) if A.nrows)
