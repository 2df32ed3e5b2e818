"""Batched products over changing sets of handles, against the CPU oracle: the
same handle several times in one call, subsets and orders that change from call
to call, more matrices than one launch takes, moduli and widths that mix 16-bit
and 32-bit packing, empty matrices, rows of several chunks, and a call captured
in a graph."""
import numpy as np
import pytest

import gen
import oracle
from helpers import rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


def _problems():
    out = []
    for j, m in enumerate([3, 65521, 65536, 65537, 2**31 - 1, 2**31, 4294967291]):
        n = 60 + 31 * j
        lengths = np.random.default_rng(j).integers(0, 30, n)
        lengths[3], lengths[7] = 1700, 513     # rows of several chunks
        out.append(gen.uniform_matrix(j, n, 2100 + j, lengths, m, pm_fraction=0.2))
    return out


def _check(lib, mats, mods, picks, widths, seed):
    import torch
    xs = [rand_block(seed + i, mods[j].ncols, s, mods[j].modulus) for i, (j, s) in enumerate(zip(picks, widths))]
    ys = [torch.full((mods[j].nrows, s), -1, dtype=torch.int32, device="cuda") for j, s in zip(picks, widths)]
    lib.spmv_batch_apply([mats[j].handle for j in picks], [to_dev(x) for x in xs], ys, widths)
    for i, (j, s) in enumerate(zip(picks, widths)):
        want = oracle.csr_spmv(mods[j], xs[i])
        assert np.array_equal(to_host(ys[i]).reshape(want.shape), want), (i, j, s)


def test_repeated_handles_and_changing_sets(lib):
    A = _problems()
    mats = [lib.Matrix.from_csr(a, transpose_mode=lib.TRANSPOSE.NONE) for a in A]
    rng = np.random.default_rng(1)
    for k in range(6):
        picks = [int(j) for j in rng.integers(0, len(A), int(rng.integers(1, 12)))]
        _check(lib, mats, A, picks, [int(s) for s in rng.integers(1, 33, len(picks))], 10 * k)
    _check(lib, mats, A, [2, 2, 2, 4], [5, 16, 1, 32], 99)


def test_more_matrices_than_one_launch_takes(lib):
    A = [gen.uniform_matrix(j, 5 + j % 7, 9, np.full(5 + j % 7, 1 + j % 4), 65521 if j % 2 else 2**31 - 1)
         for j in range(520)]
    mats = [lib.Matrix.from_csr(a, transpose_mode=lib.TRANSPOSE.NONE) for a in A]
    _check(lib, mats, A, list(range(520)), [1 + j % 5 for j in range(520)], 7)


def test_captured_batch(lib):
    import torch
    A = _problems()[:3]
    mats = [lib.Matrix.from_csr(a, transpose_mode=lib.TRANSPOSE.NONE) for a in A]
    _check(lib, mats, A, [0, 1, 2], [4, 7, 16], 3)          # builds the layouts
    xs = [to_dev(rand_block(50 + j, a.ncols, 7, a.modulus)) for j, a in enumerate(A)]
    ys = [torch.zeros((a.nrows, 7), dtype=torch.int32, device="cuda") for a in A]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        lib.spmv_batch_apply([M.handle for M in mats], xs, ys, [7] * 3)
    for _ in range(2):
        for y in ys:
            y.zero_()
        g.replay()
        torch.cuda.synchronize()
        for a, x, y in zip(A, xs, ys):
            assert np.array_equal(to_host(y), oracle.csr_spmv(a, to_host(x)))
