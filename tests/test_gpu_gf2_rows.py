"""GF(2) products where the row classes, chunks and pieces of a row of X meet:
row lengths around the class and chunk limits, word counts around the pieces of
a pass, rows of X off the 16-byte boundary, calls on one handle from two
streams.  Bit-exact against the oracle."""
import numpy as np
import pytest

import gen
from oracle import gf2

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 511, 512, 513, 1024, 1025, 2049, 0, 4100]


def _matrix(seed, reps=3):
    rng = np.random.default_rng(seed)
    lens = np.concatenate([rng.permutation(LENGTHS) for _ in range(reps)])
    ncols = 4111
    # odd entries as listed, even ones in between: the pattern is what has the lengths
    ptr, col, val = [0], [], []
    for n in lens:
        c = rng.permutation(ncols)[: n + rng.integers(0, 4)].astype(np.int32)
        v = np.where(np.arange(c.size) < n, 1, 0).astype(np.uint32)
        p = rng.permutation(c.size)
        col.append(c[p])
        val.append(v[p])
        ptr.append(ptr[-1] + c.size)
    return gen.CSR(lens.size, ncols, np.array(ptr, np.int64), np.concatenate(col), np.concatenate(val), 2)


def _words(seed, rows, w):
    return np.random.default_rng(seed).integers(0, 2**64, (rows, w), dtype=np.uint64, endpoint=False)


@pytest.mark.parametrize("words", [1, 2, 3, 6, 8, 9, 16, 17, 18, 34])
@pytest.mark.parametrize("transpose", [False, True])
def test_lengths_and_words(lib, words, transpose):
    import torch
    A = _matrix(5)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    rows, outs = (A.nrows, A.ncols) if transpose else (A.ncols, A.nrows)
    X, Y0 = _words(7 + words, rows, words), _words(8 + words, outs, words)
    want = gf2.csr_gf2(A, X, transpose=transpose)
    flat = torch.zeros(rows * words + 1, dtype=torch.int64, device="cuda")
    for off in (0, 1):   # on and off the 16-byte boundary
        x = flat[off:off + rows * words].view(rows, words)
        x.copy_(torch.from_numpy(X.view(np.int64)))
        for acc in (False, True):
            y = torch.from_numpy(Y0.view(np.int64)).cuda()
            lib.spmv_apply_gf2(M.handle, transpose, x, y, words, acc)
            got = y.cpu().numpy().view(np.uint64)
            assert np.array_equal(got, want ^ Y0 if acc else want), (words, transpose, off, acc)


def test_two_streams(lib):
    import torch
    A = _matrix(6, reps=40)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    X = [_words(20 + i, A.ncols, 4) for i in range(2)]
    x = [torch.from_numpy(v.view(np.int64)).cuda() for v in X]
    M.apply_gf2(x[0])
    streams = [torch.cuda.Stream() for _ in range(2)]
    ys = [[torch.empty((A.nrows, 4), dtype=torch.int64, device="cuda") for _ in range(20)] for _ in range(2)]
    torch.cuda.synchronize()
    for k in range(20):
        for i, s in enumerate(streams):
            lib.spmv_apply_gf2(M.handle, False, x[i], ys[i][k], 4, False, stream=s)
    torch.cuda.synchronize()
    for i in range(2):
        want = gf2.csr_gf2(A, X[i])
        assert all(np.array_equal(y.cpu().numpy().view(np.uint64), want) for y in ys[i])
