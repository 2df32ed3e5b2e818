"""GPU parity of the persistent sequence kernel at the edges of its tiling,
against the CPU oracle: sizes around one 16-row group, one CTA's groups and
their batches, odd numbers of entries per row, rows of 0 to 16 entries in one
group, merged diagonals, values and residues at their largest, small moduli,
and one to many steps (the partial projections are summed two steps later)."""
import numpy as np
import pytest

import gen
import oracle
from helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


def _check(lib, A, s, nsteps, seed=0, fill=None):
    m = A.modulus
    X = gen.uniform_block(seed + 1, A.nrows, s, m).reshape(A.nrows, s)
    Y = gen.uniform_block(seed + 2, A.nrows, s, m, key=1).reshape(A.nrows, s)
    if fill is not None:
        X[:], Y[:] = fill, fill
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    S, V = M.block_sequence(to_dev(X), to_dev(Y), nsteps, want_next=True)
    want, Vw = oracle.csr_block_sequence(A, X, Y, nsteps, want_next=True)
    assert np.array_equal(to_host(S), want)
    assert np.array_equal(to_host(V), Vw)
    assert np.array_equal(to_host(M.block_sequence(to_dev(X), to_dev(Y), nsteps)), want)   # without the last product


@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 255, 2431, 2433, 40_000])
@pytest.mark.parametrize("nsteps", [1, 2, 3, 7])
def test_sizes_and_steps(lib, n, nsteps):
    rng = np.random.default_rng(n)
    lengths = rng.integers(0, min(n, 16) + 1, n)
    _check(lib, gen.uniform_matrix(n, n, n, lengths, 65521), 16 if n < 40_000 else 5, nsteps, seed=n)


@pytest.mark.parametrize("m", [2, 3, 251, 257, 65521, 65536])
@pytest.mark.parametrize("s", [1, 7, 16])
def test_moduli_and_largest_sums(lib, m, s):
    n = 500
    A = gen.uniform_matrix(m, n, n, np.full(n, 16), m)
    A.val[:] = m - 1
    _check(lib, A, s, 6, fill=m - 1)
    _check(lib, gen.wiedemann_matrix(seed=m, n=n, p=m), s, 6, seed=3)


def test_repeated_entries_on_diagonals(lib):
    # a dense diagonal stored twice is one entry; with 14 others the row is full
    n, m = 300, 65521
    rng = np.random.default_rng(4)
    rows = []
    for i in range(n):
        c = rng.choice(np.setdiff1d(np.arange(n), [i]), 14, replace=False)
        rows.append(np.sort(np.concatenate([[i, i], c])))
    col = np.concatenate(rows).astype(np.int32)
    val = rng.integers(1, m, col.size).astype(np.uint32)
    A = gen.synth.CSR(n, n, np.arange(n + 1, dtype=np.int64) * 16, col, val, m, "twice")
    _check(lib, A, 16, 5)
