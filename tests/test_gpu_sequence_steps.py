"""GPU parity of block sequences with one launch per step (m > 2^16) against the
CPU oracle: block widths that do and do not fill four-word pieces, up to 32,
moduli on both sides of 2^31, rows of several chunks and empty rows, few and
many rows, short calls before the layout exists, and resumed sequences."""
import numpy as np
import pytest

import gen
import oracle
from helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


def _matrix(n, m, long_rows):
    rng = np.random.default_rng(n)
    lengths = rng.integers(0, min(n, 24) + 1, n)
    if long_rows:
        lengths[1], lengths[n // 2] = min(n, 1500), min(n, 513)
    A = gen.uniform_matrix(n, n, n, lengths, m, pm_fraction=0.2)
    A.val[::7] = m - 1
    return A


@pytest.mark.parametrize("m", [65537, 2**31 - 1, 2**31 + 11, 4294967291])
@pytest.mark.parametrize("n,s,long_rows", [(1, 1, False), (40, 3, False), (700, 8, False), (1601, 17, True), (2300, 32, True)])
def test_steps_against_oracle(lib, m, n, s, long_rows):
    A = _matrix(n, m, long_rows)
    X = gen.uniform_block(n, n, s, m).reshape(n, s)
    Y = gen.uniform_block(n, n, s, m, key=1).reshape(n, s)
    X[0], Y[-1] = m - 1, m - 1
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    want, Vw = oracle.csr_block_sequence(A, X, Y, 18, want_next=True)
    for nsteps in (3, 18, 2):          # before the layout, building it, with it
        S = M.block_sequence(to_dev(X), to_dev(Y), nsteps)
        assert np.array_equal(to_host(S), want[:nsteps]), nsteps
    S, V = M.block_sequence(to_dev(X), to_dev(Y), 18, want_next=True)
    assert np.array_equal(to_host(S), want) and np.array_equal(to_host(V), Vw)
    S, V = M.block_sequence(to_dev(X), to_dev(Y), 5, want_next=True)
    rest = M.resume_sequence(to_dev(X), V, 5, 13)
    assert np.array_equal(to_host(rest), want[5:]) and np.array_equal(to_host(V), Vw)
