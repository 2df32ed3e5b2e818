"""Sequences at m > 2^16 on the block layout: when it is built (a sequence long
enough, or several that are together), what runs before, and steps on it at the
widths around its pieces and groups of outputs, against the CPU oracle."""
import numpy as np
import pytest

import gen
import oracle
from helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


def _case(n, s, m):
    rng = np.random.default_rng(n + s)
    lengths = rng.integers(0, min(n, 24) + 1, n)
    if n > 600:
        lengths[1] = 530
    A = gen.uniform_matrix(n, n, n, lengths, m, pm_fraction=0.2)
    return A, gen.uniform_block(n, n, s, m).reshape(n, s), gen.uniform_block(n, n, s, m, key=1).reshape(n, s)


@pytest.mark.parametrize("m", [65537, 2**31 - 1, 4294967291])
@pytest.mark.parametrize("n,s", [(1, 1), (30, 2), (700, 5), (900, 7), (700, 8), (650, 9), (640, 16), (800, 17), (700, 24), (701, 31), (900, 32)])
def test_first_call_builds(lib, m, n, s):
    A, X, Y = _case(n, s, m)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    want, Vw = oracle.csr_block_sequence(A, X, Y, 50, want_next=True)
    for _ in range(2):
        S, V = M.block_sequence(to_dev(X), to_dev(Y), 50, want_next=True)
        assert "blocks:" in M.describe()
        assert np.array_equal(to_host(S), want) and np.array_equal(to_host(V), Vw)


def test_short_sequences_build_together(lib):
    m, n, s = 2**31 - 1, 700, 8
    A, X, Y = _case(n, s, m)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    want, Vw = oracle.csr_block_sequence(A, X, Y, 64, want_next=True)
    S, V = M.block_sequence(to_dev(X), to_dev(Y), 16, want_next=True)
    got = [to_host(S)]
    for k in range(1, 4):
        assert ("blocks:" in M.describe()) == (k > 2)      # 16, 32, then 48 steps
        got.append(to_host(M.resume_sequence(to_dev(X), V, 16 * k, 16)))
    assert np.array_equal(np.concatenate(got), want) and np.array_equal(to_host(V), Vw)


@pytest.mark.parametrize("s", [1, 7, 16])
def test_no_memory_for_the_steps(lib, s):
    # test hook 32: the scratch of the layout's steps cannot be had
    m = 2**31 - 1
    A, X, Y = _case(700, s, m)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE, test_hooks=32)
    want, Vw = oracle.csr_block_sequence(A, X, Y, 50, want_next=True)
    for _ in range(2):
        S, V = M.block_sequence(to_dev(X), to_dev(Y), 50, want_next=True)
        assert np.array_equal(to_host(S), want) and np.array_equal(to_host(V), Vw)
