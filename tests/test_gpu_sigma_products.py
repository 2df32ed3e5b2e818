"""GPU parity of the products by definition between the leaves of a
sigma-basis (up to order 200) with oracle/sigma.py, bit for bit, on both sides
of what takes them to 16-bit pairs: modulus up to 2^16, rows and columns in
multiples of four."""
import numpy as np
import pytest

from oracle import sigma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [3, 65521, 65537])
@pytest.mark.parametrize("m,n,d", [(4, 4, 70), (8, 4, 129), (12, 8, 66), (20, 16, 50), (32, 28, 49), (6, 4, 70), (8, 3, 70)])
def test_pairs(lib, p, m, n, d):
    rng = np.random.default_rng(m + d)
    F = np.where(rng.random((d, m, n)) < 0.5, p - 1, rng.integers(0, p, (d, m, n)))
    P, delta, _ = lib.sigma_basis(p, np.ascontiguousarray(F, dtype=np.uint32))
    Po, do = sigma.pmbasis(F.astype(object), d, [0] * m, p, base=32)
    want = np.zeros((d + 1, m, m), dtype=np.int64)
    want[:Po.shape[0]] = np.asarray(Po, dtype=np.int64)
    assert delta == do and np.array_equal(P.cpu().numpy().view(np.uint32).astype(np.int64), want)
