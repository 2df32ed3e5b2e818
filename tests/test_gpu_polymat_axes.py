"""GPU parity of the polynomial-matrix transforms at the edges of their tiles:
every transform length from 16 to 2^15 (one axis up to 256 points, two above),
one, two and three primes, block sizes whose entries do not fill a 32-lane
tile or a 4 x 4 output tile, and products that end just below, at and above a
power of two.  Results are integers: they equal the oracle's."""
import numpy as np
import pytest

from oracle import polymat

pytestmark = pytest.mark.gpu


def _rand(seed, d, s, p):
    return np.random.default_rng(seed).integers(0, p, (d + 1, s, s), dtype=np.int64).astype(np.uint32)


# da + db + 1 = 2^k - 1, 2^k, 2^k + 1 around the single-pass limit and every two-axis split
LENGTHS = [(7, 8), (8, 8), (100, 155), (127, 128), (128, 128), (200, 311), (500, 523), (1000, 1047), (2000, 2095),
           (4000, 4191), (8000, 8383), (16383, 16384)]


@pytest.mark.parametrize("p", [3, 65521, 2**31 - 1])    # one, two and three primes at these lengths
@pytest.mark.parametrize("da,db", LENGTHS)
def test_every_length(lib, p, da, db):
    s = 3
    A, B = _rand(da, da, s, p), _rand(db + 1, db, s, p)
    C = lib.polymat_mul(p, A, B).cpu().numpy().view(np.uint32).astype(np.int64)
    assert C.shape == (da + db + 1, s, s)
    for k in (0, 1, da // 2, da, db, da + db - 1, da + db):    # single coefficients, by definition
        lo, hi = max(0, k - db), min(da, k)
        want = np.zeros((s, s), dtype=object)
        for a in range(lo, hi + 1):
            want = want + np.dot(A[a].astype(object), B[k - a].astype(object))
        assert np.array_equal(C[k], (want % p).astype(np.int64)), (p, da, db, k)
    for x0 in (1, p - 2):                                      # all coefficients together
        rhs = np.dot(polymat.polymat_eval(A, x0, p), polymat.polymat_eval(B, x0, p)) % p
        assert np.array_equal(polymat.polymat_eval(C, x0, p), rhs), (p, da, db, x0)


@pytest.mark.parametrize("s", [1, 2, 4, 5, 7, 17, 20, 31, 32])
def test_every_block_shape(lib, s):
    p, da, db = 2**31 - 1, 21, 12
    A, B = _rand(s, da, s, p), _rand(s + 50, db, s, p)
    A[0], B[-1] = p - 1, p - 1                                 # rows of the largest terms
    got = lib.polymat_mul(p, A, B).cpu().numpy().view(np.uint32).astype(np.int64)
    assert np.array_equal(got, polymat.polymat_mul(A, B, p))
