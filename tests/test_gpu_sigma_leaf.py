"""GPU parity of one M-Basis leaf with oracle/sigma.py, bit for bit, at the
largest orders of a launch and one above, where the columns of P and of R
divide unevenly (or not at all) among the CTAs that hold them."""
import numpy as np
import pytest

from oracle import sigma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [2, 65521, 2**31 - 1])
@pytest.mark.parametrize("m,n,d", [(1, 1, 32), (3, 2, 32), (5, 5, 33), (11, 8, 32), (14, 13, 31), (27, 16, 32), (20, 17, 24),
                                   (19, 18, 25)])
@pytest.mark.parametrize("dense", [1.0, 0.2])
def test_largest_leaves(lib, p, m, n, d, dense):
    rng = np.random.default_rng(m * 1000 + d)
    F = rng.integers(0, p, (d, m, n)) * (rng.random((d, m, n)) < dense)
    shift = [int(v) for v in rng.integers(-3, 4, m)]
    P, delta, e = lib.sigma_basis(p, np.ascontiguousarray(F, dtype=np.uint32), shift=shift)
    Po, do = sigma.mbasis(F.astype(object), d, shift, p)
    want = np.zeros((d + 1, m, m), dtype=np.int64)
    want[:Po.shape[0]] = np.asarray(Po, dtype=np.int64)
    assert delta == do and np.array_equal(P.cpu().numpy().view(np.uint32).astype(np.int64), want)
    assert not np.any(want[e + 1:])
