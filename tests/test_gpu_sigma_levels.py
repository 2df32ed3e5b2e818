"""GPU parity of the sigma-basis at the edges of its levels, against
oracle/sigma.py bit for bit: orders around one leaf, around the nodes that run
without the host, and above; every register width of the leaf (n up to 8, 16,
32), p = 2 (no Montgomery form), primes on both sides of the limit from which
sums are folded, shifts far apart, and inputs whose orders lack pivots.  Where
the order is too large for the oracle: P F = 0 mod x^d through random
fingerprints, and the degrees of the oracle's own start."""
import numpy as np
import pytest

from oracle import sigma

pytestmark = pytest.mark.gpu


def _gpu(lib, p, F, shift=None, base=0):
    P, delta, e = lib.sigma_basis(p, np.ascontiguousarray(F, dtype=np.uint32), shift=shift, base=base)
    return P.cpu().numpy().view(np.uint32).astype(np.int64), delta, e


@pytest.mark.parametrize("p", [2, 3, 65521, 67108859, 67108879, 2**31 - 1])
@pytest.mark.parametrize("m,n,d", [(1, 1, 1), (2, 1, 17), (5, 3, 33), (9, 8, 16), (12, 9, 20), (17, 16, 15), (18, 17, 5),
                                   (32, 31, 4)])
def test_leaf_shapes(lib, p, m, n, d):
    rng = np.random.default_rng(m * 100 + d)
    F = rng.integers(0, p, (d, m, n))
    shift = [int(v) for v in rng.integers(-2, 5, m)]
    for Fx, sh in ((F, None), (F * (rng.random(F.shape) < 0.3), shift)):
        P, delta, e = _gpu(lib, p, Fx, sh)
        Po, do = sigma.mbasis(Fx.astype(object), d, sh or [0] * m, p)
        want = np.zeros((d + 1, m, m), dtype=np.int64)
        want[:Po.shape[0]] = np.asarray(Po, dtype=np.int64)
        assert delta == do and np.array_equal(P, want)
        assert e == max(0, min(d, max(do) - min(sh or [0])))


@pytest.mark.parametrize("d", [65, 130, 199, 201])
def test_levels(lib, d):
    p, m, n = 65521, 4, 2
    rng = np.random.default_rng(d)
    F = rng.integers(0, p, (d, m, n))
    P, delta, _ = _gpu(lib, p, F)
    Po, do = sigma.pmbasis(F.astype(object), d, [0] * m, p, base=32)
    want = np.zeros((d + 1, m, m), dtype=np.int64)
    want[:Po.shape[0]] = np.asarray(Po, dtype=np.int64)
    assert delta == do and np.array_equal(P, want)


@pytest.mark.parametrize("p,m,n,d", [(65521, 32, 16, 402), (2**31 - 1, 16, 8, 1030), (65521, 7, 5, 3001),
                                     (2**31 - 1, 31, 30, 250)])
def test_approximant_at_larger_orders(lib, p, m, n, d):
    rng = np.random.default_rng(d)
    F = rng.integers(0, p, (d, m, n))
    P, delta, e = _gpu(lib, p, F)
    assert sum(delta) == n * d and not np.any(P[e + 1:])   # det P = c x^(n d) for generic F
    for seed in (1, 2):
        fr = np.random.default_rng(seed)
        u, w = fr.integers(0, p, m), fr.integers(0, p, n)
        uP = np.array([[int(v) for v in np.dot(u.astype(object), Pk.astype(object)) % p] for Pk in P[:e + 1]])
        Fw = np.array([[int(v) for v in np.dot(Fk.astype(object), w.astype(object)) % p] for Fk in F])
        r = np.zeros(d, dtype=object)
        for j in range(m):
            # exact: 16-bit halves, sums below 2^47 2^11
            for s, half in ((0, uP[:, j] & 0xFFFF), (16, uP[:, j] >> 16)):
                r = (r + np.convolve(half, Fw[:, j])[:d].astype(object) * (1 << s)) % p
        assert not np.any(r)
