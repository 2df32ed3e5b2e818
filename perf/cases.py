"""The work that users of this library have it do, as measurable cases.

Every case goes through the public entry points, with the plan (the matrix
handle) and the inputs in hand, as a program that iterates with one matrix has
them.  Eight families:

* ``product``   y = A x, z = A^T x, or y = alpha A x + beta y: one vector;
* ``block``     the same with a block of vectors;
* ``sequence``  the block-Wiedemann sequence S_i = X^T A^i Y;
* ``rank``      the whole pipeline on one matrix: sequence, sigma-basis of
                [S; -I], deg det and codeg det of its generator;
* ``batch``     many uneven products with their own moduli in one launch;
* ``gf2``       products over GF(2) with 64 packed vectors per word;
* ``polymat``   a product of polynomial matrices;
* ``sigma``     the sigma-basis of a block sequence.

Matrices are drawn on the device from the seed: uniform, banded or power-law
rows with distinct columns, a fifth of the values +1 or -1.  Moduli are those
of the tests and the benchmark: 3 (values +-1), 251, 65521, 2^31 - 1 and
2^32 - 5.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1004_3719_gb300 as ff

P16, P31, P32 = 65521, 2**31 - 1, 2**32 - 5


def listed():
    return [
        # the smallest call: a 2000 x 2000 matrix with ten entries per row, where latency is all there is
        dict(name="product-tiny", kind="product", rows=2000, cols=2000, mean=10, shape="uniform", m=P16,
             what="both", axpby=False),
        # the headline: A x and A^T x on the 1M x 1M power-law matrix, as a Wiedemann or Lanczos iteration takes them
        dict(name="product-1m", kind="product", rows=1_000_000, cols=1_000_000, mean=16, shape="powerlaw", m=P16,
             what="both", axpby=False),
        # a word-size prime, a rectangular matrix of odd sizes, and the alpha/beta form
        dict(name="product-wide", kind="product", rows=300_007, cols=200_003, mean=22, shape="uniform", m=P31,
             what="A", axpby=True),
        # the transposed product over Z/3Z of a banded matrix, all of whose values are +-1
        dict(name="product-ternary", kind="product", rows=700_001, cols=700_001, mean=17, shape="banded", m=3,
             what="AT", axpby=False),
        # a block of 16 vectors on the 1M matrix: one step of a block method
        dict(name="block-1m", kind="block", rows=1_000_000, cols=1_000_000, mean=16, shape="powerlaw", m=P16,
             what="A", axpby=False, nvec=16),
        # a ragged block of 7 vectors, transposed, alpha/beta form, word-size prime
        dict(name="block-wide", kind="block", rows=120_011, cols=90_001, mean=23, shape="powerlaw", m=P31,
             what="AT", axpby=True, nvec=7),
        # the block-Wiedemann sequence of the 100k matrix, whole: 2 N / s + 2 steps with s = 16
        dict(name="sequence-100k", kind="sequence", rows=100_000, m=P16, s=16, steps=12_502),
        # a rank from beginning to end at a word-size prime
        dict(name="rank-wide", kind="rank", rows=4001, m=P31, s=8),
        # uneven problems in one launch, each with its own prime and block width
        dict(name="batch-48", kind="batch", count=48, rows_lo=1000, rows_hi=200_000, s_hi=32, sizes=1004),
        # 64 packed vectors over GF(2) on the 1M pattern
        dict(name="gf2-1m", kind="gf2", rows=1_000_000, cols=1_000_000, mean=16, shape="powerlaw", words=1,
             transpose=False),
        # the top product of the sigma-basis of the 100k sequence
        dict(name="polymat-6250", kind="polymat", s=16, da=6250, db=6250, m=P16),
        # the sigma-basis of the 100k sequence: the generator step of block Wiedemann
        dict(name="sigma-12502", kind="sigma", s=16, order=12_502, m=P16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "product", "block", "block", "sequence", "rank", "batch", "gf2",
                       "polymat", "sigma"])
    if kind in ("product", "block", "gf2"):
        rows = _log(rng, 2000, 1_000_000)
        cols = min(1_000_000, max(500, int(rows * rng.uniform(0.5, 1.3))))
        shape = rng.choice(["uniform", "banded", "powerlaw"])
        c = dict(kind=kind, rows=rows, cols=cols, mean=rng.randint(3, 24 if rows < 600_000 else 16), shape=shape)
        if kind == "gf2":
            return dict(c, words=rng.choice([1, 1, 2, 3, 4]), transpose=rng.random() < 0.5)
        c.update(m=rng.choice([3, 251, P16, P16, P31, P31, P32]), what=rng.choice(["A", "AT", "both"]),
                 axpby=rng.random() < 0.4)
        if kind == "block":
            c["nvec"] = rng.randint(2, min(32, max(2, 128_000_000 // (rows * c["mean"]))))
        return c
    if kind == "sequence":
        return dict(kind=kind, rows=_log(rng, 2000, 100_000), m=rng.choice([251, P16, P16]), s=rng.randint(1, 16),
                    steps=_log(rng, 60, 12_000))
    if kind == "rank":
        return dict(kind=kind, rows=_log(rng, 400, 4000), m=rng.choice([P16, P31]), s=rng.randint(4, 16))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 48), rows_lo=rng.choice([200, 1000]),
                    rows_hi=_log(rng, 5000, 200_000), s_hi=rng.choice([4, 16, 32]),
                    sizes=rng.randint(0, 10_000))
    if kind == "polymat":
        m = rng.choice([P16, P31])
        return dict(kind=kind, s=rng.randint(2, 24), da=_log(rng, 10, 6250), db=_log(rng, 10, 6250), m=m)
    return dict(kind=kind, s=rng.randint(2, 16), order=_log(rng, 40, 6000), m=rng.choice([P16, P16, P31]))


# ---------------------------------------------------------------------------
# Inputs, drawn on the device.
def _gen(seed, key):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + key)
    return g


def _bits32(v):
    """Residues below 2^32 (int64) as the 32-bit words that the library takes."""
    return torch.where(v >= 2**31, v - 2**32, v).to(torch.int32)


def _u64(t):
    """The residues of 32-bit words, as int64."""
    return t.to(torch.int64) & 0xFFFFFFFF


def _residues(g, shape, m):
    return torch.randint(0, m, shape, generator=g, device="cuda", dtype=torch.int64)


@functools.lru_cache(maxsize=None)
def _zipf_cdf(mean, lmax):
    k = np.arange(1, lmax + 1, dtype=np.float64)
    lo, hi = 0.0, 8.0
    for _ in range(60):
        a = 0.5 * (lo + hi)
        w = k ** -a
        lo, hi = (a, hi) if (k * w).sum() / w.sum() > mean else (lo, a)
    c = np.cumsum(k ** -lo)
    return c / c[-1]


def _csr(rows, cols, r, c, g, m):
    """row_ptr, col, val of the distinct positions (r, c), values mod m."""
    key = torch.unique(r * cols + c)
    r, c = key // cols, key % cols
    ptr = torch.zeros(rows + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(r, minlength=rows), 0)
    if m == 2:
        v = torch.ones_like(c)
    else:
        v = torch.randint(1, m, c.shape, generator=g, device="cuda", dtype=torch.int64)
        one = torch.rand(c.shape, generator=g, device="cuda")
        v = torch.where(one < 0.1, torch.ones_like(v), torch.where(one < 0.2, torch.full_like(v, m - 1), v))
    return ptr, c.to(torch.int32), _bits32(v)


def _matrix(g, rows, cols, mean, shape, m):
    dev = "cuda"
    if shape == "powerlaw":
        lmax = min(10_000, cols // 2)
        cdf = torch.from_numpy(_zipf_cdf(min(mean, lmax // 2), lmax)).to(dev)
        lengths = 1 + torch.searchsorted(cdf, torch.rand(rows, generator=g, device=dev, dtype=torch.float64))
        lengths.clamp_(max=lmax)
        lengths[int(rows // 3)] = lmax
    else:
        lengths = torch.randint(max(1, mean - mean // 2), mean + mean // 2 + 1, (rows,), generator=g, device=dev)
    r = torch.repeat_interleave(torch.arange(rows, device=dev), lengths)
    if shape == "banded":
        mid = r * cols // rows
        c = (mid + torch.randint(-32, 33, r.shape, generator=g, device=dev)).clamp_(0, cols - 1)
    else:
        c = torch.randint(0, cols, r.shape, generator=g, device=dev)
    return _csr(rows, cols, r, c, g, m)


def _wiedemann(g, n, m):
    """Four diagonals {0, +1, -1, +n/2} and six random entries per row."""
    i = torch.arange(n, device="cuda")
    r, c = [i.repeat_interleave(6)], [torch.randint(0, n, (6 * n,), generator=g, device="cuda")]
    for o in (0, 1, -1, n // 2):
        ok = (i + o >= 0) & (i + o < n)
        r.append(i[ok])
        c.append(i[ok] + o)
    return _csr(n, n, torch.cat(r), torch.cat(c), g, m)


def _is_prime(q):
    if any(q % f == 0 for f in (2, 3, 5, 7, 11, 13)):
        return False
    d, r = q - 1, 0
    while d % 2 == 0:
        d, r = d // 2, r + 1
    for a in (2, 3, 5, 7):
        x = pow(a, d, q)
        if x in (1, q - 1):
            continue
        if not any((x := x * x % q) == q - 1 for _ in range(r - 1)):
            return False
    return True


def _batch_problems(case):
    """(rows, mean, shape, prime, block width) of each problem: the case's own, not the seed's."""
    rng = np.random.default_rng([case["sizes"], 5])
    out = []
    for j in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["rows_lo"]), math.log(case["rows_hi"])))))
        p = int(rng.integers(2**30, 2**31)) | 1
        while not _is_prime(p):
            p = int(rng.integers(2**30, 2**31)) | 1
        out.append((n, 22, ("uniform", "banded", "powerlaw")[j % 3], p, int(rng.integers(1, case["s_hi"] + 1))))
    return out


def _rank_steps(case):
    return 2 * case["rows"] // case["s"] + 2


def _inputs(case, seed):
    """Everything that the seed decides, as device tensors."""
    g, k = _gen(seed, 1), case["kind"]
    if k in ("product", "block"):
        ptr, col, val = _matrix(g, case["rows"], case["cols"], case["mean"], case["shape"], case["m"])
        tail = (case["nvec"],) if k == "block" else ()
        d = dict(ptr=ptr, col=col, val=val)
        for name, n in (("x", case["cols"]), ("x2", case["cols"]), ("w", case["rows"]), ("w2", case["rows"])):
            d[name] = _bits32(_residues(g, (n, *tail), case["m"]))
        return d
    if k == "gf2":
        ptr, col, val = _matrix(g, case["rows"], case["cols"], case["mean"], case["shape"], 2)
        n = case["rows"] if case["transpose"] else case["cols"]
        x = torch.randint(-2**63, 2**63 - 1, (n, case["words"]), generator=g, device="cuda", dtype=torch.int64)
        return dict(ptr=ptr, col=col, val=val, x=x)
    if k in ("sequence", "rank"):
        ptr, col, val = _wiedemann(g, case["rows"], case["m"])
        X, Y = (_bits32(_residues(g, (case["rows"], case["s"]), case["m"])) for _ in range(2))
        return dict(ptr=ptr, col=col, val=val, X=X, Y=Y)
    if k == "batch":
        out = []
        for j, (n, mean, shape, p, s) in enumerate(_batch_problems(case)):
            gj = _gen(seed, 100 + j)
            out.append((n, p, s, *_matrix(gj, n, n, mean, shape, p), _bits32(_residues(gj, (n, s), p))))
        return dict(problems=out)
    if k == "polymat":
        return {v: _bits32(_residues(g, (case[d] + 1, case["s"], case["s"]), case["m"]))
                for v, d in (("A", "da"), ("B", "db"))}
    return dict(S=_bits32(_residues(g, (case["order"], case["s"], case["s"]), case["m"])))


# ---------------------------------------------------------------------------
def prepare(case, seed):
    st = dict(_inputs(case, seed), case=case)
    k = case["kind"]
    if k in ("product", "block", "gf2"):
        st["M"] = ff.Matrix(case["rows"], case["cols"], st.pop("ptr"), st.pop("col"), st.pop("val"), case.get("m", 2))
    elif k in ("sequence", "rank"):
        st["M"] = ff.Matrix(case["rows"], case["rows"], st.pop("ptr"), st.pop("col"), st.pop("val"), case["m"],
                            transpose_mode=ff.TRANSPOSE.NONE)
    elif k == "batch":
        prob = st.pop("problems")
        st["M"] = [ff.Matrix(n, n, ptr, col, val, p, transpose_mode=ff.TRANSPOSE.NONE, priority_format=ff.FMT.CSR)
                   for n, p, s, ptr, col, val, x in prob]
        st["x"] = [t[6] for t in prob]
        st["y"] = [torch.empty_like(t[6]) for t in prob]
        st["nvec"] = [t[2] for t in prob]
    return st


ALPHA, BETA = 5, 7


def run(st):
    case, M = st["case"], st.get("M")
    k = case["kind"]
    if k in ("product", "block"):
        out = []
        for on, fn, a, b in (("A", M.apply, "x", "x2"), ("AT", M.apply_transpose, "w", "w2")):
            if case["what"] in (on, "both"):
                y = fn(st[a])
                if case["axpby"]:
                    fn(st[b], y=y, alpha=ALPHA, beta=BETA)
                out.append(y)
        return out
    if k == "gf2":
        return M.apply_gf2(st["x"], transpose=case["transpose"])
    if k == "sequence":
        return M.block_sequence(st["X"], st["Y"], case["steps"], want_next=True)
    if k == "rank":
        S = M.block_sequence(st["X"], st["Y"], _rank_steps(case))
        P, delta, deg = ff.sigma_basis(case["m"], ff.sigma_wiedemann_input(case["m"], S))
        return [S, P, delta, deg, *ff.sigma_generator_degrees(case["m"], P, delta, case["s"])]
    if k == "batch":
        ff.spmv_batch_apply([h.handle for h in M], st["x"], st["y"], st["nvec"])
        return st["y"]
    if k == "polymat":
        return ff.polymat_mul(case["m"], st["A"], st["B"])
    P, delta, deg = ff.sigma_basis(case["m"], ff.sigma_wiedemann_input(case["m"], st["S"]))
    return [P, delta, deg]


# ---------------------------------------------------------------------------
def _nnz(case):
    return case["rows"] * case["mean"]


def _polymat_flops(s, n, da, db):
    """s x s by s x n, degrees da and db: three s x s transforms and one
    pointwise product at da + db + 1 points."""
    pts = da + db + 1
    return 2.0 * s * s * n * pts + 2.5 * (s * s + 2 * s * n) * pts * max(1.0, math.log2(pts))


def _sigma_flops(m, n, d):
    if d <= 32:
        return 2.0 * d * d * m * n * (m + n) / 2  # the row operations of d orders
    h = (d + 1) // 2
    e = max(1, h * n // m)
    return (_sigma_flops(m, n, h) + _sigma_flops(m, n, d - h) + _polymat_flops(m, n, e, d - 1)
            + _polymat_flops(m, m, e, e))


def work(case):
    k = case["kind"]
    if k in ("product", "block"):
        nv = case.get("nvec", 1)
        vb = 0 if case["m"] == 3 else 1 if case["m"] < 257 else 2 if case["m"] <= 65536 else 4
        n = (2 if case["what"] == "both" else 1) * (2 if case["axpby"] else 1)
        one = (4 + vb) * _nnz(case) + 4 * case["rows"] + 4 * nv * (case["rows"] + case["cols"])
        return {"bytes": n * one, "flops": 2.0 * n * _nnz(case) * nv}
    if k == "gf2":
        w = case["words"]
        return {"bytes": 4 * _nnz(case) + 4 * case["rows"] + 8 * w * (case["rows"] + case["cols"]),
                "flops": 64.0 * w * _nnz(case)}
    if k in ("sequence", "rank"):
        n, s = case["rows"], case["s"]
        steps = case["steps"] if k == "sequence" else _rank_steps(case)
        vb = 2 if case["m"] <= 65536 else 4
        out = {"bytes": 10 * n * (4 + vb) + 4 * n + 12 * n * s + 4 * steps * s * s,
               "flops": 2.0 * steps * (10 * n * s + n * s * s)}
        if k == "rank":
            out["bytes"] += 4 * steps * (2 * s) ** 2
            out["flops"] += _sigma_flops(2 * s, s, steps)
        return out
    if k == "batch":
        # the problems' expected sizes: rows log-uniform, 22 entries per row, mean block width
        lo, hi = case["rows_lo"], case["rows_hi"]
        n, s = case["count"] * (hi - lo) / math.log(hi / lo), (1 + case["s_hi"]) / 2
        return {"bytes": int(n * (22 * 8 + 4 + 8 * s)), "flops": 2.0 * 22 * n * s}
    s = case["s"]
    if k == "polymat":
        return {"bytes": 4 * s * s * 2 * (case["da"] + case["db"] + 1),
                "flops": _polymat_flops(s, s, case["da"], case["db"])}
    d = case["order"]
    return {"bytes": 4 * d * s * s + 4 * (d + 1) * 4 * s * s, "flops": _sigma_flops(2 * s, s, d)}


# ---------------------------------------------------------------------------
# The same results in plain 64-bit arithmetic.
def _mulmod(a, b, m):
    """a b mod m for int64 residues below m < 2^32 (the product in two halves)."""
    if m <= 2**31:
        return a * b % m
    return ((a * (b >> 16) % m << 16) + a * (b & 0xFFFF)) % m


def _spmm(ptr, col, val, x, n_out, m, transpose):
    """A x or A^T x mod m, one vector at a time."""
    r = torch.repeat_interleave(torch.arange(ptr.numel() - 1, device="cuda"), ptr.diff())
    c = col.to(torch.int64)
    src, dst = (r, c) if transpose else (c, r)
    v, xs = _u64(val), _u64(x).reshape(x.shape[0], -1)
    y = torch.zeros(n_out, xs.shape[1], dtype=torch.int64, device="cuda")
    for j in range(xs.shape[1]):
        y[:, j] = torch.zeros(n_out, dtype=torch.int64, device="cuda").index_add_(0, dst, _mulmod(v, xs[:, j][src], m))
    return (y % m).reshape(n_out, *x.shape[1:])


def _xt_v(X, V, m):
    """X^T V mod m through exact float64 products of 16-bit limbs."""
    out = 0
    for i in range(2):
        for j in range(2):
            a, b = ((X >> 16 * i) & 0xFFFF).double(), ((V >> 16 * j) & 0xFFFF).double()
            out = (out + _mulmod((a.T @ b).to(torch.int64) % m, torch.tensor(2**(16 * (i + j)) % m, device="cuda"), m)) % m
    return out


def _sequence(d, n, m, steps, want_next):
    r = torch.repeat_interleave(torch.arange(n, device="cuda"), d["ptr"].diff())
    c, v, X, V = d["col"].to(torch.int64), _u64(d["val"])[:, None], _u64(d["X"]), _u64(d["Y"])
    S = torch.empty(steps, X.shape[1], X.shape[1], dtype=torch.int64, device="cuda")
    for i in range(steps):
        S[i] = _xt_v(X, V, m) if m > 65536 else (X.double().T @ V.double()).to(torch.int64) % m
        if want_next or i + 1 < steps:
            V = torch.zeros_like(V).index_add_(0, r, _mulmod(v, V[c], m)) % m
    return (S, V) if want_next else S


def _poly_product(A, B, m):
    """A(x) B(x) mod m: float64 transforms of 11-bit limbs (exact after rounding)."""
    n = 1 << (A.shape[0] + B.shape[0] - 2).bit_length()
    limbs = -(-(m - 1).bit_length() // 11)
    fa, fb = ([torch.fft.rfft(((_u64(M) >> 11 * i) & 2047).double(), n, dim=0) for i in range(limbs)] for M in (A, B))
    out = 0
    for w in range(2 * limbs - 1):
        f = sum(fa[i] @ fb[w - i] for i in range(limbs) if 0 <= w - i < limbs)
        c = torch.fft.irfft(f, n, dim=0)[:A.shape[0] + B.shape[0] - 1].round().to(torch.int64) % m
        out = (out + _mulmod(c, torch.tensor(2**(11 * w) % m, device="cuda"), m)) % m
    return out


def _gf2_product(d, case):
    n_out = case["cols"] if case["transpose"] else case["rows"]
    r = torch.repeat_interleave(torch.arange(case["rows"], device="cuda"), d["ptr"].diff())
    c = d["col"].to(torch.int64)
    src, dst = (r, c) if case["transpose"] else (c, r)
    y = torch.zeros(n_out, case["words"], dtype=torch.int64, device="cuda")
    for w in range(case["words"]):
        for b in range(64):
            t = torch.zeros(n_out, dtype=torch.int32, device="cuda")
            t.index_add_(0, dst, ((d["x"][:, w] >> b) & 1).to(torch.int32)[src])
            y[:, w] |= (t & 1).to(torch.int64) << b
    return y


def exact(case, seed):
    k = case["kind"]
    if k == "sigma":
        return None  # a sigma-basis has no short statement in plain 64-bit arithmetic
    d = _inputs(case, seed)
    if k in ("product", "block"):
        m, out = case["m"], []
        for on, a, b in (("A", "x", "x2"), ("AT", "w", "w2")):
            if case["what"] in (on, "both"):
                t = on == "AT"
                n_out = case["cols"] if t else case["rows"]
                y = _spmm(d["ptr"], d["col"], d["val"], d[a], n_out, m, t)
                if case["axpby"]:
                    y = (_mulmod(_spmm(d["ptr"], d["col"], d["val"], d[b], n_out, m, t),
                                 torch.tensor(ALPHA % m, device="cuda"), m) + y * (BETA % m)) % m
                out.append(_bits32(y))
        return out
    if k == "gf2":
        return _gf2_product(d, case)
    if k == "sequence":
        return tuple(_bits32(t) for t in _sequence(d, case["rows"], case["m"], case["steps"], True))
    if k == "rank":
        S = _sequence(d, case["rows"], case["m"], _rank_steps(case), False)
        return [_bits32(S), None, None, None, None, None]
    if k == "batch":
        return [_bits32(_spmm(ptr, col, val, x, n, p, False)) for n, p, s, ptr, col, val, x in d["problems"]]
    return _bits32(_poly_product(d["A"], d["B"], case["m"]))
