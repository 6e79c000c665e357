"""Entry-by-entry precision of the float64 digit GEMM on operands with uneven
rows: which outputs the digits may give (csrc/gemm_digits.cuh) and how far off
an output can be.

Bound of an output of k products: 2 k 2^-53 sum |a b| from the digits (what they
drop is at most 2^-66 2^ea 2^eb a term, and a term of 2^-14 2^ea 2^eb is among
them), k 2^-53 sum |a b| from FMAs, and two roundings of the result and of C."""
from fractions import Fraction

import numpy as np
import pytest

from test_digit_gemm import _chain, _exact


def _digits(x):
    """Row exponents e (|x| < 2^e) and the nine balanced digits of
    F = round(x 2^(70-e)), as the split kernel forms them."""
    big = np.abs(x).max(axis=1)
    e = np.where(big > 0, np.frexp(big)[1], 0)
    F = np.array([[int(abs(Fraction(float(v))) * Fraction(2) ** (70 - int(ei)) + Fraction(1, 2)) * (1 if v >= 0 else -1)
                   for v in row] for row, ei in zip(x, e)], dtype=object)
    d = np.zeros((9,) + x.shape, dtype=object)
    for s in range(8, 0, -1):
        d[s] = (F + 128) % 256 - 128
        F = (F - d[s]) // 256
    d[0] = F
    return e, d


def _product(a, b):
    """op(A) op(B) by the kernel's arithmetic (a: m x k, b: n x k): the sums of
    d = 7 and d = 8 share an accumulator and are rounded together."""
    (ea, da), (eb, db) = _digits(a), _digits(b)
    v = np.zeros((len(a), len(b)))
    for i in range(len(a)):
        for j in range(len(b)):
            h = 0
            for k0 in range(0, a.shape[1], 256):
                s = [sum(int(x) * int(y) for p in range(d + 1)
                         for x, y in zip(da[p][i, k0:k0 + 256], db[d - p][j, k0:k0 + 256])) for d in range(9)]
                assert all(abs(x) < 2**25 for x in s)
                h += round(Fraction(s[7] * 256 + s[8], 256)) + sum(s[d] << 8 * (7 - d) for d in range(7))
            v[i, j] = np.ldexp(float(h), int(ea[i] + eb[j]) - 68)
    return v


def _from_digits(a, b):
    """The rule on rows x k operands: the outputs that the digits give."""
    def down(x):
        e = np.where(x != 0, np.frexp(np.abs(x))[1], -10**6)
        return e.max(axis=1, keepdims=True) - e
    da, db = down(a), down(b)
    hit = np.zeros((len(a), len(b)), bool)
    for u, v in ((5, 7), (7, 5), (2, 10), (10, 2)):
        hit |= ((da <= u).astype(int) @ (db <= v).T.astype(int)) > 0
    return hit | (((a != 0).astype(int) @ (b != 0).T.astype(int)) == 0)


def _decay(rng, m, k, rate):
    x = rng.standard_normal((m, k))
    return x * np.exp(-np.abs(np.arange(k) * m / k - np.arange(m)[:, None]) * rate)


def _corner(rng, m, k, tail):
    """Row and column maxima meet zeros; one term at the edge of the rule."""
    a, b = (rng.standard_normal((m, k)) * 2.0**-tail for _ in range(2))
    a[:, 0], b[:, 0], a[:, 1], b[:, 1] = 1.9, 0.0, 0.0, 1.9
    a[:, 2], b[:, 2] = 2.0**-5 * rng.uniform(1, 1.1, m), 2.0**-7 * rng.uniform(1, 1.1, m)
    return a, b


def _pairs(kind, rng, m, k):
    if kind == "decay":
        return _decay(rng, m, k, 3.0), _decay(rng, m, k, 3.0)
    if kind == "decay x identity":
        return _decay(rng, m, k, 4.0), np.eye(k)[rng.choice(k, m)]
    if kind == "spread":
        return tuple(rng.standard_normal((m, k)) * 10.0 ** (-6 * rng.random((m, k))) for _ in range(2))
    if kind == "corner":
        return _corner(rng, m, k, int(rng.integers(9, 30)))
    return tuple(rng.standard_normal((m, k)) * (rng.random((m, k)) < 0.1) for _ in range(2))  # sparse


@pytest.mark.parametrize("k", [3, 16, 40, 130])
@pytest.mark.parametrize("kind", ["decay", "decay x identity", "spread", "corner", "sparse"])
def test_rule_on_the_cpu(kind, k):
    """What the digits give is within the bound, and over the outputs no further
    off (2-norm of the errors in units of sum |a b|) than a multiply-add chain or
    half an ulp each."""
    rng = np.random.default_rng([k, len(kind)])
    d, c = [], []
    for _ in range(3):
        a, b = _pairs(kind, rng, 6, k)
        ok, p, q, ex = _from_digits(a, b), _product(a, b), _chain(a, b), _exact(a, b)
        size = np.abs(a) @ np.abs(b).T
        for i, j in zip(*np.nonzero(ok)):
            x = float(abs(Fraction(float(p[i, j])) - ex[i][j]))
            assert x <= (2 * k + 1) * 2.0**-53 * size[i, j]
            if size[i, j] > 0:
                d.append(x / size[i, j])
                c.append(max(float(abs(Fraction(float(q[i, j])) - ex[i][j])), 2.0**-54 * float(abs(ex[i][j])))
                         / size[i, j])
    assert not d or np.linalg.norm(d) <= np.linalg.norm(c)


@pytest.fixture(scope="module")
def pkg():
    import paper_2503_20700_gb300 as p
    p.load()
    return p


@pytest.mark.gpu
@pytest.mark.parametrize("segs", [1, 40])   # 40: partial tiles
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("m,n,k", [(128, 64, 130), (161, 97, 64), (96, 33, 200), (31, 129, 48)])
@pytest.mark.parametrize("kind", ["decay", "spread", "sparse"])
def test_entries_of_uneven_operands(pkg, kind, m, n, k, ta, tb, segs):
    rng = np.random.default_rng([m, n, k, segs, len(kind)])
    if kind == "decay":
        A, B = (np.stack([_decay(rng, r, k, 0.4) for _ in range(segs)]) for r in (m, n))
    else:
        A, B = (rng.standard_normal((segs, r, k)) for r in (m, n))
        if kind == "spread":
            A, B = (x * 10.0 ** (-12 * rng.random(x.shape)) for x in (A, B))
        else:
            A, B = (x * (rng.random(x.shape) < 0.05) for x in (A, B))
    B = B.transpose(0, 2, 1)
    st = [np.ascontiguousarray(x.transpose(0, 2, 1) if t else x) for x, t in ((A, ta), (B, tb))]
    C0 = rng.standard_normal((m, n + 1)) * 2.0**-40
    C = C0.copy()
    pkg.ops.grouped_gemm(st[0].ravel(), st[1].ravel(), C, [(0, m, n, n + 1, 0, segs)],
                         [(i * m * k, i * k * n, k, m if ta else k, k if tb else n, ta, tb, 0.75)
                          for i in range(segs)])
    assert np.array_equal(C[:, n:], C0[:, n:])
    rows = rng.choice(m, min(m, 16), replace=False)
    ref = 0.75 * sum(A[i, rows].astype(np.longdouble) @ B[i].astype(np.longdouble) for i in range(segs))
    size = 0.75 * sum(np.abs(A[i, rows]) @ np.abs(B[i]) for i in range(segs)) + np.abs(C0[rows, :n])
    assert np.all(np.abs(C[rows, :n] - (C0[rows, :n] + ref)) <= (2 * k + segs + 3) * 2.0**-53 * size)


@pytest.mark.gpu
def test_decaying_vectors_come_back(pkg):
    """Rows that decay over 200 columns times the identity, and Cholesky
    vectors rotated by it: every entry exactly."""
    rng = np.random.default_rng(7)
    nb, rank = 200, 30
    env = np.exp(-np.abs(np.arange(nb)[:, None] - np.arange(nb)) / 6.0)
    L = rng.standard_normal((rank, nb, nb)) * env
    L = L + L.transpose(0, 2, 1)
    h, L2 = pkg.ops.transform(np.eye(nb), L[0], L)
    assert np.array_equal(h, L[0]) and np.array_equal(L2, L)
    for ta, tb in ((0, 0), (1, 1)):
        C = np.zeros((rank, nb, nb))
        pkg.ops.grouped_gemm(L.ravel(), np.eye(nb).ravel(), C, [(i * nb * nb, nb, nb, nb, i, 1) for i in range(rank)],
                             [(i * nb * nb, 0, nb, nb, nb, ta, tb, 1.0) for i in range(rank)])
        assert np.array_equal(C, L)  # symmetric


@pytest.mark.gpu
def test_one_small_output_beside_large_ones(pkg):
    """[1, 1.23e-12] . [0, 1] among full rows."""
    m, n, k = 128, 64, 64
    rng = np.random.default_rng(9)
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    A[77], B[:, 21] = 0.0, 0.0
    A[77, :2], B[1, 21] = (1.0, 1.23e-12), 1.0  # 2^-39 of the row's maximum
    C = np.zeros((m, n))
    pkg.ops.grouped_gemm(A.ravel(), B.ravel(), C, [(0, m, n, n, 0, 1)], [(0, 0, k, k, n, 0, 0, 1.0)])
    assert C[77, 21] == 1.23e-12
