"""Batched float64 eigensolver (dmrg_eigh_batched) at the sizes where its path
changes: Jacobi up to 32, blocks of at most 16 and their merges above, rows of
the trailing matrix in shared memory or not; spectra that deflate everywhere,
nowhere, or in long runs; scales far from one.

Tolerances: a backward stable solver is off by a small multiple of
n eps ||A||, taken as 30 n eps (eps = 2.2e-16), and its vectors by 30 n eps
from orthonormal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def pkg():
    import paper_2503_20700_gb300 as p
    p.load()
    return p


def _matrix(kind, n, rng):
    x = rng.standard_normal((n, n))
    if kind == "random":
        return x + x.T
    if kind == "rank":  # most of the spectrum at zero
        y = x[:, :max(1, n // 5)]
        return y @ y.T
    if kind == "diagonal":
        return np.diag(rng.integers(-2, 3, n).astype(float))
    if kind == "pairs":  # every eigenvalue twice, and an uncoupled middle
        h = x[:(n + 1) // 2, :(n + 1) // 2]
        return np.kron(np.eye(2), h + h.T)[:n, :n]
    if kind == "chain":
        return 2.0 * np.eye(n) - np.diag(np.ones(n - 1), 1) - np.diag(np.ones(n - 1), -1)
    if kind == "graded":
        q = np.linalg.qr(x)[0]
        m = (q * 10.0 ** np.linspace(0, -25, n)) @ q.T
        return m + m.T
    if kind == "ones":
        return np.ones((n, n))
    return np.zeros((n, n))


def _check(M, w, V):
    n = len(M)
    norm = np.abs(np.linalg.eigvalsh(M)).max()
    assert np.all(np.diff(w) <= 0)
    assert np.abs(w - np.linalg.eigvalsh(M)[::-1]).max() <= 30 * n * EPS * norm
    assert np.abs(V @ M - w[:, None] * V).max() <= 30 * n * EPS * norm
    assert np.abs(V @ V.T - np.eye(n)).max() <= 30 * n * EPS
    top = np.abs(V).max(axis=1)
    first = np.argmax(np.abs(V) >= top[:, None] - 1e-12, axis=1)
    assert np.all(V[np.arange(n), first] > 0)


@pytest.mark.parametrize("kind", ["random", "rank", "diagonal", "pairs", "chain", "graded", "ones", "zero"])
def test_eigh_sizes_and_spectra(pkg, kind):
    rng = np.random.default_rng(len(kind))
    mats = [_matrix(kind, n, rng) for n in (1, 2, 15, 16, 31, 32, 33, 34, 47, 64, 65, 113, 129, 260)]
    for M, (w, V) in zip(mats, pkg.ops.eigh_batched(mats)):
        _check(M, w, V)


@pytest.mark.parametrize("scale", [1e-250, 1e-100, 1e120])
def test_eigh_scales(pkg, scale):
    rng = np.random.default_rng(3)
    mats = [_matrix(kind, n, rng) for n in (20, 100) for kind in ("random", "rank", "chain")]
    for M, (w, V) in zip(mats, pkg.ops.eigh_batched([scale * M for M in mats])):
        _check(M, w / scale, V)


def test_eigh_rows_beyond_shared_memory(pkg):
    rng = np.random.default_rng(9)
    M = _matrix("random", 1600, rng)
    (w, V), = pkg.ops.eigh_batched([M])
    _check(M, w, V)


def test_eigh_non_finite_input_returns(pkg):
    """Values are meaningless then; the call ends, and the next one is right."""
    rng = np.random.default_rng(4)
    for bad in (np.nan, np.inf):
        mats = [_matrix("random", n, rng) for n in (20, 70)]
        for M in mats:
            M[3, 5] = M[5, 3] = bad
        res = pkg.ops.eigh_batched(mats)
        assert [len(w) for w, _ in res] == [20, 70]
    M = _matrix("random", 70, rng)
    (w, V), = pkg.ops.eigh_batched([M])
    _check(M, w, V)
