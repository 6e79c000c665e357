"""Batches of the float64 eigensolver: one with more merges on a level than a
grid's y and z dimensions count (65535: two for each 33 x 33 matrix), and what
the results hold on to.

Tolerances as in test_gpu_eigh.py: 30 n eps ||A||, and 30 n eps from
orthonormal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_many_small_matrices():
    import paper_2503_20700_gb300 as pkg
    pkg.load()
    n, count = 33, 33000
    x = np.random.default_rng(8).standard_normal((60, n, n))
    base = x + x.transpose(0, 2, 1)
    res = pkg.ops.eigh_batched([base[i % 60] for i in range(count)])
    w, V = np.array([r[0] for r in res[:60]]), np.array([r[1] for r in res[:60]])
    norm = np.abs(w).max(axis=1)
    bound = 30 * n * np.finfo(float).eps
    assert np.all(np.abs(w - np.linalg.eigvalsh(base)[:, ::-1]).max(axis=1) <= bound * norm)
    assert np.all(np.abs(V @ base - w[:, :, None] * V).max(axis=(1, 2)) <= bound * norm)
    assert np.abs(V @ V.transpose(0, 2, 1) - np.eye(n)).max() <= bound
    # the same numbers wherever a matrix stands in the batch
    for i in range(60, count):
        assert np.array_equal(res[i][0], w[i % 60]) and np.array_equal(res[i][1], V[i % 60])


def test_results_are_arrays_of_their_own():
    import paper_2503_20700_gb300 as pkg
    pkg.load()
    for n in (5, 70):
        for w, V in pkg.ops.eigh_batched([np.eye(n), 2.0 * np.eye(n)]):
            assert w.base is None and V.base is None and V.flags.c_contiguous and V.flags.writeable
