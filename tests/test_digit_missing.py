"""Products that the float64 digit GEMM leaves to float64 FMAs: segments with a
graded or non-finite operand, alone and among others of the same output, at the
edges of the 32 x 32 blocks and 64-wide k-steps of the kernel that adds them.

Tolerance: a multiply-add chain of k products and the addition to C are off by
(k + 2) 2^-53 of sum |a b| + |C|; the digit products by less."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2503_20700_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("segs", [1, 3, 61])   # 61: partial tiles
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("m,n,k", [(128, 64, 64), (129, 65, 63), (33, 161, 65), (200, 31, 130), (97, 96, 200)])
def test_graded_segments(pkg, m, n, k, ta, tb, segs):
    rng = np.random.default_rng([m, n, k, segs])
    A, B = rng.standard_normal((segs, m, k)), rng.standard_normal((segs, k, n))
    g = 10.0 ** np.linspace(-40, 40, k)
    A[::2] *= g
    B[::2] /= g[:, None]
    C0 = rng.standard_normal((m, n + 2))
    C = C0.copy()
    st = [np.ascontiguousarray(x.transpose(0, 2, 1) if t else x) for x, t in ((A, ta), (B, tb))]
    pkg.ops.grouped_gemm(st[0].ravel(), st[1].ravel(), C, [(0, m, n, n + 2, 0, segs)],
                         [(i * m * k, i * k * n, k, m if ta else k, k if tb else n, ta, tb, -0.5)
                          for i in range(segs)])
    assert np.array_equal(C[:, n:], C0[:, n:])
    rows = rng.choice(m, 6, replace=False)
    ref = -0.5 * sum(A[i, rows].astype(np.longdouble) @ B[i].astype(np.longdouble) for i in range(segs))
    size = 0.5 * sum(np.abs(A[i, rows]) @ np.abs(B[i]) for i in range(segs)) + np.abs(C0[rows, :n])
    assert np.all(np.abs(C[rows, :n] - (C0[rows, :n] + ref)) <= (k + segs + 2) * 2.0**-53 * size)
    dense = C0[:, :n] - 0.5 * np.einsum("sik,skj->ij", A, B)
    assert np.abs(C[:, :n] - dense).max() < 1e-9 * np.abs(dense).max()


def test_one_bad_segment_among_others(pkg):
    """A NaN of one segment reaches its row only, an infinity its column."""
    rng = np.random.default_rng(1)
    m, n, k, segs = 150, 70, 90, 5
    A, B = rng.standard_normal((segs, m, k)), rng.standard_normal((segs, k, n))
    A[1, 140, 3] = np.nan
    B[3, 7, 66] = np.inf
    C = np.zeros((m, n))
    pkg.ops.grouped_gemm(A.ravel(), B.ravel(), C, [(0, m, n, n, 0, segs)],
                         [(i * m * k, i * k * n, k, k, n, 0, 0, 1.0) for i in range(segs)])
    with np.errstate(invalid="ignore"):
        ref = np.einsum("sik,skj->ij", A, B)
    assert np.isnan(C[140]).all()
    ok = np.arange(m) != 140
    assert np.array_equal(C[ok, 66], np.sign(A[3, ok, 7]) * np.inf)
    assert np.abs(np.delete(C[ok], 66, 1) - np.delete(ref[ok], 66, 1)).max() < 1e-11
