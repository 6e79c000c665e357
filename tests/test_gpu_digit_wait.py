"""The wait bound holds in the float64 digit GEMM too: with a bound of 0 its
first wait that is not over gives up (the kernel stops its other roles, waits
for its own copies and products, frees its tensor memory and returns), the
call says DMRG_ETIMEOUT, and with the bound restored the same call is right."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2503_20700_gb300 as p
    p.load()
    return p


def _grouped(pkg, m, n, k, segs):
    rng = np.random.default_rng([m, n, k])
    A, B = rng.standard_normal((segs, m, k)), rng.standard_normal((segs, k, n))
    C = np.zeros((m, n))
    pkg.ops.grouped_gemm(A.ravel(), B.ravel(), C, [(0, m, n, n, 0, segs)],
                         [(i * m * k, i * k * n, k, k, n, 0, 0, 1.0) for i in range(segs)])
    assert np.abs(C - np.einsum("sik,skj->ij", A, B)).max() < 1e-10


def _transform(pkg):
    rng = np.random.default_rng(3)
    nb, rank = 96, 40
    R = np.linalg.qr(rng.standard_normal((nb, nb)))[0]
    h, L = rng.standard_normal((nb, nb)), rng.standard_normal((rank, nb, nb))
    h2, L2 = pkg.ops.transform(R, h, L)
    assert np.abs(h2 - R.T @ h @ R).max() < 1e-11 and np.abs(L2 - R.T @ L @ R).max() < 1e-11


@pytest.mark.parametrize("call", [
    lambda p: _grouped(p, 256, 256, 256, 1),      # one chunk a tile
    lambda p: _grouped(p, 200, 130, 1000, 1),     # chunks, three stages refilled
    lambda p: _grouped(p, 150, 70, 90, 61),       # partial tiles and their reduction
    _transform], ids=["square", "chunks", "segments", "transform"])
def test_zero_wait_bound_times_out(pkg, call):
    try:
        pkg.set_kernel_wait_timeout(0.0)
        with pytest.raises(pkg.DmrgError) as ei:
            call(pkg)
        assert ei.value.status == pkg.DMRG_ETIMEOUT
    finally:
        pkg.set_kernel_wait_timeout(2.0)
    call(pkg)
