"""Exchange matrices of many Cholesky vectors, whose gathered copies are taken
piece by piece: the numbers against numpy, and the device memory of a call."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class _Pool:
    """High-water mark of the device's default memory pool."""
    HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH

    def __init__(self):
        self.cu, self.pool = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
        assert self.cu.cuInit(0) == 0
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def reset(self):
        assert self.cu.cuMemPoolSetAttribute(self.pool, self.HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0

    def high(self):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, self.HIGH, ctypes.byref(v)) == 0
        return v.value


def _inputs(nb, rank, na):
    rng = np.random.default_rng([nb, rank, na])
    h = rng.standard_normal((nb, nb))
    L = rng.standard_normal((rank, nb, nb), dtype=np.float32).astype(np.float64) / np.sqrt(rank)
    g = rng.standard_normal((na, na))
    G = rng.standard_normal((na, na, na, na), dtype=np.float32).astype(np.float64)
    G = G + G.transpose(1, 0, 3, 2)
    return h + h.T, L + L.transpose(0, 2, 1), g + g.T, G + G.transpose(3, 2, 1, 0)


def _fock(h, L, nc, na, gamma, Gamma):
    nb, a = len(h), slice(nc, nc + na)

    def exchange(X):  # sum_k X^k X^k^T of rank x nb x n
        Y = np.ascontiguousarray(X.transpose(1, 0, 2)).reshape(nb, -1)
        return Y, Y @ Y.T

    FI = h + 2.0 * np.tensordot(np.einsum("kii->k", L[:, :nc, :nc]), L, 1) - exchange(L[:, :, :nc])[1]
    Y, _ = exchange(L[:, :, a])
    M = (Y.reshape(nb, -1, na) @ gamma).reshape(nb, -1)
    La = L[:, a, a].reshape(len(L), -1)
    FA = np.tensordot(La @ gamma.ravel(), L, 1) - 0.5 * M @ Y.T
    W = (La @ Gamma.transpose(1, 2, 0, 3).reshape(na * na, -1)).reshape(-1, na, na)
    F = np.zeros_like(h)
    F[:nc] = 2.0 * (FI + FA).T[:nc]
    F[a] = gamma @ FI[:, a].T + np.ascontiguousarray(W.transpose(1, 0, 2)).reshape(na, -1) @ Y.T
    return F


@pytest.mark.parametrize("nb,rank,nc,na", [(240, 3000, 110, 4), (200, 1500, 20, 60)], ids=["core", "active"])
def test_exchange_by_pieces(nb, rank, nc, na):
    """The gathered columns (633 and 144 MB) exceed a piece.  Each output is a
    sum of rank x (nc or na) products of rounding 2^-53 of their size."""
    import paper_2503_20700_gb300 as pkg
    pkg.load()
    h, L, gamma, Gamma = _inputs(nb, rank, na)
    pool = _Pool()
    pool.reset()
    grad, F = pkg.ops.orbital_gradient(h, L, nc, na, gamma, Gamma, with_fock=True)
    high = pool.high()
    ref = _fock(h, L, nc, na, gamma, Gamma)
    assert np.abs(F - ref).max() < 1e-12 * np.abs(ref).max()
    # the vectors, W and La, a few pieces with their digits, and Gamma twice
    assert high < L.nbytes + 2 * 8 * rank * na * na + 2 * Gamma.nbytes + (1 << 30)
