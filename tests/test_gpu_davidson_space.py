"""Davidson solves in subspaces of more than 32 vectors (what the work space
holds at least), with other entry points' backends coming and going before."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2503_20700_gb300 as p
    p.load()
    return p


def _digit_product(pkg):
    """A product large enough for the digit GEMM, checked; its page-locked
    memory goes back to the pool."""
    a = np.random.default_rng(5).standard_normal((256, 256))
    C = np.zeros((256, 256))
    pkg.ops.grouped_gemm(a.ravel(), a.ravel(), C, [(0, 256, 256, 256, 0, 1)], [(0, 0, 256, 256, 256, 0, 0, 1.0)])
    assert np.abs(C - a @ a).max() < 1e-11


def test_solve_keeps_going_beyond_32_vectors(pkg):
    """A Hubbard chain with U = 50 t, whose low states lie close together next
    to the width of the spectrum: the solve needs some forty vectors, all kept
    (max_space), before nothing is left of a new one (the tolerance is out of
    reach)."""
    n = 12
    h, eri, ec = W.hubbard_chain(n, u=50.0)
    g = pkg.DMRG(h, eri=eri, n_elec=n, D=64, e_core=ec, max_iter=3, max_space=100)
    g.sweep(1)
    _digit_product(pkg)
    b = n // 2 - 1
    g.sweep_part(0, b - 1)
    r = g.bond_solve(b, 0, pkg.FP64, max_iter=90, tol=1e-300)
    assert r["calls"] > 36
    assert r["residual64"] < 1e-10
