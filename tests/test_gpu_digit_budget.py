"""The work space of the float64 digit GEMM counts against a context's memory
budget, and a product that it has no room for runs without it."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_integral_product_under_a_budget():
    """dmrg_init forms the integrals from 6000 Cholesky vectors of 24 x 24: 30
    MB of operands and result, 62 MB of digits (18 B per element)."""
    import paper_2503_20700_gb300 as pkg
    pkg.load()
    n, rank = 24, 6000
    h, L = W.cholesky_random(n, rank, seed=2)
    occ, path = W.aufbau_state(h, n, 0)
    held = 8 * (rank * n * n + n**4)
    digits = 18 * rank * n * n

    def energy(**kw):
        g = pkg.DMRG(h, chol=L, n_elec=n, D=16, max_iter=4, occ=occ, two_s_right=path, **kw)
        peak = g.memory()[1]
        e, _ = g.sweep(1)
        g.close()
        return e, peak

    e, peak = energy()
    assert peak >= held + digits
    for budget in (held + 3 * digits // 2, held + digits // 2):
        eb, pb = energy(hbm_budget_bytes=budget)
        assert pb <= budget and (pb >= held + digits) == (budget >= held + digits)
        assert abs(eb - e) < 1e-8
