"""The split copies of M and M^T that the FP32 products of the paper's order read (12 bytes per entry
of M) are given back when the order or the solver changes to one that
reads none, come back when it changes again, and the steps are the oracle's throughout (1e-5
norm-wise, the FP32 form's tolerance per step).
"""
import numpy as np
import pytest

from oracle import method
from synthdata import initial_factors, planted_dense

pytestmark = pytest.mark.gpu


def test_copies_follow_the_order():
    import torch
    import paper_2009_02845_gb300 as pkg
    torch.cuda.init()
    m, n, k, d = 2048, 1600, 16, 64
    M, _, _ = planted_dense(m, n, k, 1)
    U, V = initial_factors(m, n, k, 2)
    h = pkg.DSANLS(m, n, k, d, pkg.GAUSSIAN, seed=4, d_v=64, t=1)
    h.set_dense(M)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def step(reassociate):
        h.set_factors(U, V)
        h.half_step(0)
        got = h.factors()[0]
        S = method.Sketch(method.GAUSSIAN, 4, 1, 0, n, d)
        want = method.half_step(M.astype(np.float64), V.astype(np.float64), U.astype(np.float64), S, method.PGD,
                                method.mu_t(1.0, 1.0, 1), reassociate=reassociate)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)

    step(False)
    with_copies = free()
    h.set_options(order=pkg.ORDER_REASSOCIATED)
    step(True)
    assert free() - with_copies >= 8 * m * n  # 12 bytes per entry, less the form's own workspaces
    h.set_options(order=pkg.ORDER_PAPER)
    step(False)
    assert abs(free() - with_copies) <= 2 * m * n
    h.close()
