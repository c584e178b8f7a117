"""A sketch of more columns than a grid's second dimension holds in tiles of 32 (2,097,120), in the
FP32 form: the second operand of A = M S is split in more rows than that.

Tolerance: 1e-5 norm-wise on the updated factor, the FP32 form's per step.
"""
import numpy as np
import pytest

from oracle import method
from synthdata import initial_factors, planted_dense

pytestmark = pytest.mark.gpu


def test_half_step_with_a_very_wide_sketch():
    import paper_2009_02845_gb300 as pkg
    m, n, k, d = 20, 12, 2, 65535 * 32 + 70
    M, _, _ = planted_dense(m, n, 2, 5)
    U, V = initial_factors(m, n, k, 6)
    h = pkg.DSANLS(m, n, k, d, pkg.RADEMACHER, seed=9, d_v=64, t=2)
    h.set_dense(M)
    h.set_factors(U, V)
    h.half_step(0)
    got, _ = h.factors()
    h.close()
    S = method.Sketch(method.RADEMACHER, 9, 2, 0, n, d)
    want = method.half_step(M.astype(np.float64), V.astype(np.float64), U.astype(np.float64), S, method.PGD,
                            method.mu_t(1.0, 1.0, 2))
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
