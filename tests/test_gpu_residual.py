"""The dense relative error on tensor cores (csrc/error_tc.cu) against FP64 at the
sizes where its tiles end, at ranks on both sides of one 64-wide block, and for
values whose squared residuals leave binary32's range (then the FP64 form
answers).

Tolerance 1e-6 relative plus 1e-6 absolute: each residual carries the binary32
error of an inner product of at most 128 nonnegative terms (a few 2^-24 of the
entry), the squares are summed to 2^-48.
"""
import numpy as np
import pytest

from oracle import method
from synthdata import initial_factors, planted_dense

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


@pytest.mark.parametrize("m, n, k", [
    (1, 32, 1), (127, 33, 16), (128, 64, 64), (129, 65, 65), (300, 997, 10), (1000, 31, 20), (2051, 1025, 128),
    (5000, 4099, 33), (9000, 130, 100),
])
def test_error_matches_fp64(pkg, m, n, k):
    M, U0, V0 = planted_dense(m, n, min(k, 16), 3)
    U, V = initial_factors(m, n, k, 4)
    h = pkg.DSANLS(m, n, k, max(1, n // 4), pkg.GAUSSIAN, seed=0, d_v=max(1, m // 4))
    h.set_dense(M)
    near = np.zeros((m, k), np.float32), np.zeros((n, k), np.float32)
    kk = min(k, 16)
    near[0][:, :kk], near[1][:, :kk] = U0[:, :kk], V0[:, :kk]
    for A, B in ((U, V), near):  # random factors, and the planted ones: a small residual
        h.set_factors(A, B)
        want = method.rel_error(M.astype(np.float64), A.astype(np.float64), B.astype(np.float64))
        assert abs(h.rel_error() - want) <= 1e-6 * want + 1e-6
    h.close()


@pytest.mark.parametrize("scale", [1e-30, 1e-22, 1e25])
def test_error_of_badly_scaled_data(pkg, scale):
    m, n, k = 200, 150, 8
    M, _, _ = planted_dense(m, n, k, 5)
    M = (M.astype(np.float64) * scale).astype(np.float32)
    U, V = initial_factors(m, n, k, 6)
    h = pkg.DSANLS(m, n, k, 40, pkg.GAUSSIAN, seed=0)
    h.set_dense(M)
    h.set_factors(U, V)
    want = method.rel_error(M.astype(np.float64), U.astype(np.float64), V.astype(np.float64))
    assert abs(h.rel_error() - want) <= 1e-6 * want + 1e-6
    h.close()
