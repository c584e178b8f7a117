"""The bounded waits of the tensor-core kernels that serve the FP32 form, the row update and the
dense relative error, made to run out without a fault: the test switch shortens their limit to
20 ms and keeps the producer of each kernel's first operand from copying anything (nothing is in
flight).  The kernel gives its tensor memory back and returns, the next synchronising call
reports DSANLS_ETIMEOUT, and the same handle then computes what the oracle does.

Tolerance of the half-step: 1e-5 norm-wise, the FP32 form's per step; of the relative error
1e-6.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import method
from synthdata import initial_factors, planted_dense

pytestmark = pytest.mark.gpu

ETIMEOUT = -6


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


def _sparse(m, n):
    g = np.random.default_rng(7)
    M = sp.random(m, n, density=0.02, random_state=np.random.RandomState(3), format="csr", dtype=np.float32)
    M.data = (g.random(M.nnz) + 0.1).astype(np.float32)
    return M


# (sketch, rank, sparse): products by tile copies; gathered rows (copied by the splitting warps);
# the row update with R given; with the sampled rows' sums formed in it
FORMS = {"tile copies": ("GAUSSIAN", 16, False), "gathered rows": ("SUBSAMPLE", 16, False),
         "row update": ("IDENTITY", 48, True), "row update, sampled": ("SUBSAMPLE", 48, True)}


@pytest.mark.parametrize("form", FORMS)
def test_half_step_times_out_and_recovers(pkg, form):
    kind, k, sparse = FORMS[form]
    m, n, d = 515, 256, 64
    if kind == "IDENTITY":
        d = n
    h = pkg.DSANLS(m, n, k, d, getattr(pkg, kind), seed=3, d_v=m if kind == "IDENTITY" else 64, t=1)
    if sparse:
        M = _sparse(m, n)
        h.set_csr(M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data)
    else:
        M, _, _ = planted_dense(m, n, 16, 1)
        h.set_dense(M)
    U, V = initial_factors(m, n, k, 2)
    h.set_factors(U, V)
    pkg.debug_tc_wait(20_000_000, starve=True)
    try:
        h.half_step(0)
        with pytest.raises(pkg.DSANLSError) as e:
            h.sync()
        assert e.value.code == ETIMEOUT
    finally:
        pkg.debug_tc_wait(0, starve=False)
    h.set_factors(U, V)
    h.half_step(0)
    got, _ = h.factors()
    h.close()
    S = method.Sketch(getattr(method, kind), 3, 1, 0, n, d)
    want = method.half_step(M.astype(np.float64), V.astype(np.float64), U.astype(np.float64), S, method.PGD,
                            method.mu_t(1.0, 1.0, 1))
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("k", [16, 100])
def test_rel_error_times_out_and_recovers(pkg, k):
    m, n = 700, 300
    M, _, _ = planted_dense(m, n, 16, 1)
    U, V = initial_factors(m, n, k, 2)
    h = pkg.DSANLS(m, n, k, 64, pkg.GAUSSIAN, seed=0)
    h.set_dense(M)
    h.set_factors(U, V)
    pkg.debug_tc_wait(20_000_000, starve=True)
    try:
        with pytest.raises(pkg.DSANLSError) as e:
            h.rel_error()
        assert e.value.code == ETIMEOUT
    finally:
        pkg.debug_tc_wait(0, starve=False)
    want = method.rel_error(M.astype(np.float64), U.astype(np.float64), V.astype(np.float64))
    assert abs(h.rel_error() - want) <= 1e-6 * want
    h.close()
