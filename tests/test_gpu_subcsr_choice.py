"""Sampled matrices on both sides of the lines that choose how the sub-CSR is built: a row too
long for one CTA's sort, more long rows than are worth placing, and just under both.

The sketch samples every column (d = n), so a row's sampled entries are its stored ones.  One
projected-gradient step against the exact oracle, and the same bits from run to run.  Tolerance
(binary32, as in test_gpu_sparse_update.py): a row's sum is at most n rounded steps of 2^-24 in
32 interleaved chains, added in order; the product and the step 128 + 4 more, the terms at most ~8
times the result, norm-wise.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import method
from synthdata import initial_factors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


# rows, columns, number of long rows, their length
@pytest.mark.parametrize("m, n, count, length", [
    (3000, 9000, 1, 4000), (3000, 9000, 1, 9000), (30000, 700, 1200, 66), (30000, 700, 2500, 66),
])
def test_half_step(pkg, m, n, count, length):
    k = 40
    g = np.random.default_rng(count + length)
    ln = g.integers(0, 3, m)
    ln[g.permutation(m)[:count]] = length
    col = np.concatenate([np.sort(g.choice(n, l, replace=False)) for l in ln]).astype(np.int32)
    rp = np.concatenate([[0], np.cumsum(ln)]).astype(np.int64)
    val = (g.random(col.size) + 0.1).astype(np.float32)
    M = sp.csr_matrix((val.astype(np.float64), col, rp), shape=(m, n))
    U, V = initial_factors(m, n, k, 8)
    got = []
    for rep in range(2):
        h = pkg.DSANLS(m, n, k, n, pkg.SUBSAMPLE, seed=5, d_v=64, t=3)
        h.set_csr(rp, col, val)
        h.set_factors(U, V)
        h.half_step(0)
        got.append(h.factors()[0])
        h.close()
    assert np.array_equal(got[0], got[1])
    S = method.Sketch(method.SUBSAMPLE, 5, 3, 0, n, n)
    want = method.half_step(M, V.astype(np.float64), U.astype(np.float64), S, method.PGD, method.mu_t(1.0, 1.0, 3))
    bound = (length / 32 + 32 + 132) * 2.0 ** -24 * 8
    diff = got[0].astype(np.float64) - want
    assert np.linalg.norm(diff) <= bound * np.linalg.norm(want)
    assert np.all(np.linalg.norm(diff, axis=1) <= 100 * bound * np.linalg.norm(want, axis=1) + bound * np.abs(want).max())
