"""Rows of every length class of the sampled matrix, and the row update's tile edges.

The sketch samples every column (d = n), so a row's sampled entries are its stored ones:
lengths 0, 1, 2, 15, 16, 17 (one thread / a warp), 32, 33, 64, 65 (a warp / a CTA) and
longer, in the placed and sorted form (few entries per row on average) and in the
radix-sorted form (many).  k crosses the chunks of 16 columns and the atoms of 64, odd k
takes the scalar accesses, and m leaves ragged last tiles and several tiles per CTA.

One projected-gradient step against the exact oracle.  Binary32: a row's sum runs over at
most 64 + 32 rounded steps or (a long row) 50 + 32, the product z G over k <= 128, the step
itself over 4, each 2^-24 of the terms' sizes; the terms are at most ~8 times the stored
result, norm-wise: 228 * 2^-24 * 8 = 1.1e-4.  bf16 factors: 2^-8 more for the stored result.
A misplaced entry moves its row by far more; every row is held to 100 times the bound (a
row of the result may be small beside its own terms).
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import method
from synthdata import initial_factors

pytestmark = pytest.mark.gpu

LENGTHS = (0, 1, 2, 15, 16, 17, 32, 33, 64, 65, 200)


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


def _matrix(m, n, seed, few):
    g = np.random.default_rng(seed)
    length = g.integers(0, 3, m) if few else g.integers(8, 20, m)
    at = g.permutation(m)[:3 * len(LENGTHS)]
    length[at] = np.tile(LENGTHS, 3)
    length[g.integers(m)] = n  # one full row: several radix tiles
    col = np.concatenate([np.sort(g.choice(n, l, replace=False)) for l in length]).astype(np.int32)
    rp = np.concatenate([[0], np.cumsum(length)]).astype(np.int64)
    val = (g.random(col.size) + 0.1).astype(np.float32)
    return rp, col, val, sp.csr_matrix((val.astype(np.float64), col, rp), shape=(m, n))


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("few", [True, False])
@pytest.mark.parametrize("m,n,k", [(60001, 2100, 33), (700, 1500, 48), (2500, 1100, 64), (130, 600, 66),
                                   (45000, 1300, 100), (900, 1111, 112), (40037, 900, 113), (3000, 1200, 128)])
def test_half_step_rows_of_every_length(pkg, m, n, k, few, bf16):
    rp, col, val, M = _matrix(m, n, k, few)
    U, V = initial_factors(m, n, k, 8)
    if bf16:
        U, V = method.round_bf16(U), method.round_bf16(V)
    bound = 228 * 2.0 ** -24 * 8 + (2.0 ** -8 if bf16 else 0.0)
    for side in (0, 1):
        got = []
        for rep in range(2):
            h = pkg.DSANLS(m, n, k, n, pkg.SUBSAMPLE, seed=5, d_v=m, precision=pkg.BF16 if bf16 else pkg.FP32, t=3)
            h.set_csr(rp, col, val)
            h.set_factors(U, V)
            h.half_step(side)
            got.append(h.factors()[side])
            h.close()
        assert np.array_equal(got[0], got[1]), "the order of a row's entries does not depend on the run"
        X, Y, Z, K, dd = (M, V, U, n, n) if side == 0 else (M.T.tocsr(), U, V, m, m)
        S = method.Sketch(method.SUBSAMPLE, 5, 3, side, K, dd)
        exact = method.half_step(X, Y.astype(np.float64), Z.astype(np.float64), S, method.PGD,
                                 method.mu_t(1.0, 1.0, 3))
        diff = got[0].astype(np.float64) - exact
        assert np.linalg.norm(diff) <= bound * np.linalg.norm(exact)
        rows = np.linalg.norm(diff, axis=1)
        assert np.all(rows <= 100 * bound * np.linalg.norm(exact, axis=1) + bound * np.abs(exact).max())
