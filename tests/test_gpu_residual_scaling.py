"""The dense relative error of factors whose columns and rows differ in size: U D and V D^-1
give the same product for any diagonal D, rows of U and V may lie far apart, and a component
that is dead in one factor may be large in the other.  The answer has to be that of FP64
whatever the sizes of the factors' entries.

Tolerance 1e-6 of the error itself.  An inner product of at most 128 nonnegative binary32
terms in one chain is off by a few 2^-24 of its size with either sign; against residuals of
1e-3 and 5e-2 of it that adds (4 2^-24 / 1e-3)^2 / 2 = 3e-8 of the result at most.
"""
import numpy as np
import pytest

from oracle import method
from synthdata import initial_factors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


def _columns(c):
    def f(g, U, V):
        U[:, 0] *= c
        V[:, 0] /= c
        U[:, 1] /= c
        V[:, 1] *= c
    return f


def _dead(c):
    def f(g, U, V):
        U[:, 0] *= c
        V[:, 0] = 0.0
    return f


def _diagonal(lo, hi):
    def f(g, U, V):
        s = np.exp(g.uniform(np.log(lo), np.log(hi), U.shape[1])).astype(np.float32)
        U *= s
        V /= s
    return f


def _rows(lo, hi):
    def f(g, U, V):
        U *= np.exp(g.uniform(np.log(lo), np.log(hi), (U.shape[0], 1))).astype(np.float32)
        V *= np.exp(g.uniform(np.log(lo), np.log(hi), (V.shape[0], 1))).astype(np.float32)
    return f


def _both(g, U, V):
    _diagonal(1e-6, 1e6)(g, U, V)
    _rows(1e-6, 1e6)(g, U, V)


FORMS = {
    "even": lambda g, U, V: None,
    "columns 1e2": _columns(1e2), "columns 1e4": _columns(1e4), "columns 1e6": _columns(1e6),
    "columns 1e8": _columns(1e8),
    "dead component 1e6": _dead(1e6), "dead component 1e8": _dead(1e8),
    "diagonal": _diagonal(1e-6, 1e6), "rows": _rows(1e-6, 1e6), "rows and diagonal": _both,
}


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("m, n, k", [(600, 500, 8), (333, 1001, 64), (1300, 260, 100)])
def test_error_of_factors_of_any_scale(pkg, m, n, k, form):
    for noise in (1e-3, 5e-2):
        g = np.random.default_rng(m + k)
        U, V = initial_factors(m, n, k, 21)
        FORMS[form](g, U, V)
        X = U.astype(np.float64) @ V.T.astype(np.float64)
        M = (X * (1.0 + noise * g.standard_normal((m, n)))).astype(np.float32)
        h = pkg.DSANLS(m, n, k, max(1, n // 8), pkg.GAUSSIAN, seed=0)
        h.set_dense(M)
        h.set_factors(U, V)
        got = h.rel_error()
        h.close()
        want = method.rel_error(M.astype(np.float64), U.astype(np.float64), V.astype(np.float64))
        assert abs(got - want) <= 1e-6 * want, (noise, got, want)
