"""The FP32 products on tensor cores straight from binary32 operands
(csrc/gemm_split.cu), through one half-step of every form that takes them, at
the sizes where the kernel can go wrong: ranks around its 32-, 64- and
128-column tiles, rows around its 128-row tiles, reductions around its steps of
32 and blocks of 64 (and long enough to cycle every ring), and widths whose
rows are not 16-byte aligned.

Tolerance: 1e-5 norm-wise on the updated factor, the FP32 form's tolerance per
step: a product's error is at most a few 2^-24 of sum |a||b| (three-way splits,
dropped terms 2^-24, chains of at most 16 additions), and the projected step
does not expand it.
"""
import numpy as np
import pytest

from oracle import method
from synthdata import initial_factors, planted_dense

pytestmark = pytest.mark.gpu

# m, n, k, d, d_v
CASES = [
    (127, 31, 5, 9, 17),
    (128, 33, 32, 33, 64),
    (129, 65, 33, 64, 127),
    (257, 95, 64, 95, 128),
    (300, 260, 65, 97, 129),
    (385, 1030, 100, 700, 333),
    (1001, 515, 128, 129, 777),
]


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("form", ["gaussian", "reassociated", "subsample", "identity"])
@pytest.mark.parametrize("case", CASES)
def test_half_step(pkg, case, form):
    m, n, k, d, d_v = case
    M, _, _ = planted_dense(m, n, min(k, 16), 5)
    U, V = initial_factors(m, n, k, 6)
    M64 = M.astype(np.float64)
    kind = {"subsample": method.SUBSAMPLE, "identity": method.IDENTITY}.get(form, method.GAUSSIAN)
    if form == "identity":
        d, d_v = n, m
    for side, dd in ((0, d), (1, d_v)):
        h = pkg.DSANLS(m, n, k, d, kind, seed=9, d_v=d_v, t=2,
                       order=pkg.ORDER_REASSOCIATED if form == "reassociated" else pkg.ORDER_PAPER)
        h.set_dense(M)
        h.set_factors(U, V)
        h.half_step(side)
        got = h.factors()[side]
        h.close()
        X, Y, Z = (M64, V, U) if side == 0 else (M64.T, U, V)
        S = method.Sketch(kind, 9, 2, side, X.shape[1], dd)
        want = method.half_step(X, Y.astype(np.float64), Z.astype(np.float64), S, method.PGD, method.mu_t(1.0, 1.0, 2))
        assert _rel(got, want) <= 1e-5, (side, _rel(got, want))


def test_refilled_padded_matrix(pkg):
    """A width that is not a multiple of 4 keeps its zero columns over a refill, and the
    relative error sees only the matrix."""
    m, n, k = 130, 71, 12
    h = pkg.DSANLS(m, n, k, 40, pkg.SUBSAMPLE, seed=1, d_v=40)
    for seed in (1, 2):
        M, _, _ = planted_dense(m, n, k, seed)
        U, V = initial_factors(m, n, k, seed)
        h.set_dense(M)
        h.set_factors(U, V)
        want = method.rel_error(M.astype(np.float64), U.astype(np.float64), V.astype(np.float64))
        assert abs(h.rel_error() - want) <= 1e-6
    h.close()
