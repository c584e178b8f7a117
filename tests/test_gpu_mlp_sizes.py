"""The network's kernels at the sizes where their tiles end: widths around the
16- and 64-wide GEMM tiles and the 32-wide column sums, ranks around the
split products' padding, groups of uneven size (one of them a single row) whose
total crosses the 112-row tiles of the column sums and the 8-row tiles of the
activations.

Tolerances as in test_gpu_mlp.py: the passes use the weights rounded to bf16,
so the oracle with the same weights differs by binary32 arithmetic only:
outputs 1e-4, gradients 1e-3 norm-wise per parameter array.
"""
import numpy as np
import pytest

from oracle import method
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("k, h, sizes", [
    (1, 1, [1]),
    (5, 15, [7, 1, 3]),
    (8, 16, [111]),
    (17, 33, [112, 1]),
    (31, 64, [100, 13, 120, 1]),
    (32, 65, [449]),
    (32, 256, [300, 1, 600]),
])
def test_prediction_and_gradient(pkg, k, h, sizes):
    import torch
    net = pkg.MLP(k, h, max_rows=1024, max_groups=8, seed=11)
    P = omlp.unflatten(method.round_bf16(net.params()), k, h)
    g = np.random.default_rng(k * 1000 + h)
    Gs, mus, bs, xs, want, groups = [], [], [], [], [], []
    for n in sizes:
        B = g.random((k, 3 * k + 2))
        G, mu = (B @ B.T).astype(np.float32), np.float32(g.uniform(0.1, 1.0))
        b = (g.random((n, k)) * 3.0).astype(np.float32)
        x = np.maximum(g.standard_normal((n, k)), 0.0).astype(np.float32)
        Gn, bn, s, beta = omlp.normalise(G.astype(np.float64), float(mu), b.astype(np.float64))
        y, _ = omlp.forward(P, Gn, bn)
        want.append(y * (beta / s)[:, None])
        groups.append((Gn, bn, x.astype(np.float64) * s / beta[:, None]))
        Gs.append(G), mus.append(mu), bs.append(b), xs.append(x)
    off = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)).cuda()
    dev = [torch.tensor(np.stack(Gs)).cuda(), torch.tensor(np.array(mus, np.float32)).cuda(), off,
           torch.tensor(np.concatenate(bs)).cuda()]
    ref = np.concatenate(want)
    got = net.predict(*dev).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-4 * max(np.linalg.norm(ref), 1e-3)
    loss, grad = net.train_step(*dev, torch.tensor(np.concatenate(xs)).cuda(), 0.0, want_grad=True)
    loss_o, grads_o = omlp.loss_and_grads(P, groups)
    assert abs(loss - loss_o) <= 1e-4 * max(loss_o, 1e-12)
    flat = omlp.flatten(grads_o, k, h)
    at = 0
    for name, shape in omlp.param_shapes(k, h):
        n = int(np.prod(shape))
        o = flat[at:at + n]
        assert np.linalg.norm(grad[at:at + n] - o) <= 1e-3 * max(np.linalg.norm(o), 1e-9), name
        at += n
    net.close()
