"""A network for many subproblems at once holds no more than its buffers need: the Gram layer's
partial sums are those of its plan (at most 10 MB), not a slice per 64 columns for every group.

k = 32, 256 hidden, 19,456 groups: the normalised Grams take 80 MB, the two layers' sums per group 40,
the rest (1,024 rows, weights) under 20; with 30 MB for the allocator's rounding.
"""
import numpy as np
import pytest

from oracle import method
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


def test_memory_and_prediction_of_many_groups():
    import torch
    import paper_2009_02845_gb300 as pkg
    k, h, groups = 32, 256, 19456
    torch.cuda.init()
    pkg.MLP(k, h, max_rows=8, max_groups=1).close()  # primes the device outside the measurement
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net = pkg.MLP(k, h, max_rows=1024, max_groups=groups, seed=3)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 170 << 20
    # batches of few groups (K split) and of as many as there are rows
    P = omlp.unflatten(method.round_bf16(net.params()), k, h)
    g = np.random.default_rng(1)
    for n in (1, 130, 1024):
        B = g.random((n, k, 40))
        G, mu = np.einsum("gik,gjk->gij", B, B).astype(np.float32), g.uniform(0.1, 1.0, n).astype(np.float32)
        b = (g.random((1024, k)) * 3.0).astype(np.float32)
        off = np.linspace(0, 1024, n + 1).astype(np.int64)
        got = net.predict(*(torch.tensor(x).cuda() for x in (G, mu, off, b))).cpu().numpy()
        for i in (0, n // 2, n - 1):
            rows = slice(off[i], off[i + 1])
            Gn, bn, s, beta = omlp.normalise(G[i].astype(np.float64), float(mu[i]), b[rows].astype(np.float64))
            y, _ = omlp.forward(P, Gn, bn)
            want = y * (beta / s)[:, None]
            assert np.linalg.norm(got[rows] - want) <= 1e-4 * max(np.linalg.norm(want), 1e-3)
    net.close()
