"""A prediction whose bounded waits run out (the test switch starves its products; nothing is in
flight) says so by itself: its output is NaN, the next call that reads or writes the parameters
reports DSANLS_ETIMEOUT once, and a training step in between is neither blamed nor changed.

Values are compared bit for bit with those of a network that never timed out.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ETIMEOUT = -6


@pytest.fixture(scope="module")
def pkg():
    import paper_2009_02845_gb300 as p
    return p


def test_prediction_reports_its_own_timeout(pkg):
    import torch
    k, h, rows, groups = 8, 64, 300, 3
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    Y = torch.rand((groups, 50, k), generator=g, device="cuda")
    G = torch.bmm(Y.transpose(1, 2), Y).contiguous()
    mu = torch.rand(groups, generator=g, device="cuda") + 0.5
    off = torch.tensor([0, 100, 101, rows], device="cuda")
    b = torch.rand((rows, k), generator=g, device="cuda")
    x = torch.rand((rows, k), generator=g, device="cuda")
    nets = [pkg.MLP(k, h, max_rows=512, max_groups=4, seed=2) for _ in range(2)]
    want = nets[1].predict(G, mu, off, b).cpu().numpy()
    pkg.debug_tc_wait(20_000_000, starve=True)
    try:
        got = nets[0].predict(G, mu, off, b).cpu().numpy()
        step = nets[0].train_step(G, mu, off, b, x, 1e-3, want_grad=True)
    finally:
        pkg.debug_tc_wait(0, starve=False)
    assert np.isnan(got).all()
    ref = nets[1].train_step(G, mu, off, b, x, 1e-3, want_grad=True)
    assert step[0] == ref[0] and np.array_equal(step[1], ref[1])
    with pytest.raises(pkg.DSANLSError) as e:
        nets[0].params()
    assert e.value.code == ETIMEOUT
    assert np.array_equal(nets[0].params(), nets[1].params())
    again = nets[0].predict(G, mu, off, b).cpu().numpy()
    assert np.isfinite(want).all() and np.array_equal(again, nets[1].predict(G, mu, off, b).cpu().numpy())
    nets[0].params()  # nothing left to report
    for n in nets:
        n.close()
