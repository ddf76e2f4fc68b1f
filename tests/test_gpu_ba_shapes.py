"""Bundle adjustment at the edges of its kernels: two cameras, a point seen by more cameras than a point has
lanes, observation lists of several staging blocks, cameras beyond one mask word, the largest blocked solve
and the first packed one; and solves whose candidates are rejected, where the state left behind must be the one
whose cost is reported (the device decides and moves the state without the host).

Tolerances: the backward error bound of a step as derived in test_gpu_ba (2e-4); the reported cost against
the oracle's at the returned state, 1e-9 relative as there."""
import numpy as np
import pytest

from oracle import ba as O
from tests.test_gpu_ba import BACKWARD_TOL, DELTA, SIGMA, _backward_error, _dev, _setup

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,n,tracks", [(2, 9, False), (3, 2500, False), (12, 64, False), (33, 150, True),
                                        (37, 200, True), (38, 200, True)])
def test_step(C, n, tracks):
    from paper_2601_17354_gb300 import ba as B
    p, obs, R, t, P = _setup(100 + C, C, n, tracks)
    ba = B.BundleAdjuster(C, n, len(obs[0]))
    dcam, dP, cost = ba.step(*_dev(R, t, P, obs), p.K, SIGMA, DELTA, 1e-3)
    R64, t64, P64 = (x.astype(np.float64) for x in (R, t, P))
    want = O.cost_terms(R64, t64, P64, obs, p.K, SIGMA, DELTA)[3].sum()
    assert abs(cost - want) <= 1e-9 * want
    eta = _backward_error(R, t, P, obs, p.K, 1e-3, O.gauge_axis(R64, t64), dcam.cpu().numpy().astype(np.float64),
                          dP.cpu().numpy().astype(np.float64))
    assert eta <= BACKWARD_TOL, eta


@pytest.mark.parametrize("iters", [0, 1, 2, 9])
@pytest.mark.parametrize("spread", [0.01, 0.6])  # a start near the solution, and one whose first candidates fail
def test_state_matches_reported_cost(iters, spread):
    from paper_2601_17354_gb300 import ba as B
    p, obs, R, t, P = _setup(31, 7, 130, True)
    P = (P + np.random.default_rng(5).normal(0, spread, P.shape)).astype(np.float32)
    ba = B.BundleAdjuster(7, 130, len(obs[0]))
    dev = _dev(R, t, P, obs)
    costs, acc = ba.solve(*dev, p.K, SIGMA, DELTA, iters=iters, lam0=1e-8)
    assert len(costs) == iters + 1 and np.all(np.diff(costs) <= 0)
    assert acc == int((np.diff(costs) < 0).sum())
    got = [x.cpu().numpy().astype(np.float64) for x in dev[:3]]
    want = O.cost_terms(*got, obs, p.K, SIGMA, DELTA)[3].sum()
    assert abs(costs[-1] - want) <= 1e-9 * want
