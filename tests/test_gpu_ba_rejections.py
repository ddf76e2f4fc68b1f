"""Solves whose candidates are rejected: a rejected candidate leaves the state and the linearization, the next one is
taken from both at ten times the damping, wherever the solve ends.

Two starts far from the solution reject their first candidates, one near it the last ones, when FP32 states no
longer get better.  The state after each trial is the one that a solve of that trial alone makes, bit for bit, of the state
before (as long as camera 1's fixed axis, which a solve chooses at its start, is the same).  Tolerances: costs of the
same state differ by the order of the cost's sum alone (1e-12); the reported cost against the oracle's at the returned
state, 1e-9 relative, as in test_gpu_ba."""
import numpy as np
import pytest

from oracle import ba as O
from tests.test_gpu_ba import DELTA, SIGMA, _dev, _setup

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ITERS, LAM0 = 14, 2.0 ** -27  # 10 to 10^10 times it are FP32 numbers


@pytest.mark.parametrize("C,n,seed,spread,first", [(9, 200, 33, 1.0, False), (4, 40, 35, 2.0, False),
                                                   (7, 130, 31, 0.6, True)])
def test_rejected_candidates(C, n, seed, spread, first):
    from paper_2601_17354_gb300 import ba as B
    p, obs, R, t, P = _setup(seed, C, n, True)
    P = (P + np.random.default_rng(5).normal(0, spread, P.shape)).astype(np.float32)
    ba = B.BundleAdjuster(C, n, len(obs[0]))

    def solved(iters):
        dev = _dev(R, t, P, obs)
        return (dev, *ba.solve(*dev, p.K, SIGMA, DELTA, iters=iters, lam0=LAM0))

    def cost(Rc, tc, Pc, behind):  # an observation behind its camera carries no weight in a state and rules out a candidate
        rho = O.cost_terms(Rc, tc, Pc, obs, p.K, SIGMA, DELTA)[3]
        z = np.einsum("mj,mj->m", Rc[obs[0], 2], Pc[obs[1]]) + tc[obs[0], 2]
        return np.where(z > 1e-6, rho, behind).sum()

    runs = [solved(k) for k in range(ITERS + 1)]
    costs = runs[-1][1]
    taken = np.diff(costs) < 0
    assert np.all(np.diff(costs) <= 0) and runs[-1][2] == taken.sum()
    assert 0 < taken.sum() < ITERS and taken[0] == first
    assert np.any(taken[:-1] & ~taken[1:]) if first else np.any(~taken[:-1] & taken[1:])
    lam, axis = LAM0, O.gauge_axis(R.astype(np.float64), t.astype(np.float64))
    for k, (dev, c, accepted) in enumerate(runs):  # among them the ones that end on a rejected candidate
        assert accepted == taken[:k].sum()
        assert np.allclose(c, costs[:k + 1], rtol=1e-12)
        state = [x.cpu().numpy().astype(np.float64) for x in dev[:3]]
        assert abs(cost(*state, 0.0) - c[-1]) <= 1e-9 * c[-1]
        if k == ITERS:
            break
        if O.gauge_axis(*state[:2]) == axis:  # a solve of one trial from here takes the same candidate
            one = [x.clone() for x in dev]
            c1, _ = ba.solve(*one, p.K, SIGMA, DELTA, iters=1, lam0=lam)
            assert np.allclose(c1, costs[k:k + 2], rtol=1e-12)
            assert all(torch.equal(a, b) for a, b in zip(one[:3], runs[k + 1][0][:3]))
        if not taken[k]:
            assert all(torch.equal(a, b) for a, b in zip(dev[:3], runs[k + 1][0][:3]))
        lam = lam / 10 if taken[k] else lam * 10
