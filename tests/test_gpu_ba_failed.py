"""A solve that ends because the reduced system is not positive definite leaves the caller's costs after its last
decision alone, and the context solves the next problem.

Two cameras and one point give a reduced system of rank one: the damping 1e-30 is far below FP32's rounding, so
some of the four other pivots come out at or below zero on most problems."""
import ctypes as C

import numpy as np
import pytest

from paper_2601_17354_gb300 import _lib as L
from tests.test_gpu_ba import DELTA, SIGMA, _dev, _setup

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_costs_of_a_failed_solve():
    from paper_2601_17354_gb300 import ba as B
    failed = 0
    for seed in range(12):
        p, obs, R, t, P = _setup(200 + seed, 2, 1, False)
        if len(obs[0]) != 2:
            continue
        ba = B.BundleAdjuster(2, 1, 2)
        big = ba.solve(*_dev(R, t, P, obs), p.K, SIGMA, DELTA, iters=9, lam0=1e12)  # other costs in the context's buffer
        dev = _dev(R, t, P, obs)
        costs, accepted = np.full(10, -7.0), C.c_int32(-7)
        rc = ba._lib.pgs_ba_solve(ba._b, *(B._p(x) for x in dev), ba._K(p.K), SIGMA, DELTA, 9, 1e-30,
                                  costs.ctypes.data_as(C.POINTER(C.c_double)), C.byref(accepted))
        if rc == L.PGS_ERR_NOT_PD:
            failed += 1
            known = int((costs != -7.0).sum())
            assert 1 <= known < 10 and np.all(costs[known:] == -7.0) and np.all(np.diff(costs[:known]) <= 0)
            assert accepted.value == -7
        else:
            assert rc == 0 and np.all(costs != -7.0)
        again = ba.solve(*_dev(R, t, P, obs), p.K, SIGMA, DELTA, iters=9, lam0=1e12)
        assert abs(again[0][0] - big[0][0]) <= 1e-12 * abs(big[0][0])
    assert failed
