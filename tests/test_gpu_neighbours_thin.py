"""Neighbour lists of sets whose grid is one cell thick: a line along an axis (a single row of cells, wide boxes) and
planes, alone and with outliers that make most cells empty; lists exact, as elsewhere."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [3, 32])
@pytest.mark.parametrize("n", [40, 2500])
@pytest.mark.parametrize("axes", [(0,), (1,), (2,), (0, 1), (0, 2), (1, 2)])
@pytest.mark.parametrize("outliers", [0, 5])
def test_lists(axes, n, k, outliers):
    from paper_2601_17354_gb300 import initializer as I
    rng = np.random.default_rng(10 * n + k)
    P = np.zeros((3, n), np.float32)
    P[list(axes)] = rng.uniform(-1, 1, (len(axes), n))
    P[axes[0], :outliers] *= 50
    nb = I.Initializer().knn(torch.from_numpy(P).cuda(), k).cpu().numpy()
    assert np.array_equal(nb, oracle.knn(P, k))
