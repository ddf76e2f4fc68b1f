"""Neighbour lists, features and seeding where the grid search and the two-float arithmetic have their
edges: fewer points than neighbours, duplicates and exact ties, a line, flat and clustered sets, an outlier
that stretches the grid, strong anisotropy, and coordinates far from unit scale.

Tolerances: lists exact; features and seeding as the FP64 oracle rounds to FP32 (a relative half unit,
6e-8, of values up to 1 and of logarithms up to 100; 1e-5 absolute covers both, as elsewhere)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def points(kind: str, n: int) -> np.ndarray:
    rng = np.random.default_rng(n)
    u = rng.uniform(-1, 1, (3, n))
    p = {"uniform": u, "line": u * [[1], [0], [0]], "flat": u * [[1], [1], [1e-4]],
         "lattice": rng.integers(0, 6, (3, n)), "clusters": rng.integers(0, 3, (3, n)) + 1e-3 * u,
         "outlier": np.where(np.arange(n) == 0, 40.0, 1e-2 * u), "long": u * [[1e3], [1], [1e-2]],
         "far": u + 100.0, "small": 1e-6 * u, "large": 1e6 * u}[kind]
    return np.ascontiguousarray(p, np.float32)


@pytest.mark.parametrize("k", [3, 16, 32])
@pytest.mark.parametrize("kind,n", [("uniform", 1), ("uniform", 2), ("uniform", 33), ("uniform", 2049), ("line", 700),
                                    ("lattice", 1500), ("clusters", 1200), ("outlier", 900), ("long", 1300)])
def test_lists(kind, n, k):
    from paper_2601_17354_gb300 import initializer as I
    P = points(kind, n)
    nb = I.Initializer().knn(torch.from_numpy(P).cuda(), k).cpu().numpy()
    assert np.array_equal(nb, oracle.knn(P, k))


@pytest.mark.parametrize("kind", ["uniform", "flat", "clusters", "far", "small", "large"])
@pytest.mark.parametrize("n", [33, 65, 500])
def test_features(kind, n):
    from paper_2601_17354_gb300 import initializer as I
    P = points(kind, n)
    pi = I.Initializer().paper_init(torch.from_numpy(P).cuda(), sh_degree=0)
    nb = oracle.knn(P, 32)
    f, fq = oracle.features(P, nb)
    o, g = oracle.pca_init(P, nb), pi.paper.numpy()
    assert np.allclose(pi.features.cpu().numpy(), f, rtol=1e-5, atol=1e-5)
    assert np.allclose(pi.frame_q.cpu().numpy(), fq, atol=1e-5)
    assert np.allclose(g["log_scales"], o["log_scales"], rtol=1e-6, atol=1e-5)
    assert np.allclose(g["quats"], o["quats"], atol=1e-5)
