"""Features and seeding where two floats do not carry the decision: flat patches, whose smallest eigenvalue is far
below the covariance's rounding; 16 neighbours that coincide or lie close together beside the other 16.

Tolerances: a flat patch's shares of the eigenvalue sum are compared with the squared singular values of the
centred offsets in FP64 (these are known to about 1e-15 of the largest, so a share of 1e-13 to 1e-8): one
rounding to FP32 is 6e-8 of the value, 2e-7 allows three.  Quaternions, scales and the other features against the FP64
oracle with the 1e-5 used elsewhere."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _init(P):
    from paper_2601_17354_gb300 import initializer as I
    return I.Initializer().paper_init(torch.from_numpy(P).cuda(), sh_degree=0)


@pytest.mark.parametrize("thickness", [0.0, 1e-5, 1e-3])
@pytest.mark.parametrize("at", [0.0, 2.0])
def test_flat_patches(thickness, at):
    rng = np.random.default_rng(3)
    turn = np.linalg.qr(rng.normal(size=(3, 3)))[0]
    P = np.ascontiguousarray(turn @ (rng.uniform(-1, 1, (3, 3000)) * [[1], [1], [thickness]]) + at, np.float32)
    nb = oracle.knn(P, 32)
    x = P.T[nb].astype(np.float64)
    x -= x.mean(1, keepdims=True)
    w = np.linalg.svd(x, compute_uv=False)[:, ::-1] ** 2
    w /= w.sum(1, keepdims=True)
    got = _init(P).features.cpu().numpy()[:, :3]
    assert np.all(np.abs(got - w) <= 2e-7 * w), np.abs(got / w - 1).max(0)


@pytest.mark.parametrize("kind", ["coincident", "tight", "tight and flat"])
def test_close_neighbours_beside_far_ones(kind):
    """300 groups of 17 points among 3,000 spread ones: a group's 16 nearest are the group."""
    rng = np.random.default_rng(4)
    group = rng.normal(size=(3, 300 * 17)) * {"coincident": 0.0, "tight": 2e-7,
                                              "tight and flat": np.array([[5e-7], [5e-7], [2e-8]])}[kind]
    group += np.repeat(rng.uniform(-0.1, 0.1, (3, 300)), 17, axis=1)
    P = np.ascontiguousarray(np.concatenate([group, rng.uniform(-0.1, 0.1, (3, 3000))], axis=1), np.float32)
    nb = oracle.knn(P, 32)
    own = np.arange(300 * 17) // 17
    assert np.all(nb[:300 * 17, :16] // 17 == own[:, None])
    pi = _init(P)
    f, fq = oracle.features(P, nb)
    o, g = oracle.pca_init(P, nb), pi.paper.numpy()
    for k, pairs in ((16, [(g["quats"].T, o["quats"].T)]), (32, [(pi.features.cpu().numpy(), f), (pi.frame_q.cpu().numpy().T, fq.T)])):
        x = P.T[nb[:, :k]].astype(np.float64)
        w = np.linalg.svd(x - x.mean(1, keepdims=True), compute_uv=False)[:, ::-1] ** 2
        # neighbours on one line have no normal to compare; coincident ones have the definition's, the first axis
        ok = (w[:, 1] - w[:, 0] > 1e-9 * w[:, 2]) | (w[:, 2] == 0)
        assert ok[:300 * 17].mean() > 0.85
        for got, want in pairs:
            assert np.allclose(got[ok], want[ok], rtol=1e-5, atol=1e-5)
    assert np.allclose(g["log_scales"], o["log_scales"], rtol=1e-6, atol=1e-5)
