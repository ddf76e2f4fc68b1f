"""MVS kernels at the edges of their splits, against the oracle, exactly: plane counts on both sides of each
number of planes per lane (with and without one access for a lane's planes) on images narrower than a tile,
and the depth range's order statistics over equal, clustered, few and many depths."""
import numpy as np
import pytest

from oracle import mvs as M
from paper_2601_17354_gb300 import synthetic as S
from tests.test_gpu_mvs import _check_view, _cuda

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [31, 32, 33, 63, 65, 66, 96, 97, 126])
def test_planes_per_lane(D):
    from paper_2601_17354_gb300 import mvs
    w, h = [(33, 17), (45, 70), (130, 9)][D % 3]
    sc = S.mvs_scene(D, n_cameras=12, width=w, height=h, focal=0.8 * w, n_sparse=1500, views=[4, 5, 6])
    _check_view(mvs, sc, 5, D)


DEPTHS = {
    "one": lambda r: [1.25],
    "two": lambda r: [3.0, 2.0],
    "equal": lambda r: np.full(5000, 2.5),
    "list": lambda r: r.uniform(1, 9, 256),
    "list + 1": lambda r: r.uniform(1, 9, 257),
    "many": lambda r: np.exp(r.normal(size=100_000)) + 0.3,
    "cluster and outlier": lambda r: np.concatenate([1.0 + 1e-6 * r.random(7000), [1e6]]),
    "three equal groups": lambda r: np.repeat([1.0, 1.5, 40.0], 700),
    "neighbouring values": lambda r: 4.0 + np.spacing(np.float32(4.0)) * r.integers(0, 3, 3000),
    "tails in one bucket": lambda r: np.concatenate([1.0 + 1e-5 * r.random(1000), 3.0 + 1e-5 * r.random(1000),
                                                     r.uniform(1.2, 2.8, 100), [1e5]]),
}


@pytest.mark.parametrize("name", list(DEPTHS))
def test_depth_range_order_statistics(name):
    from paper_2601_17354_gb300 import mvs
    rng = np.random.default_rng(len(name))
    z = rng.permutation(np.asarray(DEPTHS[name](rng), np.float32))
    cam = S.Camera(64, 48, 50.0, 50.0, 32.0, 24.0, np.eye(4, dtype=np.float32)[:3])
    pts = np.zeros((z.size, 3), np.float32)
    pts[:, 2] = z
    mv = mvs.MultiViewStereo(64, 48, 32)
    assert mv.depth_range(cam, _cuda(pts)) == M.depth_range(pts, cam)
