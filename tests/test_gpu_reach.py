"""The projection's and the binning's warp-collective reach tests where their numbering changes form: warps
whose lanes have no, one, few, many (rectangles of more than 32 tiles, within and beyond 2 x 2 super-tiles)
and more than 1,024 candidate tiles, thin and round.  Keys, values and ranges bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2601_17354_gb300 import synthetic as S
from tests.test_gpu_parity import R, check_keys, render_gpu  # noqa: F401  (R: a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CAM = S.Camera(637, 413, 500.0, 500.0, 318.5, 206.5, np.eye(4, dtype=np.float32)[:3])


def _scene(kind, seed):
    rng = np.random.default_rng(seed)
    n = 32 * 40 + 5
    z = rng.uniform(2.0, 6.0, n)
    means = np.stack([rng.uniform(-0.75, 0.75, n) * z, rng.uniform(-0.5, 0.5, n) * z, z]).astype(np.float32)
    g = S.random_params(rng, means, 0, -4.0, 0.6, 0.0, 1.0, 0.0)
    lane = np.arange(n) % 32
    if kind == "mixed":  # a candidate to a thousand of them, beside one another
        g.log_scales[:] = rng.uniform(-6.0, -1.5, (3, n))
    elif kind == "thin":  # long and thin: rectangles full of tiles that are not reached
        g.log_scales[:] = np.array([-1.6, -6.0, -6.0])[:, None] + rng.normal(0, 0.3, (3, n))
    elif kind == "one lane":  # the rest of each warp behind the camera
        g.means[2, lane != (np.arange(n) // 32) % 32] *= -1.0
        g.log_scales[:] = rng.uniform(-4.0, -1.0, (3, n))
    elif kind == "wide":  # some warps hold a rectangle of more than 1,024 tiles
        g.log_scales[:, :] = rng.uniform(-6.0, -3.0, (3, n))
        g.log_scales[:, lane == 7] = rng.uniform(-1.0, 0.3, (3, int((lane == 7).sum())))
    g.log_scales[:] = g.log_scales.astype(np.float32)
    return g


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("kind", ["mixed", "thin", "one lane", "wide"])
def test_lists(R, kind, tile):  # noqa: F811
    g = _scene(kind, tile + len(kind))
    rast, _, _, _, _, code, pairs = render_gpu(R, g, CAM, R.Rasterizer(tile=tile))
    assert code == 0 and pairs == check_keys(rast, g, CAM, tile)
