"""Backward compositing of paired-pixel strips at the edges of its rounds: lists of one round less,
exactly and more than one of its eight-entry rounds and of a staged batch, on an image no tile edge
divides.  The gradients are those of the one-pixel strips, which sum without rounds or products.

Tolerance: both walks rebuild T from T_final by one approximate reciprocal per entry (relative error
2^-22, rounded differently in each), so after the longest list, 129 entries, T differs by at most
2 * 129 * 2^-22 = 6.2e-5; the sums over a tile's pixels add a few 2^-24.  1e-4 relative L2 per group."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def stack(k: int, seed: int):
    """k translucent Gaussians over one view, each reaching most of its pixels."""
    from paper_2601_17354_gb300 import synthetic as S
    rng = np.random.default_rng(seed)
    means = np.stack([rng.uniform(-0.3, 0.3, k), rng.uniform(-0.2, 0.2, k), np.linspace(0.0, 1.0, k)])
    g = S.random_params(rng, means, 1, -1.2, 0.3, -3.0, 0.5, 0.05)
    cam = S.Camera(43, 25, 60.0, 60.0, 21.5, 12.5, np.eye(3, 4, dtype=np.float32) + np.float32([[0] * 4] * 2 + [[0, 0, 0, 3]]))
    return g, cam, S.random_image(seed + 1, 43, 25)


@pytest.mark.parametrize("tile,strip", [(8, 2), (16, 2), (16, 4)])
@pytest.mark.parametrize("k", [1, 2, 7, 8, 9, 15, 16, 17, 63, 64, 65, 129])
def test_rounds(tile, strip, k):
    from paper_2601_17354_gb300 import rasterizer as R
    g, cam, up = stack(k, 7 * k + tile)
    params, dl = R.GaussianBuffer.from_arrays(g), torch.from_numpy(up).cuda()
    got = {}
    for pix in (1, strip):
        rast = R.Rasterizer(tile=tile)
        rast.set_variant(pix, 64)
        rast.render(params, cam)
        grads = params.zeros_like()
        rast.backward(dl, grads)
        rast.check_status()
        got[pix] = grads
    for name in R.GROUPS:
        a, b = (getattr(got[p], name).double() for p in (strip, 1))
        assert float((a - b).norm()) <= 1e-4 * float(b.norm()), name
