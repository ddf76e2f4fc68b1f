"""D-SSIM at the edges of its 32 x 22 tiles, against the oracle with the tolerances of test_gpu_dssim.py."""
import pytest

from tests import test_gpu_dssim as D

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
R = D.R


@pytest.mark.parametrize("shape", [(1, 1), (21, 31), (22, 32), (23, 33), (24, 64), (43, 95), (66, 40)])
def test_tile_edges(R, shape):
    D.test_dssim_matches_oracle(R, shape, 0.2)
