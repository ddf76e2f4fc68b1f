"""Backgrounds and camera collections that can be gone through only once are taken as lists are."""
from types import SimpleNamespace

import numpy as np
import pytest

pytest.importorskip("torch")
from paper_2601_17354_gb300.rasterizer import camera_array, camera_struct  # noqa: E402


def _camera(k, bg):
    return SimpleNamespace(width=8 + k, height=6, fx=5.0, fy=5.5, cx=4.0, cy=3.0, viewmat=np.eye(4)[:3] + k, bg=bg)


class Stream:
    """A sized collection that makes its cameras as it is gone through."""

    def __init__(self, n, bg):
        self.n, self.bg, self.passes = n, bg, 0

    def __len__(self):
        return self.n

    def __iter__(self):
        self.passes += 1
        return (_camera(k, self.bg(k)) for k in range(self.n))


@pytest.mark.parametrize("values", [3, 2])
def test_iterated_once(values):
    bg = lambda k: (0.1 * k + 0.2 * v for v in range(values))
    want = b"".join(bytes(camera_struct(c)) for c in Stream(5, bg))
    assert b"".join(bytes(camera_struct(_camera(k, list(bg(k))))) for k in range(5)) == want
    cams = Stream(5, bg)
    assert bytes(camera_array(cams)) == want and cams.passes == 1
