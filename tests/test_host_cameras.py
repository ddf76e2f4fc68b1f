"""Cameras marshalled in bulk are byte for byte the cameras marshalled one by one, whatever the viewmat's type and
strides, and what the one refuses the other does."""
from types import SimpleNamespace

import numpy as np
import pytest

pytest.importorskip("torch")
from paper_2601_17354_gb300 import _lib as L  # noqa: E402
from paper_2601_17354_gb300 import synthetic as S  # noqa: E402
from paper_2601_17354_gb300.rasterizer import camera_array, camera_struct  # noqa: E402


def _cameras(n):
    rng = np.random.default_rng(n)
    out = []
    for k in range(n):
        vm = rng.normal(size=(3, 4))
        vm = [vm, vm.astype(np.float32), np.asfortranarray(vm.astype(np.float32)), vm.reshape(-1).tolist(),
              rng.normal(size=(3, 8)).astype(np.float32)[:, ::2]][k % 5]
        c = SimpleNamespace(width=np.int64(640 + k), height=480, fx=rng.uniform(100, 900), fy=np.float32(500.1), cx=320.3,
                            cy=240, viewmat=vm)
        if k % 3 == 0:
            c.near, c.bg = 0.1 * (k + 1), (0.1, np.float64(1 / 3), 1)
        out.append(c)
    return out


@pytest.mark.parametrize("n", [0, 1, 2, 64])
def test_same_bytes(n):
    cams = _cameras(n)
    want = (L.PgsCamera * n)(*[camera_struct(c) for c in cams])
    assert bytes(camera_array(cams)) == bytes(want)
    for c, w in zip(cams, want):
        assert np.array_equal(np.array(w.viewmat[:]), np.asarray(c.viewmat, np.float32).reshape(-1))


def test_extreme_values_and_odd_lengths():
    cam = S.Camera(2 ** 33 + 5, 480, 1e300, 500.0, float("nan"), -0.0, np.eye(4, dtype=np.float32)[:3], bg=[1e39, 0, 0])
    assert bytes(camera_array([cam, cam])) == bytes((L.PgsCamera * 2)(camera_struct(cam), camera_struct(cam)))
    short = S.Camera(4, 4, 1.0, 1.0, 2.0, 2.0, np.arange(9, dtype=np.float32))  # zeros after the values given
    assert bytes(camera_array([short])) == bytes(camera_struct(short))
    for bad in (np.eye(4, dtype=np.float32), np.zeros(13)):
        cam = S.Camera(4, 4, 1.0, 1.0, 2.0, 2.0, bad)
        for call in (camera_struct, lambda c: camera_array([c])):
            with pytest.raises((IndexError, ValueError)):
                call(cam)
