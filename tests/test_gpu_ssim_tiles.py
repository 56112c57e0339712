"""The L1 + DSSIM loss at image sizes around its 32 x 54 pixel tiles, against
the FP64 oracle, and an infinite pixel, which reaches exactly the gradients
whose two filter windows hold it."""
import numpy as np
import pytest

from oracle import ssim
from paper_2501_18630_gb300 import scenes
from tests.test_gpu_ssim import _run, _views
import torch  # noqa: F401

pytestmark = pytest.mark.gpu


def _cam(w, h):
    return scenes.pinhole(*scenes.look_at((0, 0, -3)), w, h)


@pytest.mark.parametrize("w,h", [(1, 1), (5, 3), (31, 53), (32, 54), (33, 55), (37, 64), (64, 108), (65, 109), (10, 200)])
def test_sizes_around_the_tile(w, h):
    rng = np.random.default_rng(w * 1000 + h)
    cams = [_cam(w, h), _cam(h, w)]
    n = 6 * w * h
    target = rng.random(n)
    color = np.clip(target + rng.normal(0.0, 0.1, n), 0.0, 1.0)
    loss, d = _run(cams, color, target, 0.2)
    for v, (cx, ty, dv) in enumerate(zip(_views(cams, color), _views(cams, target), _views(cams, d))):
        # the tolerances of the other DSSIM tests (fp32 statistics, C2 = 9e-4)
        assert loss[v] == pytest.approx(ssim.loss(cx, ty, 0.2), rel=2e-5, abs=1e-7)
        ref = ssim.grad(cx, ty, 0.2)
        assert np.abs(dv - ref).max() <= 2e-4 * np.abs(ref).max()


@pytest.mark.parametrize("x,y", [(0, 0), (31, 53), (32, 54), (40, 60)])
def test_infinite_pixel_reaches_its_windows_only(x, y):
    w, h = 70, 116
    rng = np.random.default_rng(1)
    color, target = rng.random((3, h, w)), rng.random((3, h, w))
    color[1, y, x] = np.inf
    _, d = _run([_cam(w, h)], color.reshape(-1), target.reshape(-1), 0.2)
    bad = ~np.isfinite(d.reshape(3, h, w))
    ys, xs = np.mgrid[0:h, 0:w]
    assert not bad[0].any() and not bad[2].any()
    assert np.array_equal(bad[1], (np.abs(ys - y) <= 10) & (np.abs(xs - x) <= 10))
