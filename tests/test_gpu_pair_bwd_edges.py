"""The pixel-pair and quad backward at the pixels a record does not cover: they
add nothing to its 2D gradient and keep their transmittance and suffix colour,
whatever dL/dC holds there and however large a colour is."""
import numpy as np
import pytest
import torch

from paper_2501_18630_gb300 import _lib, render, scenes
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu

# the top left pixel of a 16 x 8 block and of a quad, of 16 x 16 and of 32 x 16 tiles
PX, PY = 32, 16
SMALL, LARGE = (64, 48), (4097, 2041)          # pairs / quads
SHAPES = [((8, 8), 64, SMALL), ((16, 8), 64, SMALL), ((16, 16), 256, SMALL), ((16, 8), 64, LARGE), ((16, 16), 128, LARGE),
          ((32, 16), 64, LARGE)]


def _camera(size):
    return scenes.pinhole(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), *size)


def _planes(cam, discs):
    """Discs (pixel x, y, radius, depth, opacity logit, colour) as Betas facing the camera."""
    n = len(discs)
    pl = np.zeros((15, scenes.round_pitch(n)), np.float32)
    pl[6] = 1.0
    for i, (x, y, rad, z, logit, colour) in enumerate(discs):
        pl[:3, i] = (x + 0.5 - cam.cx) / cam.fx * z, (y + 0.5 - cam.cy) / cam.fy * z, z
        pl[3:6, i] = np.log(rad * z / cam.fx)
        pl[5, i] -= 5.0                         # flat: no skew of the disc off the optical axis
        pl[10, i] = logit
        pl[12:15, i] = colour
    return pl


def _covers(rast, i, x, y):
    r = gc.proj_arrays(rast)[0][0, i].astype(np.float64)
    dx, dy = (x - r[0]) + r[2], (y - r[1]) + r[3]
    return (r[4] * dx) ** 2 + (r[6] * dx + r[5] * dy) ** 2 < 1.0


class _Case:
    def __init__(self, discs, tile, batch, size, hit_masks):
        gc.ensure_built()
        self.cam = _camera(size)
        pl = _planes(self.cam, discs)
        self.n = len(discs)
        self.planes = torch.from_numpy(pl).cuda()
        opts = _lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=batch)
        self.rast = render.Rasterizer(self.n, pl.shape[1], 0, [self.cam], opts, hit_masks=hit_masks)
        self.rast.forward(self.planes)
        gen = torch.Generator(device="cuda").manual_seed(3)
        self.dL = torch.rand(self.rast.color.numel(), device="cuda", generator=gen) - 0.5

    def grad2d(self, at_p):
        """The 2D gradients of every record with dL/dC = at_p at pixel (PX, PY)."""
        dL = self.dL.clone()
        self.rast.image(dL, 0)[:, PY, PX] = torch.tensor(at_p, device="cuda")
        self.rast.grad2d.zero_()
        self.rast.raster_bwd(self.planes, dL)
        torch.cuda.synchronize()
        return self.rast.grad2d.view(-1, 12)[:self.n].cpu().numpy()


@pytest.mark.parametrize("hit_masks", [False, True])
@pytest.mark.parametrize("tile,batch,size", SHAPES)
@pytest.mark.parametrize("bad", [float("inf"), float("nan"), 3e38])
def test_records_that_do_not_cover_a_pixel_ignore_its_dl_dc(tile, batch, size, hit_masks, bad):
    # small ones on the pixel's row neighbour, on the row below and on the pixel
    # itself, and a large one that covers every lane of the block but not the pixel
    c = _Case([(PX + 1, PY, 0.8, 2.0, 0.0, 0.5), (PX, PY + 1, 0.8, 2.1, 0.0, 0.5), (PX, PY, 0.8, 2.2, 0.0, 0.5),
               (PX + 7.5, PY + 3.5, 8.1, 2.3, 0.0, 0.5)], tile, batch, size, hit_masks)
    assert [_covers(c.rast, i, PX, PY) for i in range(4)] == [False, False, True, False]
    assert _covers(c.rast, 0, PX + 1, PY) and _covers(c.rast, 1, PX, PY + 1) and _covers(c.rast, 3, PX + 1, PY + 1)
    want, got = c.grad2d([0.0, 0.0, 0.0]), c.grad2d([bad, 0.25, 0.25])
    others = [0, 1, 3]
    assert np.isfinite(want).all() and np.isfinite(got[others]).all()
    # the same terms; the large record's are added in another order
    assert np.abs(got[others] - want[others]).max() <= 1e-5 * np.abs(want[others]).max()
    assert np.abs(got[2]).max() > 1e30 or not np.isfinite(got[2]).all()


@pytest.mark.parametrize("hit_masks", [False, True])
@pytest.mark.parametrize("tile,batch,size", SHAPES)
def test_a_product_that_overflows_stays_with_its_pixel(tile, batch, size, hit_masks):
    """A colour of 10 where dL/dC is 3e38 next to it: the record in front, on that pixel
    only, has the gradient it has with a colour of 0.5 behind it."""
    grads = []
    for colour in (0.5, 10.0):
        c = _Case([(PX, PY, 0.8, 2.0, 0.0, 0.01), (PX + 1, PY, 0.8, 2.1, 0.0, colour), (PX, PY + 1, 0.8, 2.2, 0.0, colour)],
                  tile, batch, size, hit_masks)
        assert [_covers(c.rast, i, PX, PY) for i in range(3)] == [True, False, False]
        grads.append(c.grad2d([3e38, 0.0, 0.0]))
    assert np.isfinite(grads[0][0]).all() and np.abs(grads[0][0]).max() > 1e30
    np.testing.assert_array_equal(grads[1][0], grads[0][0])
    assert np.isfinite(grads[1]).all()


@pytest.mark.parametrize("hit_masks", [False, True])
@pytest.mark.parametrize("tile,batch,size", SHAPES)
def test_records_that_do_not_cover_a_pixel_keep_its_transmittance(tile, batch, size, hit_masks):
    """The first record, on one pixel only, in front of 1500 that cover only its neighbours:
    its gradient is bit for bit that without them."""
    front = [(PX + 0.1, PY + 0.07, 0.8, 2.0, 0.0, 0.3)]
    behind = [(PX + k % 2, PY + 1 - k % 2, 0.8, 2.1 + k * 1e-3, -6.0, 0.5) for k in range(1500)]
    a = _Case(front, tile, batch, size, hit_masks)
    b = _Case(front + behind, tile, batch, size, hit_masks)
    assert _covers(b.rast, 0, PX, PY) and not any(_covers(b.rast, i, PX, PY) for i in (1, 2, 1499, 1500))
    at = [0.7, -0.3, 0.9]
    want, got = a.grad2d(at)[0], b.grad2d(at)[0]
    assert np.abs(want[:10]).min() > 0.0
    np.testing.assert_array_equal(got, want)
