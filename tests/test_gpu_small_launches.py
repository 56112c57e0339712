"""The tile schedule around the number of tiles that one CTA takes, and the sum of
the L1 loss around the numbers of partial sums that a warp and a CTA take."""
import numpy as np
import pytest
import torch

from paper_2501_18630_gb300 import _lib, render, scenes
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(8, 4), (1024, 252), (1024, 256), (1024, 260)])
def test_schedule_around_one_launch(w, h):
    gc.ensure_built()
    sc = scenes.config_scene(3, n=4000)
    planes = torch.from_numpy(sc.planes).cuda()
    r = render.Rasterizer(sc.n, sc.pitch, sc.n_lobes, [scenes.ring_camera(4.0, 15.0, 0.3, w, h)],
                          _lib.default_opts(tile_w=8, tile_h=4, batch_s=64), persistent=True)
    r.project(planes)
    r.bin_sort(planes)
    r.sched.fill_(-1)
    r.schedule()
    torch.cuda.synchronize()
    order = r.sched.cpu().numpy()[144:144 + r.total_tiles]
    assert np.array_equal(np.sort(order), np.arange(r.total_tiles))
    bits = np.array([int(n).bit_length() for n in np.diff(r.ranges.cpu().numpy().astype(np.int64))])[order]
    assert (np.diff(bits) <= 0).all()


@pytest.mark.parametrize("blocks", [[1], [8, 9], [255, 1, 256], [257], [4095, 4096, 4097], [9000, 3]])
def test_l1_sums(blocks):
    """Views of 256 pixels times `blocks`: one partial sum per 256 pixels."""
    gc.ensure_built()
    cams = [scenes.pinhole(*scenes.look_at((0, 0, -3)), 256, b) for b in blocks]
    r = render.Rasterizer(32, 32, 0, cams)
    gen = torch.Generator(device="cuda").manual_seed(len(blocks))
    r.color.copy_(torch.rand(r.color.numel(), device="cuda", generator=gen))
    target = torch.rand(r.color.numel(), device="cuda", generator=gen)
    loss, _ = r.l1_loss(target)
    for v in range(len(blocks)):
        want = (r.image(r.color, v).double() - r.image(target, v).double()).abs().mean().item()
        # 256 pixels in fp32, at most 17 additions in a row (17 x 2^-24 = 1e-6), fp64 from there
        assert loss[v].item() == pytest.approx(want, rel=1e-5)
