"""The 2 x 2 quad raster kernels with every tile shape and batch that takes them on
a view just large enough, hit masks on and off, against 8x8 tiles (pixel pairs);
and the line itself, which the size of the hit masks shows."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2501_18630_gb300 import _lib, build, render, scenes
from tests import gpu_common as gc

FEWEST = 31000


@pytest.mark.parametrize("tile,h,quads", [((16, 8), 1976, False), ((16, 8), 1984, True), ((16, 16), 1968, False),
                                          ((16, 16), 1984, True), ((32, 16), 1968, False), ((32, 16), 1984, True)])
def test_fewest_blocks_of_quads(tile, h, quads):
    build.build()
    L, o = _lib.load(), _lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=64)
    cams = _lib.make_cameras([scenes.pinhole(*scenes.look_at((0, 0, -3)), 2000, h)])
    tiles = L.beta_total_tiles(cams, 1, ctypes.byref(o))
    assert (tiles * tile[0] * tile[1] // 128 >= FEWEST) == quads
    lanes = tile[0] * tile[1] // (4 if quads else 2)
    assert L.beta_hit_mask_bytes(cams, 1, ctypes.byref(o), 10000) == ((10000 >> 5) + tiles + 1) * (lanes + lanes // 32) * 4


def _run(p, cam, tile, batch, fused, persistent, hit_masks):
    r = render.Rasterizer(400, p.shape[1], 1, [cam], _lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=batch),
                          persistent=persistent, hit_masks=hit_masks)
    target = torch.from_numpy(scenes.target_images([cam], seed=3)[0].reshape(-1)).cuda()
    r.forward(p)
    grad = torch.zeros_like(p)
    if fused:
        r.raster_fwd_bwd_l1(p, target)
    else:
        r.raster_fwd_l1(p, target)
        r.raster_bwd(p, r.dL_dcolor)
    r.project_bwd(p, grad)
    torch.cuda.synchronize()
    return r.color.cpu().numpy(), grad.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("tile,batch", [((16, 8), 64), ((16, 16), 64), ((16, 16), 128), ((32, 16), 64), ((32, 16), 128),
                                        ((32, 16), 256)])
@pytest.mark.parametrize("fused,persistent,hit_masks", [(True, False, False), (True, True, False), (False, False, False),
                                                        (False, True, True)])
def test_quads_equal_pairs(tile, batch, fused, persistent, hit_masks):
    gc.ensure_built()
    cam = scenes.pinhole(*scenes.look_at((0.0, 0.0, -3.0)), 2049, 2001)
    rng = np.random.Generator(np.random.PCG64(12))
    p = torch.from_numpy(scenes.random_scene(400, 1, rng, mean_lo=-0.6, mean_hi=0.6, logscale=(-2.6, 0.5))).cuda()
    c0, g0 = _run(p, cam, (8, 8), 64, False, False, False)
    c1, g1 = _run(p, cam, tile, batch, fused, persistent, hit_masks)
    np.testing.assert_array_equal(c1, c0)
    # fp32 terms summed in another order
    assert np.max(np.abs(g1 - g0) / (np.max(np.abs(g0), axis=1, keepdims=True) + 1e-30)) < 1e-4
