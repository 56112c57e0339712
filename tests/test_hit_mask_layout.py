"""The hit masks' layout does not depend on the batch size: a forward's masks
serve a backward with another one."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2501_18630_gb300 import _lib, build, render, scenes
from tests import gpu_common as gc

# blocks of 128 pixels: few, 16320, 32640 and 65280
VIEWS = [(640, 480, 1), (1920, 1080, 1), (1920, 1080, 2), (1920, 1080, 4)]


@pytest.mark.parametrize("tile", [(8, 4), (8, 8), (16, 8), (16, 16), (32, 16)])
@pytest.mark.parametrize("w,h,views", VIEWS)
def test_size_is_the_same_for_every_batch_size(tile, w, h, views):
    build.build()
    L = _lib.load()
    cams = _lib.make_cameras([scenes.pinhole(*scenes.look_at((0, 0, -3)), w, h)] * views)
    sizes = {L.beta_hit_mask_bytes(cams, views, ctypes.byref(_lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=s)), 100_000)
             for s in (64, 128, 256)}
    assert len(sizes) == 1 and sizes.pop() > 0


@pytest.mark.gpu
@pytest.mark.parametrize("tile", [(16, 8), (16, 16), (32, 16)])
@pytest.mark.parametrize("fwd,bwd", [(64, 256), (256, 64)])
def test_backward_with_another_batch_size(tile, fwd, bwd):
    """On a view of 32379 blocks of 128 pixels: quads with one of the batches alone,
    were the batch to decide."""
    gc.ensure_built()
    cam = scenes.pinhole(*scenes.look_at((0.0, 0.0, -3.0)), 2049, 2001)
    rng = np.random.Generator(np.random.PCG64(12))
    p = torch.from_numpy(scenes.random_scene(300, 1, rng, mean_lo=-0.6, mean_hi=0.6, logscale=(-2.6, 0.5))).cuda()
    out = []
    for masks in (False, True):
        r = render.Rasterizer(300, p.shape[1], 1, [cam], _lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=fwd),
                              hit_masks=masks)
        dL = torch.rand(r.color.numel(), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1)) - 0.5
        r.forward(p)
        r.opts.batch_s = bwd
        grad = torch.zeros_like(p)
        r.raster_bwd(p, dL)
        r.project_bwd(p, grad)
        torch.cuda.synchronize()
        out.append(grad.cpu().numpy())
    g0, g1 = out
    assert np.isfinite(g0).all() and np.abs(g0).max() > 0.0
    # fp32 terms summed in another order
    assert np.max(np.abs(g1 - g0) / (np.max(np.abs(g0), axis=1, keepdims=True) + 1e-30)) < 1e-4
