"""The packed pixel-pair raster kernels against the one-pixel kernels (8x4
tiles) where packed arithmetic could differ: a record with an infinite colour
must leave the pixels it does not cover, its pair's other pixel among them,
exactly as they are, in images and gradients."""
import numpy as np
import pytest
import torch

from paper_2501_18630_gb300 import _lib, render, scenes
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


def _scene(odd):
    rng = np.random.Generator(np.random.PCG64(11))
    planes = scenes.random_scene(60, 1, rng, mean_lo=-0.6, mean_hi=0.6, logscale=(-2.6, 0.5))
    if odd:
        k = int(np.argsort(planes[2, :60])[20])       # some Betas in front of it, some behind
        planes[12, k] = 3e38                           # base colour + lobe colour overflow
        planes[15 + 2, k] = -20.0                      # lobe exponent ~ 0: weight 1 where it faces the view
        planes[18, k] = 3e38
        planes[15, k], planes[16, k] = np.pi / 2, 0.0
        d = planes[0:3, k] - np.array([0.0, 0.0, -3.0])
        planes[15, k], planes[16, k] = np.arccos(d[2] / np.linalg.norm(d)), np.arctan2(d[1], d[0])
    return planes


def _odd_index():
    return int(np.argsort(_scene(False)[2, :60])[20])


def _run(planes_np, cam, tile, s, fused):
    gc.ensure_built()
    planes = torch.from_numpy(planes_np).cuda()
    opts = _lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=s)
    r = render.Rasterizer(60, planes.shape[1], 1, [cam], opts)
    target = torch.from_numpy(scenes.target_images([cam], seed=3)[0].reshape(-1)).cuda()
    r.forward(planes)
    grad = torch.zeros_like(planes)
    if fused:
        r.raster_fwd_bwd_l1(planes, target)
    else:
        r.raster_fwd_l1(planes, target)
        r.raster_bwd(planes, r.dL_dcolor)
    r.project_bwd(planes, grad)
    torch.cuda.synchronize()
    return r.color.cpu().numpy(), grad.cpu().numpy()


@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("tile,s,fused", [((8, 8), 64, False), ((16, 8), 64, True), ((16, 16), 128, False),
                                          ((16, 16), 256, True), ((32, 16), 64, True)])
@pytest.mark.parametrize("w,h", [(37, 29), (64, 48)])
def test_pair_kernels_equal_one_pixel_kernels(odd, tile, s, fused, w, h):
    cam = scenes.pinhole(*scenes.look_at((0.0, 0.0, -3.0)), w, h)
    planes = _scene(odd)
    c0, g0 = _run(planes, cam, (8, 4), 64, False)
    c1, g1 = _run(planes, cam, tile, s, fused)
    assert np.isfinite(c0).all() != odd and (not odd or np.isfinite(c0).mean() > 0.2)
    np.testing.assert_array_equal(c1, c0)              # NaN and infinities in the same places too
    fin = np.isfinite(g0)
    assert (np.isfinite(g1) == fin).all() and fin.any()
    # fp32 terms summed in another order: 60 Betas on a few thousand pixels,
    # each sum off by at most ~sqrt(terms) roundings of its largest partial sums
    scale = np.max(np.abs(np.where(fin, g0, 0.0)), axis=1, keepdims=True) + 1e-30
    assert np.max(np.abs(np.where(fin, g1 - g0, 0.0)) / scale) < 1e-4


@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("tile,s,fused,persistent", [((16, 8), 64, True, False), ((16, 8), 64, False, True),
                                                     ((16, 16), 64, True, True), ((16, 16), 128, False, False),
                                                     ((32, 16), 64, False, False), ((32, 16), 128, True, False),
                                                     ((32, 16), 256, True, True)])
def test_quad_kernels_equal_one_pixel_kernels(odd, tile, s, fused, persistent):
    """The same at an odd-sized view large enough for two pairs a lane; the split
    path with hit masks."""
    cam = scenes.pinhole(*scenes.look_at((0.0, 0.0, -3.0)), 2049, 1001)
    assert -(-2049 // 16) * -(-1001 // 8) >= 16000
    planes = _scene(odd)
    c0, g0 = _run(planes, cam, (8, 4), 64, False)
    gc.ensure_built()
    p = torch.from_numpy(planes).cuda()
    r = render.Rasterizer(60, p.shape[1], 1, [cam], _lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=s),
                          persistent=persistent, hit_masks=True)
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
    np.testing.assert_array_equal(r.color.cpu().numpy(), c0)
    g1 = grad.cpu().numpy()
    fin = np.isfinite(g0)
    assert (np.isfinite(g1) == fin).all() and fin.any()
    if odd:
        # the infinite record's own lobe-direction gradients are 3e38 times sums that
        # cancel (they differ between any two tilings): compared for finiteness only
        g0[:, _odd_index()] = g1[:, _odd_index()] = 0.0
    scale = np.max(np.abs(np.where(fin, g0, 0.0)), axis=1, keepdims=True) + 1e-30
    with np.errstate(invalid="ignore"):
        assert np.max(np.abs(np.where(fin, g1 - g0, 0.0)) / scale) < 1e-4


@pytest.mark.parametrize("tile,s,fused,persistent", [((16, 8), 128, True, False), ((16, 8), 256, False, True),
                                                     ((16, 16), 256, True, True), ((16, 16), 256, False, False)])
def test_quads_of_large_batches_equal_pairs_of_one_warp(tile, s, fused, persistent):
    """Batches of more records than a quad CTA stages at a time, on views large
    enough for quads with them; 8x8 tiles (one warp, pairs) as the reference."""
    cam = scenes.pinhole(*scenes.look_at((0.0, 0.0, -3.0)), 4097, 2041)
    assert -(-4097 // 16) * -(-2041 // 8) >= 64000
    rng = np.random.Generator(np.random.PCG64(12))
    p = torch.from_numpy(scenes.random_scene(400, 1, rng, mean_lo=-0.6, mean_hi=0.6, logscale=(-2.6, 0.5))).cuda()
    target = torch.from_numpy(scenes.target_images([cam], seed=3)[0].reshape(-1)).cuda()
    gc.ensure_built()
    out = []
    for t, b, per in (((8, 8), 64, False), (tile, s, persistent)):
        r = render.Rasterizer(400, p.shape[1], 1, [cam], _lib.default_opts(tile_w=t[0], tile_h=t[1], batch_s=b),
                              persistent=per, hit_masks=True)
        r.forward(p)
        grad = torch.zeros_like(p)
        if fused:
            r.raster_fwd_bwd_l1(p, target)
        else:
            r.raster_fwd_l1(p, target)
            r.raster_bwd(p, r.dL_dcolor)
        r.project_bwd(p, grad)
        torch.cuda.synchronize()
        out.append((r.color.cpu().numpy(), grad.cpu().numpy()))
    np.testing.assert_array_equal(out[1][0], out[0][0])
    g0, g1 = out[0][1], out[1][1]
    # fp32 terms summed in another order
    assert np.max(np.abs(g1 - g0) / (np.max(np.abs(g0), axis=1, keepdims=True) + 1e-30)) < 1e-4


@pytest.mark.parametrize("w,h,tile", [(1, 1, (8, 4)), (257, 129, (16, 16)), (1024, 512, (8, 4)), (1032, 512, (8, 4))])
def test_schedule_orders_every_tile_longest_first(w, h, tile):
    """One CTA up to 16384 tiles, three launches above: a permutation of the tiles
    by descending bit length of their list."""
    gc.ensure_built()
    sc = scenes.config_scene(3, n=4000)
    planes = torch.from_numpy(sc.planes).cuda()
    r = render.Rasterizer(sc.n, sc.pitch, sc.n_lobes, [scenes.ring_camera(4.0, 15.0, 0.3, w, h)],
                          _lib.default_opts(tile_w=tile[0], tile_h=tile[1], batch_s=64), persistent=True)
    r.project(planes)
    r.bin_sort(planes)
    r.sched.fill_(-1)
    r.schedule()
    torch.cuda.synchronize()
    sched, ranges = r.sched.cpu().numpy(), r.ranges.cpu().numpy().astype(np.int64)
    order = sched[144:144 + r.total_tiles]
    assert (sched[:4] == 0).all() and np.array_equal(np.sort(order), np.arange(r.total_tiles))
    bits = np.array([int(n).bit_length() for n in np.diff(ranges)])[order]
    assert (np.diff(bits) <= 0).all()


@pytest.mark.parametrize("persistent", [False, True])
def test_forward_grows_the_pair_buffers_behind_launched_rasters(persistent):
    """An overflow found after the raster kernels were launched: they wrote
    nothing, and the image after growing is that of large buffers."""
    gc.ensure_built()
    sc = scenes.config_scene(1)
    planes = torch.from_numpy(sc.planes).cuda()
    r0 = render.Rasterizer(sc.n, sc.pitch, sc.n_lobes, sc.cameras, persistent=persistent)
    r1 = render.Rasterizer(sc.n, sc.pitch, sc.n_lobes, sc.cameras, persistent=persistent, pair_capacity=100)
    want = r0.forward(planes).clone()
    for _ in range(2):
        assert torch.equal(r1.forward(planes), want)
    assert r1.cap > 100 and r1.device_status() == (0, int(r0.count.item()))
