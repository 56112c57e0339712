"""The list sort and the tile scan where their variants change: list lengths at
the edges of the warp and CTA sorts with distinct, tied and clustered depth
keys, and tile counts at the edges of the scan's block sizes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_18630_gb300 import _lib, render, scenes
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


def _depths(n, mode, rng):
    if mode == "distinct":
        z = np.exp(rng.uniform(0.0, 3.0, n))
    elif mode == "pairs":                       # every depth twice: neighbours out of order
        z = np.repeat(np.exp(rng.uniform(0.0, 1.0, (n + 1) // 2)), 2)[:n]
    elif mode == "ties":                        # three depths in all
        z = rng.choice([2.0, 2.5, 3.0], n)
    else:                                       # a cluster next to a far outlier: keys collapse when shifted
        z = 3.0 + rng.integers(0, 4 * n, n) * 2.0 ** -22
        z[0] = 1e6
    return rng.permutation(z).astype(np.float32)


@pytest.mark.parametrize("mode", ["distinct", "pairs", "ties", "cluster"])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 128, 129, 256, 257, 511, 512, 513, 1024, 1025, 2048, 2049, 4096,
                               4097])
def test_one_list_of_every_length(n, mode):
    gc.ensure_built()
    rng = np.random.Generator(np.random.PCG64(n))
    pitch = scenes.round_pitch(n)
    planes = np.zeros((15, pitch), np.float32)
    planes[6] = 1.0
    z = _depths(n, mode, rng)
    planes[2, :n] = z
    planes[3:6, :n] = np.log(0.1 * z)           # about the same size on the image at every depth
    cam = scenes.pinhole(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 16, 16)
    rast, _ = gc.rasterize(planes, n, 0, [cam])
    K, ranges, vals = gc.sorted_pairs(rast)
    assert K == n and list(ranges) == [0, n]
    keys = gc.proj_arrays(rast)[2][0, :n].astype(np.int64)
    assert np.array_equal(vals, np.lexsort((np.arange(n), keys)))


@pytest.mark.parametrize("w,h,tiles", [(8, 4, 1), (1024, 256, 8192), (1032, 256, 8256), (2048, 256, 16384),
                                       (1024, 516, 16512), (1024, 1024, 32768), (1024, 1028, 32896)])
def test_scan_block_sizes(w, h, tiles):
    sc = scenes.config_scene(3, n=6000)
    cams = [scenes.ring_camera(4.0, 15.0, 0.3, w, h)]
    opts = _lib.default_opts(tile_w=8, tile_h=4, batch_s=64)
    rast, _ = gc.rasterize(sc.planes, sc.n, sc.n_lobes, cams, opts=opts)
    assert rast.total_tiles == tiles
    K, ranges, vals = gc.sorted_pairs(rast)
    _, recs, oranges = oracle.bin_pairs(sc.planes, sc.n, sc.n_lobes, cams, tile_w=8, tile_h=4, pitch=sc.pitch)
    assert K == len(recs)
    assert np.array_equal(ranges, oranges)
    assert np.array_equal(vals, recs)
