"""The projection backward's persistent loop over blocks of 128 primitives (the
next block's parameters and 2D gradients copied in ahead): bit for bit the
gradients of calls on ranges small enough that every CTA takes one block, with
padding columns untouched and the 2D-gradient slots cleared."""
import numpy as np
import pytest
import torch

from paper_2501_18630_gb300 import render, scenes
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lobes,views", [(1, 0, 1), (127, 3, 2), (128, 1, 1), (129, 3, 3), (60_001, 3, 2),
                                           (60_001, 8, 1), (120_005, 0, 1)])
def test_persistent_blocks_equal_single_blocks(n, lobes, views):
    gc.ensure_built()
    rng = np.random.Generator(np.random.PCG64(n + lobes))
    planes_np = scenes.random_scene(n, lobes, rng)
    planes_np[3, :n:7] = np.nan                       # culled: zero gradients, slots untouched
    planes = torch.from_numpy(planes_np).cuda()
    cams = scenes.ring_cameras(views, 3.0, 10.0, (64, 48))
    r = render.Rasterizer(n, planes.shape[1], lobes, cams)
    g2 = torch.randn(r.grad2d.numel(), device="cuda", generator=torch.Generator(device="cuda").manual_seed(n)) * 1e-3
    g2.view(-1, 12)[::5] = 0.0
    r.status.zero_()

    def run(chunk):
        r.grad2d.copy_(g2)
        grad = torch.full_like(planes, 7.0)
        for c0 in range(0, n, chunk):
            r.project_bwd(planes, grad, c0, min(n, c0 + chunk))
        torch.cuda.synchronize()
        return grad, r.grad2d.clone()

    whole, left = run(n)
    parts, left_parts = run(4096)
    assert torch.equal(whole.nan_to_num(nan=-1.0), parts.nan_to_num(nan=-1.0))
    assert torch.equal(left, left_parts)
    assert bool((whole[:, n:] == 7.0).all()) and bool((whole[:, :n:7] == 0.0).all())
    live = torch.ones(n, dtype=torch.bool, device="cuda")
    live[::7] = False
    slots = left.view(views, planes.shape[1], 12)[:, :n]
    assert bool((slots[:, live] == 0.0).all())
