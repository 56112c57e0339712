"""The projection backward at the number of lobes where it stops copying the next
block's parameters ahead: one call over many blocks of primitives gives what calls
on a few blocks each give, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2501_18630_gb300 import render, scenes
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lobes", [4, 5, 8])
@pytest.mark.parametrize("n,views", [(3, 2), (129, 1), (60_001, 3)])
def test_whole_range_equals_parts(lobes, n, views):
    gc.ensure_built()
    rng = np.random.Generator(np.random.PCG64(n + lobes))
    planes_np = scenes.random_scene(n, lobes, rng)
    planes_np[3, 1:n:7] = np.nan                      # culled
    planes = torch.from_numpy(planes_np).cuda()
    r = render.Rasterizer(n, planes.shape[1], lobes, scenes.ring_cameras(views, 3.0, 10.0, (64, 48)))
    g2 = torch.randn(r.grad2d.numel(), device="cuda", generator=torch.Generator(device="cuda").manual_seed(n)) * 1e-3
    r.status.zero_()
    out = []
    for chunk in (n, 384):
        r.grad2d.copy_(g2)
        grad = torch.full_like(planes, 7.0)
        for c0 in range(0, n, chunk):
            r.project_bwd(planes, grad, c0, min(n, c0 + chunk))
        torch.cuda.synchronize()
        out.append((grad, r.grad2d.clone()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert bool((out[0][0][:, n:] == 7.0).all()) and bool((out[0][0][:, 1:n:7] == 0.0).all())
    assert bool(torch.isfinite(out[0][0]).all()) and float(out[0][0][:, :n].abs().max()) > 0.0
