"""Relocation where the scan of the block sums takes another round (more than
1048576 primitives), with whole blocks dead and with most primitives dead, against
the oracle."""
import numpy as np
import pytest
import torch

from oracle import optim
from paper_2501_18630_gb300 import scenes
from paper_2501_18630_gb300.optim import BetaAdam
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dead_share,runs", [(255, 0.5, False), (256, 0.9, False), (257, 0.05, False), (8193, 0.9, True),
                                               (262_145, 0.05, True), (100_003, 0.9, False), (1_048_576, 0.05, False),
                                               (1_048_577, 0.05, True), (2_500_003, 0.02, True)])
def test_sources_counts_and_copies(n, dead_share, runs):
    gc.ensure_built()
    rng = np.random.default_rng(n)
    pitch = scenes.round_pitch(n)
    p = rng.normal(size=(15, pitch)).astype(np.float32)
    p[10, rng.random(pitch) < dead_share] = -9.0
    if runs:                                     # blocks of 256 that weigh nothing: first, last and in between
        for a, b in ((0, 700), (n // 3, n // 3 + 5000), (n // 2, n // 2 + 256), (n - 900, n)):
            p[10, a:b] = -9.0
    rnd = rng.integers(0, 2 ** 32, size=n, dtype=np.uint64).astype(np.uint32)
    dead = np.flatnonzero(p[10, :n] == -9.0)
    rnd[dead[0]], rnd[dead[-1]] = 0, 0xFFFFFFFF  # the first and the last source
    ref_p, _, _, ref_src, ref_k = optim.relocate(p, p, p, rnd.astype(np.uint64), n, 0.005)
    P = torch.from_numpy(p.copy()).cuda()
    opt = BetaAdam(P, n, 0)
    opt.m.fill_(1.0)
    count, src = opt.relocate(P, 0.005, torch.from_numpy(rnd.view(np.int32)).cuda())
    torch.cuda.synchronize()
    assert int(count.item()) == ref_k == len(dead)
    assert np.array_equal(src.cpu().numpy()[:n], ref_src)
    G = P.cpu().numpy()
    keep = np.arange(15) != 10
    assert np.array_equal(G[keep, :n], ref_p[keep, :n].astype(np.float32))
    # the tolerance of the other relocation test
    sig = lambda x: 1.0 / (1.0 + np.exp(-x.astype(np.float64)))
    assert np.allclose(sig(G[10, :n]), sig(ref_p[10, :n]), rtol=2e-6, atol=0)
    m = opt.m.cpu().numpy()[:, :n]
    assert np.all(m[:, ref_src >= 0] == 0.0) and np.all(m[:, ref_src < 0] == 1.0)
