"""The list sort with many primitives at the same depth: lists of one, few and
several depths at the lengths where its variants change."""
import numpy as np
import pytest

from paper_2501_18630_gb300 import scenes
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depths", [1, 2, 7, 16, 100])
@pytest.mark.parametrize("n", [3, 64, 128, 129, 256, 257, 512, 513, 4096, 4097, 9000])
def test_equal_depths_stay_in_record_order(n, depths):
    gc.ensure_built()
    rng = np.random.Generator(np.random.PCG64(n + depths))
    planes = np.zeros((15, scenes.round_pitch(n)), np.float32)
    planes[6] = 1.0
    z = rng.choice(2.0 + 0.01 * np.arange(depths), n).astype(np.float32)
    planes[2, :n] = z
    planes[3:6, :n] = np.log(0.1 * z)
    cam = scenes.pinhole(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 16, 16)
    rast, _ = gc.rasterize(planes, n, 0, [cam])
    K, ranges, vals = gc.sorted_pairs(rast)
    assert K == n and list(ranges) == [0, n]
    keys = gc.proj_arrays(rast)[2][0, :n].astype(np.int64)
    assert len(np.unique(keys)) == len(np.unique(z))
    assert np.array_equal(vals, np.lexsort((np.arange(n), keys)))
