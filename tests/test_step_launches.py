"""The number of kernels bench.py charges to a captured step, against the rule of
the schedule's launches in the library's source."""
import os
import re

import bench
from paper_2501_18630_gb300 import build


def test_schedule_launches_follow_the_library():
    src = open(os.path.join(build.CSRC, "beta_raster.cu")).read()
    one = int(re.search(r"kSchedOneTiles = (\d+)", src).group(1))
    assert bench.SCHEDULE_ONE_LAUNCH == one
    assert [bench.launches_per_step(t, True) for t in (0, 1, one, one + 1)] == [9, 10, 10, 12]
    assert bench.launches_per_step(0, False) == 10 and bench.launches_per_step(0, True, 8) == 16
