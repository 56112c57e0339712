"""A tuned configuration is looked up again after a change to the kernels it was
timed on: the cache key holds the library's sources."""
import os
import shutil

from paper_2501_18630_gb300 import autotune, build, scenes


def test_key_changes_with_the_kernel_sources(monkeypatch, tmp_path):
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda dev=None: "fake GB300")
    cams = [scenes.ring_camera(4.0, 15.0, 0.0, 320, 240)]
    key = lambda: autotune.workload_key(1000, 3, cams, "cuda:0")
    first = key()
    csrc = tmp_path / "csrc"
    shutil.copytree(build.CSRC, csrc)
    monkeypatch.setattr(build, "CSRC", str(csrc))
    assert key() == first
    with open(os.path.join(csrc, "beta_raster.cu"), "a") as fh:
        fh.write("// another kernel\n")
    assert key() != first
