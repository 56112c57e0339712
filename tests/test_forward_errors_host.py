"""Rasterizer.forward when the binning reports an error: the raster kernels launched
behind it have ended before the pair buffers are replaced and before the error is
raised.  The entry points are replaced by a record of their order: no GPU needed."""
import numpy as np
import pytest

from paper_2501_18630_gb300 import _lib, render


class _Lib:
    @staticmethod
    def beta_status_string(st):
        return b"status"


def _rasterizer(monkeypatch, statuses):
    calls, left = [], list(statuses)
    r = object.__new__(render.Rasterizer)
    r.L, r.persistent, r.color = _Lib(), True, "colour"
    r._host_status, r._host_count = np.zeros(1, np.int32), np.array([1000], np.int64)

    class _Stream:
        @staticmethod
        def synchronize():
            calls.append("sync")

    class _Event:
        record = staticmethod(lambda: None)
        synchronize = staticmethod(lambda: calls.append("wait for the count"))

    def read_state():
        r._host_status[0] = left.pop(0)

    monkeypatch.setattr(render.torch.cuda, "current_stream", lambda *a: _Stream())
    r._state_read, r._read_state = _Event(), read_state
    for name in ("project", "bin_sort", "raster_fwd"):
        setattr(r, name, lambda planes, name=name: calls.append(name))
    r.schedule = lambda: calls.append("schedule")
    r._alloc_pairs = lambda cap: calls.append("grow")
    return r, calls


def test_no_error_does_not_wait_for_the_rasters(monkeypatch):
    r, calls = _rasterizer(monkeypatch, [_lib.BETA_OK])
    assert r.forward(None) == "colour"
    assert calls == ["project", "bin_sort", "schedule", "raster_fwd", "wait for the count"]


def test_buffers_are_replaced_after_the_rasters_ended(monkeypatch):
    r, calls = _rasterizer(monkeypatch, [_lib.BETA_ERR_CAPACITY, _lib.BETA_OK])
    r.forward(None)
    first = calls.index("raster_fwd")
    assert "sync" in calls[first:calls.index("grow")]
    assert calls[-2:] == ["schedule", "raster_fwd"]


def test_an_error_is_raised_after_the_rasters_ended(monkeypatch):
    r, calls = _rasterizer(monkeypatch, [_lib.BETA_ERR_TIMEOUT])
    with pytest.raises(_lib.BetaError):
        r.forward(None)
    assert "sync" in calls[calls.index("raster_fwd"):]
