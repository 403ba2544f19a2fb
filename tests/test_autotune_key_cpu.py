"""The autotuner times the kernel that its caller will run and uses no knobs of another one."""
import json
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1711_06277_gb300 import art as A
from paper_1711_06277_gb300 import autotune as T


@pytest.fixture
def timed(monkeypatch):
    """Fakes the device work; returns the force arguments of the traces that are timed."""
    seen = []

    class Event:
        def __init__(self, enable_timing=False): pass
        def record(self, stream): pass
        def synchronize(self): pass
        def elapsed_time(self, other): return 1.0

    class Grid:
        def __init__(self, *a, **kw): pass
        def add_sources(self, pos, L): pass
        def trace(self, p, force=True, stats=True): seen.append(force)
        def stats(self): return {"status": 0}
        def close(self): pass

    monkeypatch.setattr(T, "torch", types.SimpleNamespace(cuda=types.SimpleNamespace(
        Event=Event, current_stream=lambda device: None)))
    monkeypatch.setattr(T.A, "Grid", Grid)
    return seen


def _tune(path, **kw):
    return T.tune(torch.ones((8, 8, 8)), 1.0 / 8, np.full((3, 3), 0.5), np.ones(3),
                  A.Params(level0=2, d_max=kw.pop("d_max", 0.0)), cache_path=str(path),
                  space={"block_threads": [320, 640]}, **kw)


@pytest.mark.parametrize("kw,want", [({}, True), (dict(force=True), True), (dict(force=False), False)])
def test_candidates_are_timed_with_the_callers_outputs(timed, tmp_path, kw, want):
    _tune(tmp_path / "c.json", **kw)
    assert timed and set(timed) == {want}


def test_knobs_of_another_kernel_are_not_used(timed, tmp_path, monkeypatch):
    path = tmp_path / "c.json"
    shape, p = (8, 8, 8), A.Params(level0=2)
    # an entry whose key names no kernel, as earlier versions wrote them
    path.write_text(json.dumps({"8x8x8|src3|l02|m4.0": {"knobs": {"block_threads": 128}}}))
    assert _tune(path).block_threads in (320, 640)
    for other in (dict(force=False), dict(d_max=0.3)):
        timed.clear()
        _tune(path, **other)
        assert timed  # searched again
    timed.clear()
    _tune(path)
    assert not timed  # a hit
    assert T._key(shape, 3, p) in json.loads(path.read_text())
    monkeypatch.setattr(T, "_kernel_version", lambda: "other")
    _tune(path)
    assert timed
