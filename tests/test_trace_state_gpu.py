"""Scheduler state and counters between traces: cleared by each trace for the next, through graph
capture and replay, traces of both directions, and a trace that gave up at a barrier."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1711_06277_gb300 import synth

pytestmark = pytest.mark.gpu


def test_counters_repeat_through_capture_replay_and_failure():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import _lib as C
    from paper_1711_06277_gb300 import art
    n = 24
    rho = torch.from_numpy(synth.lognormal_field(n, 1.0, seed=5).astype(np.float32)).cuda()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        g = art.Grid(rho, 1.0 / n, stream=stream)
        g.add_sources(synth.uniform_positions(3, seed=5), [1.0, 0.5, 0.25])
        p = art.Params(level0=3, tau_max=30.0, sigma_H=4.0)
        out = {"gamma": torch.empty_like(rho), "force": torch.empty((3, n, n, n), device="cuda")}
        want = g.trace(p, out=out)["stats"]
        w = torch.ones_like(rho)
        back = g.trace_backward(p, w)[2]
        g.trace(p, stats=False, out=out)     # the reverse sweep changed the source table
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            g.trace(p, stats=False, out=out)
        for _ in range(3):
            graph.replay()
            assert g.stats()["crossings"] == want["crossings"]
        with pytest.raises(C.ArtError):
            g.trace(art.Params(level0=3, tau_max=30.0, sigma_H=4.0, wait_limit_s=-1.0), out=out)
        graph.replay()
        assert g.stats()["crossings"] == want["crossings"]
        assert g.trace_backward(p, w)[2]["crossings"] == back["crossings"]
        assert g.trace(p, out=out)["stats"] == want or \
            g.trace(p, out=out)["stats"]["rays_per_level"] == want["rays_per_level"]
        g.close()
