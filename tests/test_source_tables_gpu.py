"""Calls that only enqueue work keep their own sources: traces and sweeps queued behind a busy
stream, with other directions, sources and parameters in between, equal those of a stream that is
waited for, and a captured trace keeps its sources through calls of the other direction."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1711_06277_gb300 import synth

pytestmark = pytest.mark.gpu

N = 24
# FP32 sums of hundreds of positive terms in an order of their own; gradients cancel by less than 100
TOL = 1e-4


def _close(a, b):
    return float((a - b).norm() / b.norm()) < TOL


def _calls(art, g, w, wait):
    """Outputs of a series of calls without stats, waited for one by one or not at all."""
    pos = synth.uniform_positions(6, seed=5)
    p4, p3 = art.Params(level0=4, tau_max=30.0, sigma_H=4.0, sigma_d=1.0), art.Params(level0=3, m_ray=8.0, tau_max=30.0, sigma_H=4.0, sigma_d=1.0)
    out = []

    def sources(k, ln=None):
        g.clear_sources()
        g.add_sources(pos[:k], np.arange(1.0, k + 1.0) * 10.0 ** k)
        if ln is not None:
            g.set_nonionizing(ln * np.arange(1.0, k + 1.0))

    def trace(p):
        out.append(g.trace(p, force=False, stats=False)["gamma"])
        if wait:
            torch.cuda.synchronize()

    def sweep(p):
        grad, dL, _ = g.trace_backward(p, w, stats=False)
        out.extend([grad, dL])
        if wait:
            torch.cuda.synchronize()

    sources(6, 3.0), trace(p4)      # the largest first: nothing is allocated behind the busy stream
    sources(6), trace(p4), sweep(p4), trace(p3)
    torch.cuda.synchronize()
    if not wait:
        torch.cuda._sleep(200_000_000)
    sources(6), trace(p4), sweep(p4), trace(p4)
    sources(4), sweep(p3), trace(p3)
    sources(5, 3.0), trace(p4)
    sources(5, 1.0), trace(p4)
    sources(5), sweep(p4), trace(p4)
    return out


def test_queued_calls_keep_their_sources():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    rho = torch.from_numpy(synth.lognormal_field(N, 1.0, seed=5).astype(np.float32)).cuda()
    w = torch.rand((N, N, N), device="cuda")
    res = []
    for wait in (True, False):
        g = art.Grid(rho, 1.0 / N, nH=rho)
        res.append(_calls(art, g, w, wait))
        torch.cuda.synchronize()
        g.close()
    for k, (a, b) in enumerate(zip(*res)):
        assert _close(b, a), k


def test_captured_trace_keeps_its_sources():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    rho = torch.from_numpy(synth.lognormal_field(N, 1.0, seed=5).astype(np.float32)).cuda()
    w = torch.rand((N, N, N), device="cuda")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        g = art.Grid(rho, 1.0 / N, stream=stream)
        pos = synth.uniform_positions(3, seed=5)
        g.add_sources(pos, [10.0, 5.0, 2.5])
        p = art.Params(level0=4, tau_max=30.0, sigma_H=4.0)
        out = {"gamma": torch.empty_like(rho)}
        want = g.trace(p, force=False)["gamma"]
        grad = g.trace_backward(p, w)[0]
        g.trace(p, force=False)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):   # unchanged: no table in the graph
            g.trace(p, force=False, stats=False, out=out)
        assert _close(g.trace_backward(p, w, stats=False)[0], grad)
        graph.replay()
        assert _close(out["gamma"], want)
        g.clear_sources()
        g.add_sources(pos, [1.0, 2.0, 4.0])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):   # changed: the graph stores the table
            g.trace(p, force=False, stats=False, out=out)
        eager = g.trace(p, force=False)["gamma"].clone()   # the graph has not run yet
        g.clear_sources()
        g.add_sources(pos, [10.0, 5.0, 2.5])
        assert _close(g.trace(p, force=False)["gamma"], want)
        graph.replay()
        assert _close(out["gamma"], eager) and not _close(eager, want)
        assert _close(g.trace(p, force=False)["gamma"], want)
        g.close()
