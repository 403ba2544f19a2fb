"""Reverse sweep at the edges of its fronts: one or two rays per lane, the smallest capacities
(many expand and collapse phases), partial blocks, warps with rays of several sources, and
weights that are not finite in cells no ray enters."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1711_06277_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def art():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art as A
    return A


def _case(art, shape, nsrc, force, seed, **kw):
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    rho = (0.2 + rng.random(shape)).astype(np.float32)
    dx = 1.0 / max(shape)
    pos = np.array([nx, ny, nz]) * dx * rng.uniform(0.1, 0.9, (nsrc, 3))
    L = synth.power_law_luminosities(nsrc, seed=seed)
    w = rng.random(shape).astype(np.float32)
    v = rng.uniform(-1, 1, (3,) + shape).astype(np.float32) if force else None
    p = art.Params(tau_max=30.0, sigma_H=3.0, **kw)
    g = art.Grid(torch.from_numpy(rho).cuda(), dx)
    g.add_sources(pos, L)
    prob = O.Problem(nH0=rho, pos=pos, L=L, dx=dx, sigma_H=3.0, level0=p.level0, tau_max=30.0)
    return g, p, w, v, prob


@pytest.mark.parametrize("shape,nsrc,force,kw", [
    ((14, 17, 12), 3, False, dict(level0=0)),
    ((14, 17, 12), 3, True, dict(level0=1, queue_capacity=4)),
    ((20, 24, 18), 2, False, dict(level0=2, queue_capacity=100, block_threads=64)),
    ((33, 31, 34), 7, True, dict(level0=3, block_threads=96)),
    ((40, 40, 40), 30, False, dict(level0=4)),
])
def test_sweep_edges_match_oracle(art, shape, nsrc, force, kw):
    g, p, w, v, prob = _case(art, shape, nsrc, force, 11 + nsrc, **kw)
    grad, dL, st = g.trace_backward(p, torch.from_numpy(w).cuda(),
                                    v=None if v is None else torch.from_numpy(v).cuda())
    rg, rL, _ = O.trace_adjoint(prob, w.astype(np.float64), nthreads=8,
                                v=None if v is None else v.astype(np.float64))
    # FP32 walks and sums: the parity bar of the sweep, relative to the largest gradient
    err = np.abs(grad.cpu().numpy() - rg).max() / np.abs(rg).max()
    assert err <= 1e-5, err
    assert np.abs(dL.cpu().numpy() / rL - 1).max() <= 1e-6
    assert st["destroy"] == st["destroy_expected"]
    g.close()


def test_weights_of_cells_no_ray_enters_do_not_matter(art):
    """A wall that uses up every ray: infinite and NaN weights behind it change nothing."""
    shape = (24, 24, 24)
    g, p, w, _, prob = _case(art, shape, 1, False, 3, level0=2)
    g.clear_sources()
    pos = np.array([[0.3, 0.5, 0.5]])
    g.add_sources(pos, [1.0])
    rho = prob.nH0.copy()
    rho[:, :, 16] = 1e4                     # opaque plane across x
    rho[:, 16, :] = rho[:, 4, :] = rho[16, :, :] = rho[4, :, :] = 1e4
    g.update_fields(torch.from_numpy(rho).cuda())
    w2 = w.copy()
    w2[:, :, 18:] = np.nan
    w2[:, 18:, :] = np.inf
    a, la, _ = g.trace_backward(p, torch.from_numpy(w).cuda())
    b, lb, _ = g.trace_backward(p, torch.from_numpy(w2).cuda())
    assert torch.isfinite(b).all() and torch.isfinite(lb).all()
    torch.testing.assert_close(la, lb, rtol=1e-12, atol=0.0)  # FP64 sums of equal terms
    torch.testing.assert_close(a, b, rtol=0.0, atol=1e-5 * float(a.abs().max()))
    g.close()
