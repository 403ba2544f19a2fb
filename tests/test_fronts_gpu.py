"""Fronts of the forward trace at the edges of their cases: one or two rays per lane, base rays
in whole groups of 64 or not, the smallest front capacities, partial blocks, and boxes whose
length leaves few fraction bits for the distances."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1711_06277_gb300 import synth
from tests import parity as PA

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def art():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art as A
    return A


@pytest.mark.parametrize("shape,nsrc,kw", [
    ((20, 24, 18), 3, dict(level0=0)),                          # 12 base rays, no groups of 64
    ((20, 24, 18), 3, dict(level0=1, queue_capacity=4)),        # smallest capacity
    ((20, 24, 18), 2, dict(level0=2, queue_capacity=17)),       # phases smaller than a group
    ((20, 24, 18), 5, dict(level0=3, queue_capacity=520)),      # phases of whole groups
    ((33, 31, 34), 7, dict(level0=4, block_threads=96)),        # widths change between levels
    ((33, 31, 34), 7, dict(level0=4, schedule="plain", block_threads=64)),
    ((64, 64, 64), 40, dict(level0=5, blocks_per_sm=1)),        # fronts of many rounds
    ((1, 3, 20000), 2, dict(level0=1, m_ray=0.05)),             # 46 fraction bits
])
def test_front_edges_match_oracle(art, shape, nsrc, kw):
    nz, ny, nx = shape
    rng = np.random.default_rng(nx + nsrc)
    rho = (0.2 + rng.random(shape)).astype(np.float32)
    dx = 1.0 / max(shape)
    pos = np.array([nx, ny, nz]) * dx * rng.uniform(0.1, 0.9, (nsrc, 3))
    L = synth.power_law_luminosities(nsrc, seed=nsrc)
    p = art.Params(tau_max=30.0, sigma_H=3.0, **kw)
    g = art.Grid(torch.from_numpy(rho).cuda(), dx)
    g.add_sources(pos, L)
    out = g.trace(p, force=True, energy=True)
    st = out["stats"]
    ref = O.trace(O.Problem(nH0=rho, pos=pos, L=L, dx=dx, sigma_H=3.0, level0=p.level0,
                            m_ray=p.m_ray, tau_max=30.0), nthreads=8, count_hits=True)
    # summation bounds of the cells' deposit counts, as in the other parity tests
    PA.compare_field(out["gamma"].cpu().numpy(), ref.gamma, what="gamma", hits=ref.hits)
    PA.compare_force(out["force"].cpu().numpy(), ref.force,
                     rho.astype(np.float64) * 3.0 * ref.energy, hits=ref.hits)
    assert st["rays_per_level"] == ref.rays_per_level.tolist()
    assert abs(st["crossings"] - ref.crossings) <= 4 * ref.near_tie_rays
    assert st["destroy"] == st["destroy_expected"]
    assert abs(st["L_escaped"] - ref.escaped) <= PA.CONS * ref.L_in
    g.close()
